"""Representative work of the library, one case per way it is used.

A case is a dict of plain values; `prepare` builds what a user's program holds before the call (a
configured context, batch or server and the input fields), `run` is one pass through the public
entry points, `work` its irreducible bytes and flops, and `exact` the same outputs from plain
FP64 torch. Sizes come from the workloads of inputs.py and from the tests and the benchmark.

Kinds:
  local   a local-stencil context: set the field, advance `steps` steps, read the field
  pu      the same with the partition-of-unity method
  global  the same with the global method, solved and evaluated every step
  card    the same with the global method in cardinal form (steady flow)
  batch   many independent local problems advanced together, fields read on the host
  serve   requests submitted to the serving loop, run to completion, results collected
"""
import math

import numpy as np
import torch

from paper_1804_01609_gb300 import inputs, rbfsl

DEV = "cuda"


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the README's first example: one tracer rotated on a coarse node set, FP64; what counts is
        # the latency of a step of a small model
        dict(name="direct-2562-n31-f64", kind="local", mode="direct", N=2562, n=31, ell=2, power=3, T=1,
             precision="f64", vel="rigid", steps=1),
        # a ragged mid-size run in mixed precision, stencils of the middle class
        dict(name="direct-12347-n55-mixed", kind="local", mode="direct", N=12347, n=55, ell=3, power=7, T=5,
             precision="mixed", vel="nl", steps=1),
        # the benchmark's headline step: deformational flow, largest stencils, 32 tracers
        dict(name="direct-40962-n84-mixed", kind="local", mode="direct", N=40962, n=84, ell=4, power=9, T=32,
             precision="mixed", vel="deform", steps=1),
        # the paper's own local method (stencil of the nearest node) at the same size
        dict(name="center-40962-n84-mixed", kind="local", mode="center", N=40962, n=84, ell=4, power=9, T=32,
             precision="mixed", vel="deform", steps=1),
        # centre stencils on a fine node set, FP64, few tracers
        dict(name="center-163842-n31-f64", kind="local", mode="center", N=163842, n=31, ell=2, power=5, T=4,
             precision="f64", vel="rigid", steps=1),
        # partition of unity as inputs.config_pu_rotation has it: two tracers, FP64
        dict(name="pu-10242-n100-f64", kind="pu", N=10242, n=100, ell=3, power=7, T=2, precision="f64",
             vel="rigid", steps=1),
        # partition of unity with many tracers on the finer set, mixed precision
        dict(name="pu-40962-n84-mixed", kind="pu", N=40962, n=84, ell=3, power=7, T=16, precision="mixed",
             vel="nl", steps=1),
        # the global method at the size of inputs.config_global_rotation, tensor-core evaluation
        dict(name="global-10242-mixed", kind="global", N=10242, kernel="gauss", T=64, precision="mixed",
             vel="rigid", steps=1),
        # a smaller, odd-sized global run in FP64 with the paper's kernel
        dict(name="global-4999-f64", kind="global", N=4999, kernel="imq", T=9, precision="f64", vel="deform",
             steps=1),
        # steady flow: the global step as one dense product
        dict(name="cardinal-5003-mixed", kind="card", N=5003, kernel="imq", T=64, precision="mixed", vel="rigid",
             steps=1),
        # many problems of inputs.batched_problems in one launch per step
        dict(name="batch-24-mixed", kind="batch", P=24, nmax=10242, precision="mixed", steps=2),
        # the serving loop: local and partition-of-unity requests of mixed sizes, run to the end
        dict(name="serve-10", kind="serve", R=10, nmax=10242, precision="mixed", steps=12),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["local"] * 4 + ["pu"] * 2 + ["global", "card", "batch", "serve"])
    prec = rng.choice(["f64", "mixed"])
    vel = rng.choice(["rigid", "deform", "nl"])
    if kind == "local":
        n = rng.choice([31, 55, 84, rng.randint(17, 84)])
        ell = int(math.floor(0.5 * (math.sqrt(n) - 1.0)))  # the paper's rule, with r^(2 ell + 1)
        top = 40962 if n > 55 else 81921 if n > 31 else 163842
        return dict(kind=kind, mode=rng.choice(["direct", "center"]), N=_logint(rng, 642, top), n=n, ell=ell,
                    power=2 * ell + 1, T=_logint(rng, 1, 32), precision=prec, vel=vel, steps=1)
    if kind == "pu":
        n = rng.randint(31, 100)
        ell = int(math.floor(0.5 * (math.sqrt(n) - 1.0))) if n < 49 else 3
        return dict(kind=kind, N=_logint(rng, 2562, 40962), n=n, ell=ell, power=2 * ell + 1, T=rng.randint(1, 16),
                    precision=prec, vel=vel, steps=1)
    if kind == "global":
        return dict(kind=kind, N=_logint(rng, 1000, 7001), kernel=rng.choice(["gauss", "imq"]), T=_logint(rng, 1, 64),
                    precision=prec, vel=vel, steps=1)
    if kind == "card":
        return dict(kind=kind, N=_logint(rng, 1000, 5003), kernel=rng.choice(["gauss", "imq"]), T=_logint(rng, 1, 64),
                    precision=prec, vel="rigid", steps=rng.randint(1, 3))
    if kind == "batch":
        return dict(kind=kind, P=rng.randint(3, 20), nmax=rng.choice([2562, 10242]), precision=prec, steps=rng.randint(1, 2))
    return dict(kind=kind, R=rng.randint(3, 9), nmax=rng.choice([2562, 10242]), precision=prec, steps=rng.randint(6, 12))


# ------------------------------------------------------------------------------- inputs
_VEL = {"rigid": rbfsl.VEL_RIGID, "deform": rbfsl.VEL_DEFORM_Y2, "nl": rbfsl.VEL_NL}
_PREC = {"f64": rbfsl.FP64, "mixed": rbfsl.MIXED}
_NSET = (642, 1200, 2562, 5121, 10242)


def _vel_params(kind, rng):
    if kind == "rigid":
        return inputs.rigid_rotation_params(inputs.random_unit_vectors(1, rng)[0], 1.0)
    if kind == "deform":
        return inputs.deformation_params(float(rng.uniform(1.5, 2.4)), 1.0)
    return inputs.nl_deformation_params(5.0)


def _fields(X, T, rng):
    """Two kinds of tracer in turn: Gaussian hills and smooth random fields (max |q| ~ 1)."""
    q = np.empty((X.shape[0], T))
    for t in range(T):
        if t % 2 == 0:
            q[:, t] = 0.1 + inputs.gaussian_hills(X, inputs.random_unit_vectors(2, rng), 5.0, 0.9)
        else:
            f = inputs.plane_wave_field(rng, 6.0)(X)
            q[:, t] = f / np.abs(f).max()
    return q


def _eps(case):
    # shape parameters that grow with sqrt(N): the conditioning does not depend on N
    return (0.16 if case["kernel"] == "gauss" else 0.10) * math.sqrt(case["N"])


def _single(case, seed):
    """Nodes, field, velocity and start time of a single-problem case (host arrays)."""
    rng = np.random.default_rng([seed, case["N"], case["T"]])
    X = inputs.nodes(case["N"], int(rng.integers(1 << 31)))
    return dict(X=X, q=_fields(X, case["T"], rng), vp=_vel_params(case["vel"], rng),
                dt=(1.0 / 600 if case["vel"] == "deform" else 1.0 / 100 if case["vel"] == "rigid" else 5.0 / 50),
                t0=float(rng.uniform(0.0, 0.3)))


def _centers(N, n):
    return inputs.fibonacci_nodes(int(math.ceil(2.5 * N / n)))


def _problems(case, seed):
    """Descriptors of the independent problems of a batch (as inputs.batched_problems draws them)."""
    rng = np.random.default_rng([seed, case["P"]])
    Ns = [v for v in _NSET if v <= case["nmax"]]
    out = []
    for d in range(case["P"]):
        n, ell = [(31, 2), (55, 3), (84, 4)][d % 3]
        vel = ["rigid", "deform"][int(rng.integers(2))]
        N = Ns[(d * 2 + d // 3) % len(Ns)]
        X = inputs.nodes(N, int(rng.integers(1 << 31)))
        T = 1 + (5 * d) % 16
        out.append(dict(X=X, q=_fields(X, T, rng), n=n, ell=ell, power=2 * ell + 1,
                        mode="center" if d % 4 == 3 else "direct", vel=vel, vp=_vel_params(vel, rng), dt=1.0 / 100,
                        t0=0.0))
    return out


def _requests(case, seed):
    rng = np.random.default_rng([seed, case["R"]])
    Ns = [v for v in _NSET if v <= case["nmax"]]
    out = []
    for d in range(case["R"]):
        N = Ns[d % len(Ns)]
        X = inputs.nodes(N, int(rng.integers(1 << 31)))
        T = 1 + (3 * d) % 16
        vel = ["rigid", "deform"][d % 2]
        r = dict(X=X, q=_fields(X, T, rng), vel=vel, vp=_vel_params(vel, rng), dt=1.0 / 100, t0=0.0,
                 steps=case["steps"] + d % 3)
        if d % 3 == 2:
            r.update(method="pu", n=100 if N >= 2562 else 60, ell=3, power=7)
        else:
            n, ell = [(31, 2), (55, 3), (84, 4)][(d // 3) % 3]
            r.update(method="local", n=n, ell=ell, power=2 * ell + 1, mode="center" if d % 4 == 1 else "direct")
        out.append(r)
    return out


# ------------------------------------------------------------------------------- one pass
def prepare(case, seed):
    if case["kind"] == "batch":
        probs = _problems(case, seed)
        stream = torch.cuda.Stream()
        b = rbfsl.Batch(0, stream=stream)
        ids = [b.add(p["X"], p["q"], p["n"], p["ell"], p["power"], _VEL[p["vel"]], p["vp"], p["dt"],
                     mode=rbfsl.CENTER if p["mode"] == "center" else rbfsl.DIRECT, precision=_PREC[case["precision"]],
                     t0=p["t0"]) for p in probs]
        b.step(0)  # the problem table
        return dict(kind="batch", b=b, ids=ids, stream=stream, steps=case["steps"])
    if case["kind"] == "serve":
        return dict(kind="serve", s=rbfsl.Server(0, budget_bytes=40 * 10 ** 9, max_slots=32),
                    reqs=_requests(case, seed), precision=_PREC[case["precision"]])
    p = _single(case, seed)
    c = rbfsl.Context(0)
    c.set_nodes(p["X"])
    c.set_velocity(_VEL[case["vel"]], p["vp"])
    if case["kind"] == "local":
        c.set_method(rbfsl.LOCAL, rbfsl.CENTER if case["mode"] == "center" else rbfsl.DIRECT)
    else:
        c.set_method(rbfsl.PU if case["kind"] == "pu" else rbfsl.GLOBAL)
    if case["kind"] in ("local", "pu"):
        c.set_stencil_size(case["n"])
        c.set_sh_degree(case["ell"])
        c.set_kernel(rbfsl.PHS, case["power"])
    else:
        c.set_kernel(rbfsl.GAUSS if case["kernel"] == "gauss" else rbfsl.IMQ, _eps(case))
    if case["kind"] == "pu":
        c.set_pu(_centers(case["N"], case["n"]))
    if case["kind"] == "card":
        c.set_global_form(rbfsl.GLOBAL_CARDINAL)
    c.set_precision(_PREC[case["precision"]])
    c.set_dt(p["dt"])
    c.set_time(p["t0"])
    q = torch.from_numpy(p["q"]).to(DEV)
    c.set_tracers(q)
    c.step(0)  # index, factors: set up once
    # the tensor-core evaluation's results are FP32 numbers; the other forms keep FP64 accuracy
    dt = torch.float32 if case["kind"] == "global" and case["precision"] == "mixed" else torch.float64
    return dict(kind="ctx", c=c, q=q, t0=p["t0"], steps=case["steps"], out=torch.empty_like(q, dtype=dt))


def run(state):
    if state["kind"] == "batch":
        state["b"].step(state["steps"])
        return [state["b"].get_q(i) for i in state["ids"]]
    if state["kind"] == "serve":
        s = state["s"]
        tickets = []
        for r in state["reqs"]:
            kw = dict(method=rbfsl.PU, centers=_centers(len(r["X"]), r["n"])) if r["method"] == "pu" else \
                dict(mode=rbfsl.CENTER if r["mode"] == "center" else rbfsl.DIRECT)
            tickets.append(s.submit(r["X"], r["q"], r["n"], r["ell"], r["power"], _VEL[r["vel"]], r["vp"], r["dt"],
                                    r["steps"], precision=state["precision"], t0=r["t0"], **kw))
        s.wait_idle()
        return [s.result(t)[0] for t in tickets]
    c = state["c"]
    c.set_time(state["t0"])
    c.set_tracers(state["q"])
    c.step(state["steps"])
    return c.get_q(state["out"])


# ------------------------------------------------------------------------------- what a pass needs
def _local_work(N, n, ell, T, steps, center):
    m = n + (ell + 1) ** 2
    # direct: assemble and factorise one symmetric m x m system per node; centre: read its stored
    # triangular factor and substitute
    flops = 2.0 * m * m if center else m ** 3 / 3.0 + 2.0 * m * m
    byts = 16.0 * T + 24 + (4.0 * m * (m + 1) if center else 0)
    return N * steps * (byts), N * steps * (flops + 2.0 * n * T)


def _pu_work(N, n, ell, T, steps):
    m = n + (ell + 1) ** 2
    Mp = math.ceil(2.5 * N / n)
    return steps * (8.0 * Mp * m * m + N * (16.0 * T + 24)), steps * (2.0 * Mp * m * m * T + 2.5 * N * m * (2.0 * T + 15))


def work(case):
    k = case["kind"]
    if k == "local":
        b, f = _local_work(case["N"], case["n"], case["ell"], case["T"], case["steps"], case["mode"] == "center")
    elif k == "pu":
        b, f = _pu_work(case["N"], case["n"], case["ell"], case["T"], case["steps"])
    elif k == "global":
        N, T = case["N"], case["T"]
        b, f = case["steps"] * (8.0 * N * N + 16.0 * N * T), case["steps"] * (4.0 * N * N * T + 20.0 * N * N)
    elif k == "card":
        N, T = case["N"], case["T"]
        b, f = case["steps"] * (8.0 * N * N + 16.0 * N * T), case["steps"] * 2.0 * N * N * T
    elif k == "batch":
        b = f = 0.0
        for d in _shapes_batch(case):
            x, y = _local_work(*d)
            b, f = b + x, f + y
    else:
        b = f = 0.0
        for m, d in _shapes_serve(case):
            x, y = _pu_work(*d) if m == "pu" else _local_work(*d)
            b, f = b + x, f + y
    return {"bytes": b, "flops": f}


def _shapes_batch(case):
    return [(len(p["X"]), p["n"], p["ell"], p["q"].shape[1], case["steps"], p["mode"] == "center")
            for p in _problems(case, 0)]


def _shapes_serve(case):
    return [(r["method"], (len(r["X"]), r["n"], r["ell"], r["q"].shape[1], r["steps"]) +
             (() if r["method"] == "pu" else (r["mode"] == "center",))) for r in _requests(case, 0)]


# ------------------------------------------------------------------------------- plain FP64
def _velocity(kind, vp, P, t):
    x, y, z = P[:, 0], P[:, 1], P[:, 2]
    if kind == "rigid":
        return vp[3] * torch.linalg.cross(torch.as_tensor(np.array(vp[:3]), device=P.device).expand_as(P), P)
    if kind == "deform":
        g = 2.0 * vp[0] * y * math.cos(math.pi * t / vp[1])
        return torch.stack([-g * z, torch.zeros_like(y), g * x], 1)
    c = 2.0 * math.pi * t / vp[1]
    b, k = y * math.cos(c) - x * math.sin(c), 2.0 * vp[0] * math.cos(math.pi * t / vp[1])
    grad = torch.stack([-k * b * math.sin(c), k * b * math.cos(c), torch.full_like(x, -2.0 * math.pi / vp[1])], 1)
    return torch.linalg.cross(P, grad)


def _departure(kind, vp, X, t1, dt):
    unit = torch.nn.functional.normalize
    k1 = _velocity(kind, vp, X, t1)
    k2 = _velocity(kind, vp, unit(X - 0.5 * dt * k1, dim=1), t1 - 0.5 * dt)
    k3 = _velocity(kind, vp, unit(X - 0.5 * dt * k2, dim=1), t1 - 0.5 * dt)
    k4 = _velocity(kind, vp, unit(X - dt * k3, dim=1), t1 - dt)
    return unit(X - dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4), dim=1)


def _harmonics(ell, P):
    """A basis of the polynomials of degree <= ell on the sphere (any basis gives the same interpolant)."""
    x, y, z = P[..., 0], P[..., 1], P[..., 2]
    out, c, s = [], torch.ones_like(x), torch.zeros_like(x)
    for m in range(ell + 1):
        if m:
            c, s = c * x - s * y, c * y + s * x
        a, b = torch.zeros_like(x), torch.full_like(x, float(np.prod(np.arange(1, 2 * m, 2))) if m else 1.0)
        for l in range(m, ell + 1):
            if l > m:
                a, b = b, ((2 * l - 1) * z * b - (l + m - 1) * a) / (l - m)
            k = math.sqrt((1 if m == 0 else 2) * (2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            out += [k * b * c] + ([k * b * s] if m else [])
    return torch.stack(out, -1)


def _dist(A, B):
    d = A.unsqueeze(-2) - B.unsqueeze(-3)
    return torch.linalg.vector_norm(d, dim=-1)


def _sqdist(A, B):
    d = (A[:, None, 0] - B[None, :, 0]) ** 2
    for i in (1, 2):
        d += (A[:, None, i] - B[None, :, i]) ** 2
    return d


def _nearest(X, P, k):
    out = [torch.topk(_sqdist(P[a:a + 1024], X), k, dim=1, largest=False).indices for a in range(0, len(P), 1024)]
    return torch.cat(out)


def _local_weights(X, P, n, ell, power, center):
    S = _nearest(X, X, n)[_nearest(X, P, 1)[:, 0]] if center else _nearest(X, P, n)
    W = torch.empty(len(P), n, dtype=torch.float64, device=X.device)
    M = (ell + 1) ** 2
    for a in range(0, len(P), 4096):
        Y, p = X[S[a:a + 4096]], P[a:a + 4096, None]
        H = _harmonics(ell, Y)
        A = torch.cat([torch.cat([_dist(Y, Y) ** power, H], 2),
                       torch.cat([H.mT, H.new_zeros(len(Y), M, M)], 2)], 1)
        b = torch.cat([_dist(p, Y)[:, 0] ** power, _harmonics(ell, p)[:, 0]], 1)
        W[a:a + 4096] = torch.linalg.solve(A, b)[:, :n]
    return S, W


def _local_run(p, mode, n, ell, power, steps, X, q):
    t, S = p["t0"], None
    for _ in range(steps):
        if S is None or p["vel"] != "rigid":
            S, W = _local_weights(X, _departure(p["vel"], p["vp"], X, t + p["dt"], p["dt"]), n, ell, power, mode == "center")
        q = torch.cat([torch.einsum("ij,ijt->it", W[a:a + 8192], q[S[a:a + 8192]]) for a in range(0, len(X), 8192)])
        t += p["dt"]
    return q


def _pu_run(p, n, ell, power, steps, X, q):
    N = len(X)
    R = 2.0 * math.sqrt(n / N)
    C = torch.from_numpy(_centers(N, n)).to(X.device)
    members = [torch.nonzero(c)[:, 0] for c in _sqdist(C, X) < R * R]
    M = (ell + 1) ** 2
    t = p["t0"]
    fac = []
    for I in members:
        H = _harmonics(ell, X[I])
        fac.append(torch.linalg.lu_factor(torch.cat([torch.cat([_dist(X[I], X[I]) ** power, H], 1),
                                                     torch.cat([H.T, H.new_zeros(M, M)], 1)], 0)))
    for _ in range(steps):
        P = _departure(p["vel"], p["vp"], X, t + p["dt"], p["dt"])
        own = _sqdist(C, P) < R * R
        num, den = torch.zeros_like(q), q.new_zeros(N, 1)
        for l, I in enumerate(members):
            j = torch.nonzero(own[l])[:, 0]
            if not len(j):
                continue
            c = torch.linalg.lu_solve(*fac[l], torch.cat([q[I], q.new_zeros(M, q.shape[1])], 0))
            s = torch.cat([_dist(P[j], X[I]) ** power, _harmonics(ell, P[j])], 1) @ c
            r = (torch.linalg.vector_norm(P[j] - C[l], dim=1, keepdim=True) / R).clamp(max=1.0)
            w = (1 - r) ** 4 * (4 * r + 1)
            num.index_add_(0, j, w * s)
            den.index_add_(0, j, w)
        q = num / den
        t += p["dt"]
    return q


def _global_run(case, p, X, q):
    e = _eps(case)

    def phi(A, B):
        d2 = _sqdist(A, B)
        return torch.exp(-e * e * d2) if case["kernel"] == "gauss" else torch.rsqrt(1 + e * e * d2)

    F = torch.linalg.lu_factor(phi(X, X))
    t = p["t0"]
    for _ in range(case["steps"]):
        q = phi(_departure(p["vel"], p["vp"], X, t + p["dt"], p["dt"]), X) @ torch.linalg.lu_solve(*F, q)
        t += p["dt"]
    return q


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] in ("batch", "serve"):
            out = []
            for p in (_problems if case["kind"] == "batch" else _requests)(case, seed):
                X, q = torch.from_numpy(p["X"]).to(DEV), torch.from_numpy(p["q"]).to(DEV)
                steps = p.get("steps", case["steps"])
                q = _pu_run(p, p["n"], p["ell"], p["power"], steps, X, q) if p.get("method") == "pu" else \
                    _local_run(p, p["mode"], p["n"], p["ell"], p["power"], steps, X, q)
                out.append(q.cpu().numpy())
            return out
        p = _single(case, seed)
        p["vel"] = case["vel"]
        X, q = torch.from_numpy(p["X"]).to(DEV), torch.from_numpy(p["q"]).to(DEV)
        if case["kind"] == "local":
            return _local_run(p, case["mode"], case["n"], case["ell"], case["power"], case["steps"], X, q)
        if case["kind"] == "pu":
            return _pu_run(p, case["n"], case["ell"], case["power"], case["steps"], X, q)
        return _global_run(case, p, X, q)
