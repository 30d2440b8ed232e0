// Weights of the augmented local interpolant (Eqs. rbf_poly, rbf_poly_linsys) by elimination of
// the harmonics: the saddle-point system [[A, P], [P^T, 0]] [w; lambda] = [phi; Y] restricted to
// the null space of P^T, the form in which the PHS block is definite.
//
// The evaluation point is appended to the n stencil nodes as an (n+1)-th point. LU with partial
// pivoting of the harmonics' values at all of them picks M = (ell+1)^2 pivot nodes and gives
// W = P2 P1^-1 (every other point's values in the pivots' cardinal polynomials; the point's own
// row is u = P1^-T Y(p)). The reduced matrix
//     B = A22 - W Y^T - Y W^T,  Y = A21 - W A11 / 2        (= Z^T A Z, Z = [-W^T; I])
// over the K = n - M other nodes and the point has the right-hand side g as its last row, so an
// L D L^T of B without interchanges also does the forward substitution; then w2 = B^-1 g and
// w1 = u - W^T w2. For r^p with (p-1)/2 <= ell, r^p is conditionally definite of an order the
// harmonics cover and B is definite: no pivoting (Sec. 2.4's exponents satisfy it).
//
// Bound: the FP64 pipe, 16 cycles per warp instruction and SM whatever the number of active
// lanes, so the measure of every phase is FP64 warp instructions with full lanes; shared-memory
// loads (two per FMA) hide under them. Against the symmetric indefinite factorisation of the
// whole (n + M)-system (device_ops.cuh) the multiplications are as many, but they are in three
// products with flat element ranges and no pivot tests: M + K / 8 short serial steps instead of a
// tested pivot column per unknown. N = 40,962, n = 84, ell = 4: 9,817 FP64 warp instructions per
// point with the pipe 85% busy, 24.4 ms; the indefinite factorisation 30.3 ms (80% busy).
#pragma once

#include "common.cuh"
#include "device_ops.cuh"

namespace rbfsl {

constexpr int kRedPanel = 8;  // columns per panel of the L D L^T of B

// Whether the reduced form serves the system (B definite, at least one node besides the pivots).
__host__ __device__ inline bool reduced_form(int n, int ell, int half) {
    return half <= ell && n > (ell + 1) * (ell + 1);
}

// Offsets (doubles) of one point's shared region.
struct RedLayout {
    int S, S2;                       // column strides of P / W and of Y (odd: lanes along a row hit all banks)
    int A21, A11, B, C, dinv, ints;  // P at 0
    int total;
    __host__ __device__ RedLayout(int n, int M) {
        const int n1 = n + 1, K1 = n1 - M;
        S = n1 | 1;
        S2 = K1 | 1;
        const int y = M * S2 > kRedPanel * K1 ? M * S2 : kRedPanel * K1;  // Y, later a panel's columns
        A21 = M * S;
        A11 = A21 + y;
        B = A11 + M * (M - 1) / 2;
        C = B + K1 * (K1 + 1) / 2;
        dinv = C + 3 * n1;
        ints = dinv + M;
        total = ints + (n1 + 4 + 1) / 2;
    }
};

// Shared doubles of one point: the reduced form's region or the indefinite factorisation's (the
// path of systems without the reduced form, and of a point whose reduced matrix breaks down),
// whichever is larger.
__host__ __device__ inline int weights_doubles(int n, int m, int ell, int half) {
    const int ldl = ldl_doubles(n, m);
    if (!reduced_form(n, ell, half)) return ldl;
    const int red = RedLayout(n, m - n).total;
    return red > ldl ? red : ldl;
}

// sqrt(v) by Heron's iteration in residual form, g <- g + (v - g^2) / (2 sqrt v), from an FP32
// reciprocal square root of v's leading bits (its exponent halved by integer operations): two
// steps double the ~22 correct bits twice, five FP64 operations. Zero, subnormal, extreme and
// non-finite v take the library's square root.
__device__ __forceinline__ double sqrt_heron(double v) {
    const long long b = __double_as_longlong(v);
    const int e = (int)(b >> 52);
    if (e < 128 || e > 1918) return sqrt(v);  // a negative v has its sign in e
    const int odd = (e - 1023) & 1, e2 = (e - 1023 - odd) / 2;
    const float mf = __int_as_float(((127 + odd) << 23) | (int)((b >> 29) & 0x7fffff));  // [1, 4)
    const int yb = __float_as_int(rsqrtf(mf));
    const long long ye = (long long)((yb >> 23) - 127 - e2 + 1023);
    const long long y = (ye << 52) | ((long long)(yb & 0x7fffff) << 29);
    const double h = __longlong_as_double(y - (1LL << 52));
    double g = v * __longlong_as_double(y);
    g = fma(fma(-g, g, v), h, g);
    return fma(fma(-g, g, v), h, g);
}

__device__ __forceinline__ bool zero_or_not_finite(double v) {
    const long long b = __double_as_longlong(v) & 0x7fffffffffffffffLL;
    return b == 0 || b >= 0x7ff0000000000000LL;
}

// Weights of one point by a group of NW warps (thread t of the group) in the reduced form, in the
// region R (RedLayout). Each element gets the same operations whichever thread takes it, so any
// NW gives the same bits. Returns RBFSL_OK with the weights (n doubles, stencil order) in `out`
// (valid for warp 0), RBFSL_EKNN for a stencil index < 0, RBFSL_ESINGULAR for two coincident
// stencil nodes, and 1 where a pivot of P or of B vanishes, is not finite or has the wrong sign.
template <int NW>
__device__ __forceinline__ int weights_point_reduced(double *__restrict__ R, const double *__restrict__ X,
                                                     const int32_t *__restrict__ stencil, int n, int M, int ell,
                                                     int half, double px, double py, double pz, int t,
                                                     double *&out) {
    constexpr int GT = NW * kWarp;
    const int warp = t >> 5, lane = t & 31;
    const int n1 = n + 1, K = n - M, K1 = K + 1;
    const RedLayout lay(n, M);
    const int S = lay.S, S2 = lay.S2;
    double *P = R, *Y = R + lay.A21, *A11 = R + lay.A11, *B = R + lay.B;
    double *cx = R + lay.C, *cy = cx + n1, *cz = cy + n1, *dinv = R + lay.dinv;
    int *st = reinterpret_cast<int *>(R + lay.ints), *ord = st + 4;
    // st[0]: error code, st[1]: breakdown
    auto gsync = [] {
        if (NW == 1) __syncwarp(); else __syncthreads();
    };
    out = cx;
    if (t < 2) st[t] = 0;
    gsync();
    // ---- coordinates and harmonics, a thread per point
    for (int j = t; j < n1; j += GT) {
        double x = px, y = py, z = pz;
        if (j < n) {
            const int64_t s = stencil[j];
            if (s < 0) { st[0] = RBFSL_EKNN; continue; }  // a failed neighbour search leaves -1
            x = X[3 * s];
            y = X[3 * s + 1];
            z = X[3 * s + 2];
        }
        cx[j] = x;
        cy[j] = y;
        cz[j] = z;
        ord[j] = j;
        sh_eval(ell, x, y, z, [&](int c, double v) { P[c * S + j] = v; });
    }
    gsync();
    if (st[0]) return st[0];
    // ---- P = C R with C lower (rows interchanged) and R unit upper; the point's row n takes no
    // part in the pivot search. Warp 0 searches, interchanges and scales the pivot row.
    for (int k = 0; k < M; ++k) {
        if (warp == 0) {
            long long best = 0;
            int p = n;
            for (int i = k + lane; i < n; i += kWarp) {
                const long long b = __double_as_longlong(P[k * S + i]) & 0x7fffffffffffffffLL;
                if (b > best || p == n) { best = b; p = i; }
            }
            warp_max_key_row(best, p);
            const double d = P[k * S + p];
            __syncwarp();  // every lane has the pivot before the interchange moves it
            const double di = recip_nr(d);
            for (int c = lane; c < M; c += kWarp) {
                const double a = P[c * S + k], b = P[c * S + p];
                P[c * S + p] = a;
                P[c * S + k] = c > k ? b * di : b;
            }
            if (lane < 3) {
                double *q = lane == 0 ? cx : (lane == 1 ? cy : cz);
                const double a = q[k];
                q[k] = q[p];
                q[p] = a;
            } else if (lane == 3) {
                const int a = ord[k];
                ord[k] = ord[p];
                ord[p] = a;
                dinv[k] = di;
                if (zero_or_not_finite(d)) st[1] = 1;
            }
        }
        gsync();
        if (st[1]) return 1;
        const int rows = n - k, E = rows * (M - 1 - k);
        const float inv = 1.0f / (float)rows;
        for (int e = t; e < E; e += GT) {
            const int c = (int)(((float)e + 0.5f) * inv);
            const int j = k + 1 + c, i = k + 1 + (e - c * rows);
            P[j * S + i] = fma(-P[k * S + i], P[j * S + k], P[j * S + i]);
        }
        gsync();
    }
    // ---- W = C2 C1^-1, a thread per row (rows M..n of P; the last is u)
    for (int r = t; r < K1; r += GT) {
        double *row = P + M + r;
        for (int k = M - 1; k >= 0; --k) {
            const double w = row[k * S] * dinv[k];
            row[k * S] = w;
#pragma unroll 4
            for (int j = 0; j < k; ++j) row[j * S] = fma(-w, P[j * S + k], row[j * S]);
        }
    }
    // ---- kernel values of all pairs of points, in pivot order
    for (int e = t; e < n1 * n / 2; e += GT) {
        const int i = tri_row(e) + 1, j = e - tri(i - 1);
        const double dx = cx[i] - cx[j], dy = cy[i] - cy[j], dz = cz[i] - cz[j];
        const double d2 = fma(dz, dz, fma(dy, dy, dx * dx));
        if (d2 == 0.0 && i < n) st[0] = RBFSL_ESINGULAR;  // two coincident nodes: two equal rows
        double v = sqrt_heron(d2), q = d2;  // r^p = r (r^2)^half, the power by repeated squaring
        for (int h = half; h > 0; h >>= 1) {
            if (h & 1) v *= q;
            if (h > 1) q *= q;
        }
        if (i < M) A11[tri(i - 1) + j] = v;
        else if (j < M) Y[j * S2 + i - M] = v;
        else B[tri(i - M) + j - M] = v;
    }
    for (int r = t; r < K; r += GT) B[tri(r) + r] = 0.0;
    gsync();
    if (st[0]) return st[0];
    // ---- Y = A21 - W A11 / 2
    const double *W = P + M;  // W[k * S + r]
    {
        const float inv = 1.0f / (float)K1;
        for (int e = t; e < K1 * M; e += GT) {
            const int c = (int)(((float)e + 0.5f) * inv), r = e - c * K1;
            double acc = 0.0;
            for (int k = 0; k < c; ++k) acc = fma(W[k * S + r], A11[tri(c - 1) + k], acc);
            for (int k = c + 1; k < M; ++k) acc = fma(W[k * S + r], A11[tri(k - 1) + c], acc);
            Y[c * S2 + r] = fma(-0.5, acc, Y[c * S2 + r]);
        }
    }
    gsync();
    // ---- B = A22 - W Y^T - Y W^T (lower triangle and the point's row; its own diagonal is unused)
    for (int e = t; e < tri(K1) - 1; e += GT) {
        const int i = tri_row(e), j = e - tri(i);
        double v = B[e];
#pragma unroll 4
        for (int k = 0; k < M; ++k) {
            v = fma(-W[k * S + i], Y[k * S2 + j], v);
            v = fma(-Y[k * S2 + i], W[k * S + j], v);
        }
        B[e] = v;
    }
    gsync();
    // ---- B = L D L^T without interchanges, panels of kRedPanel columns: warp 0 factorises a
    // panel (U: its columns before scaling), all warps update the rest once per panel
    double *U = Y;
    const long long neg = (half & 1) ? 0LL : 1LL;  // sign of B: (-1)^(half + 1)
    for (int k0 = 0; k0 < K; k0 += kRedPanel) {
        const int nb = K - k0 < kRedPanel ? K - k0 : kRedPanel, k1 = k0 + nb;
        if (warp == 0) {
            for (int k = k0; k < k1; ++k) {
                const double d = B[tri(k) + k];
                if (lane == 0 && (zero_or_not_finite(d) ||
                                  ((unsigned long long)__double_as_longlong(d) >> 63) != (unsigned long long)neg))
                    st[1] = 1;
                const double di = recip_nr(d);
                double *u = U + (k - k0) * K1;
                for (int i = k + lane; i < K1; i += kWarp) u[i] = B[tri(i) + k];
                __syncwarp();
                for (int i = k + 1 + lane; i < K1; i += kWarp) {
                    double *bi = B + tri(i);
                    const double l = u[i] * di;
                    bi[k] = l;
                    const int je = i < k1 ? i + 1 : k1;
                    for (int j = k + 1; j < je; ++j) bi[j] = fma(-l, u[j], bi[j]);
                }
                __syncwarp();
            }
        }
        gsync();
        if (st[1]) return 1;
        const int Rr = K1 - k1, E = tri(Rr) - 1;
        for (int e = t; e < E; e += GT) {
            const int q = tri_row(e), i = k1 + q, j = k1 + (e - tri(q));
            const double *li = B + tri(i) + k0;
            double v = li[j - k0];
            if (nb == kRedPanel) {
#pragma unroll
                for (int c = 0; c < kRedPanel; ++c) v = fma(-li[c], U[c * K1 + j], v);
            } else {
                for (int c = 0; c < nb; ++c) v = fma(-li[c], U[c * K1 + j], v);
            }
            B[tri(i) + j] = v;
        }
        gsync();
    }
    if (warp != 0) return RBFSL_OK;
    // ---- L^T w2 = z (the last row of L), then w1 = u - W^T w2
    double *z = B + tri(K);
    for (int j = K - 1; j > 0; --j) {
        const double wj = z[j];
        const double *lj = B + tri(j);
        for (int i = lane; i < j; i += kWarp) z[i] = fma(-lj[i], wj, z[i]);
        __syncwarp();
    }
    for (int k = lane; k < M; k += kWarp) {
        const double *wk = W + k * S;
        double a0 = wk[K], a1 = 0.0;  // u
        int i = 0;
        for (; i + 1 < K; i += 2) {
            a0 = fma(-wk[i], z[i], a0);
            a1 = fma(-wk[i + 1], z[i + 1], a1);
        }
        if (i < K) a0 = fma(-wk[i], z[i], a0);
        out[ord[k]] = a0 + a1;
    }
    for (int i = lane; i < K; i += kWarp) out[ord[M + i]] = z[i];
    __syncwarp();
    return RBFSL_OK;
}

// Weights of one point: the reduced form where it serves the system, else (and where it breaks
// down) the pivoted indefinite factorisation. Region and contract of both.
template <int NW>
__device__ __forceinline__ int weights_point(double *__restrict__ R, const double *__restrict__ X,
                                             const int32_t *__restrict__ stencil, int n, int m, int ell, int half,
                                             double px, double py, double pz, int t, double *&out) {
    if (reduced_form(n, ell, half)) {
        const int rc = weights_point_reduced<NW>(R, X, stencil, n, m - n, ell, half, px, py, pz, t, out);
        if (rc <= 0) return rc;
        if (NW == 1) __syncwarp(); else __syncthreads();  // every thread has read the breakdown flag
    }
    return weights_point_ldl<NW>(R, X, stencil, n, m, ell, half, px, py, pz, t, out);
}

}  // namespace rbfsl
