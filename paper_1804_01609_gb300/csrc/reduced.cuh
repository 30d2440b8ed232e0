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
// loads hide under them. From 16 harmonics on, the two large products (W A11 and W Y^T + Y W^T,
// 40% of those instructions) run on the tensor cores as exact sums of digit products (split_mma.cuh),
// closer to the exact product than FP64 sums. The serial parts (M pivot steps, K / 4 panels, each by
// warp 0 with the next step's search or panel ahead of the others' updates) are kept short because
// only four points share an SM at m = 109: reciprocals and square roots take their first iteration
// in FP32 arithmetic. N = 40,962, n = 84, ell = 4: the symmetric indefinite factorisation of the
// whole system (device_ops.cuh) 30.3 ms (FP64 pipe 80% busy); reduced form with FP64 products
// 24.4 ms, 9,817 FP64 warp instructions per point (85% busy); products on the tensor cores 18.5 ms,
// 6,138 (72%); panels of four columns instead of eight, digits formed once, split rows of W, the
// search ahead and the FP32 first iterations 15.7 ms, the digit sums made doubles by integers 15.0 ms.
#pragma once

#include "common.cuh"
#include "device_ops.cuh"
#include "split_mma.cuh"

namespace rbfsl {

constexpr int kRedPanel = 4;  // columns per panel of the L D L^T of B

// Whether the reduced form serves the system (B definite, at least one node besides the pivots).
__host__ __device__ inline bool reduced_form(int n, int ell, int half) {
    return half <= ell && n > (ell + 1) * (ell + 1);
}

// Whether the two large products run on the tensor cores: from 16 harmonics on (inner dimension at
// least one 16-deep MMA step). The rule looks at the system alone, so that every launch shape gives
// the same bits.
__host__ __device__ inline bool reduced_on_tensor(int M) { return M >= 16; }

// Offsets (doubles) of one point's shared region.
struct RedLayout {
    int S, S2;                       // column strides of P / W and of Y (odd: lanes along a row hit all banks)
    int A21, A11, B, C, dinv, ints;  // P at 0
    int total;
    __host__ __device__ RedLayout(int n, int M) {
        const int n1 = n + 1, K1 = n1 - M;
        S = n1 | 1;
        S2 = K1 | 1;
        const int y = M * S2 > 2 * kRedPanel * K1 ? M * S2 : 2 * kRedPanel * K1;  // Y, later two panels' columns
        A21 = M * S;
        A11 = A21 + y;
        B = A11 + M * (M - 1) / 2;
        C = B + K1 * (K1 + 1) / 2;
        dinv = C + 3 * n1;
        ints = dinv + M;
        total = ints + (n1 + 6 + 1) / 2;
    }
};

// Stored factors of one centre stencil in the reduced form (doubles): the M x M factor of P1
// (row-major: R above the diagonal, C below it, 1 / C_kk on it), then W, G = A21 - W A11 (K x M,
// column-major), W^T (row k of W after the other) and the triangles D^-1 L^-1 and L^-T of B = L D L^T:
// n^2 + K (M + 1) doubles, against the (n + M)^2 of an LU factor of the whole system.
// A triangle is folded, row i and row K - 1 - i in one column of K + 1 values, so that lanes along the
// columns have equal work: entry (i, j), j <= i, at fold(i, j); L^-T with both indexes reversed.
struct CenterLayout {
    int W, G, WT, T, H, K, total;  // H: columns of a folded triangle
    __host__ __device__ CenterLayout(int n, int M) {
        K = n - M;
        H = (K + 1) / 2;
        W = M * M;
        G = W + K * M;
        WT = G + K * M;
        T = WT + K * M;
        total = T + 2 * H * (K + 1);
    }
    __host__ __device__ int fold(int i, int j) const { return i < H ? j * H + i : (j + K - i) * H + K - 1 - i; }
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
// reciprocal square root y of v's leading bits (its exponent halved by integer operations). The
// first step runs in FP32 arithmetic on v's significand split into its leading 24 and its other 29
// bits, merged into an FP64 number by integer operations (~2^-43); the second in FP64, two
// operations. Zero, subnormal, extreme and non-finite v take the library's square root.
__device__ __forceinline__ double sqrt_heron(double v) {
    const long long b = __double_as_longlong(v);
    const int e = (int)(b >> 52);
    if (e < 128 || e > 1918) return sqrt(v);  // a negative v has its sign in e
    const int odd = (e - 1023) & 1, e2 = (e - 1023 - odd) / 2;
    const float scale = odd ? 2.0f : 1.0f;
    const float vh = scale * __int_as_float(0x3f800000 | (int)((b >> 29) & 0x7fffff));  // [1, 4)
    const float vl = (scale * 0x1p-52f) * (float)(int)(b & 0x1fffffff);
    const float y = rsqrtf(vh), gh = vh * y, h = 0.5f * y;
    const int add = __float2int_rn((fmaf(-gh, gh, vh) + vl) * h * 0x1p52f);
    const long long eb = (long long)(e2 + 1023 - 127) << 52;  // gh in [1, 2) up to rounding
    const double g = __longlong_as_double(eb + ((long long)__float_as_int(gh) << 29) + add);
    const double hd = __longlong_as_double(((long long)(1023 - 127 - e2) << 52) + ((long long)__float_as_int(h) << 29));
    return fma(fma(-g, g, v), hd, g);
}

// r^p = r (r^2)^half from r^2, the power by repeated squaring.
__device__ __forceinline__ double phs_pow(double d2, int half) {
    double v = sqrt_heron(d2), q = d2;
    for (int h = half; h > 0; h >>= 1) {
        if (h & 1) v *= q;
        if (h > 1) q *= q;
    }
    return v;
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
// kFactor: instead of weights, store the factors that centre stencils keep (CenterLayout; kFactorCenter)
// at F and the nodes' pivot order at order (p: any point, its row is not stored). kFactorPatch: L^-1 in the
// triangles' place (K x K, row-major) and D's diagonal in W^T's (K doubles).
constexpr int kNoFactor = 0, kFactorCenter = 1, kFactorPatch = 2;
template <int NW, bool kTensor, int kFactor = kNoFactor>
__device__ __forceinline__ int weights_point_reduced(double *__restrict__ R, const double *__restrict__ X,
                                                     const int32_t *__restrict__ stencil, int n, int M, int ell,
                                                     int half, double px, double py, double pz, int t,
                                                     double *&out, double *F = nullptr,
                                                     int32_t *order = nullptr) {
    constexpr int GT = NW * kWarp;
    const int warp = t >> 5, lane = t & 31;
    const int n1 = n + 1, K = n - M, K1 = K + 1;
    const RedLayout lay(n, M);
    const int S = lay.S, S2 = lay.S2;
    double *P = R, *Y = R + lay.A21, *A11 = R + lay.A11, *B = R + lay.B;
    double *cx = R + lay.C, *cy = cx + n1, *cz = cy + n1, *dinv = R + lay.dinv;
    int *st = reinterpret_cast<int *>(R + lay.ints), *ord = st + 6;
    // st[0]: error code, st[1]: breakdown, st[2..4]: largest exponent fields of W, A11 and Y
    auto gsync = [] {
        group_sync<NW>();
    };
    out = cx;
    if (t < 5) st[t] = 0;
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
    // part in the pivot search. Warp 0 interchanges and scales the pivot row, then updates the next
    // column and searches it while the other warps update the rest.
    long long pkey = 0;
    int p = 0;
    double di = 0.0;
    auto search = [&](int k) {
        pkey = 0;
        p = n;
        for (int i = k + lane; i < n; i += kWarp) {
            const long long b = __double_as_longlong(P[k * S + i]) & 0x7fffffffffffffffLL;
            if (b > pkey || p == n) { pkey = b; p = i; }
        }
        warp_max_key_row(pkey, p);
        const double d = P[k * S + p];
        di = recip_nr(d);
        if (lane == 0 && zero_or_not_finite(d)) st[1] = 1;
        __syncwarp();
    };
    if (warp == 0) search(0);
    gsync();
    for (int k = 0; k < M; ++k) {
        if (st[1]) return 1;  // set by a search, which is always between two barriers without this test
        if (warp == 0) {
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
            }
        }
        gsync();
        if (k + 1 == M) break;
        const int rows = n - k;
        if (warp == 0) {
            const double r = P[(k + 1) * S + k];
            for (int i = k + 1 + lane; i <= n; i += kWarp)
                P[(k + 1) * S + i] = fma(-P[k * S + i], r, P[(k + 1) * S + i]);
            __syncwarp();
            search(k + 1);
        }
        if (NW == 1 || warp > 0) {
            constexpr int step = NW == 1 ? kWarp : GT - kWarp;
            const int E = rows * (M - 2 - k);
            const float inv = 1.0f / (float)rows;
            for (int e = NW == 1 ? t : t - kWarp; e < E; e += step) {
                const int c = (int)(((float)e + 0.5f) * inv);
                const int j = k + 2 + c, i = k + 1 + (e - c * rows);
                P[j * S + i] = fma(-P[k * S + i], P[j * S + k], P[j * S + i]);
            }
        }
        gsync();
    }
    // ---- W = C2 C1^-1 by rows (rows M..n of P; the last is u): kSplit lanes of one warp share a
    // row's columns, so that all the warps of a large system take part
    constexpr int kSplit = NW == 1 ? 1 : 2, kRows = kWarp / kSplit;
    int emax = 0;
    for (int r0 = warp * kRows; r0 < K1; r0 += NW * kRows) {
        const int r = r0 + lane % kRows, h = lane / kRows;
        const bool on = r < K1;
        double *row = P + M + (on ? r : 0);
        for (int k = M - 1; k >= 0; --k) {
            const double w = row[k * S] * dinv[k];
            if (kSplit > 1) __syncwarp();  // both lanes of a row have read it
            if (on) {
                if (h == 0) row[k * S] = w;
                if (kTensor) emax = max(emax, exp_field(w));
#pragma unroll 4
                for (int j = h; j < k; j += kSplit) row[j * S] = fma(-w, P[j * S + k], row[j * S]);
            }
            if (kSplit > 1) __syncwarp();
        }
    }
    if (kTensor) {
        emax = __reduce_max_sync(0xffffffffu, emax);
        if (lane == 0) atomicMax(&st[2], emax);
        emax = 0;
    }
    // ---- kernel values of all pairs of points, in pivot order
    for (int e = t; e < n1 * n / 2; e += GT) {
        const int i = tri_row(e) + 1, j = e - tri(i - 1);
        const double dx = cx[i] - cx[j], dy = cy[i] - cy[j], dz = cz[i] - cz[j];
        const double d2 = fma(dz, dz, fma(dy, dy, dx * dx));
        if (__double_as_longlong(d2) == 0 && i < n) st[0] = RBFSL_ESINGULAR;  // two coincident nodes: two equal rows
        const double v = phs_pow(d2, half);
        if (i < M) {
            A11[tri(i - 1) + j] = v;
            if (kTensor) emax = max(emax, exp_field(v));
        } else if (j < M) Y[j * S2 + i - M] = v;
        else B[tri(i - M) + j - M] = v;
    }
    for (int r = t; r < K; r += GT) B[tri(r) + r] = 0.0;
    if (kTensor) {
        emax = __reduce_max_sync(0xffffffffu, emax);
        if (lane == 0) atomicMax(&st[3], emax);
    }
    gsync();
    if (st[0]) return st[0];
    const CenterLayout fl(n, M);
    if (kFactor) {  // P1's factor (reciprocal diagonal), W and its transpose, the order
        for (int e = t; e < M * M; e += GT) {
            const int k = e / M, j = e - k * M;
            F[e] = j == k ? dinv[k] : P[j * S + k];
        }
        for (int e = t; e < M * K; e += GT) {
            const int k = e / K, i = e - k * K;
            const double w = P[k * S + M + i];
            F[fl.W + e] = w;
            if (kFactor == kFactorCenter) F[fl.WT + i * M + k] = w;
        }
        for (int i = t; i < n; i += GT) order[i] = ord[i];
        if (kTensor) gsync();
    }
    // A21 - W A11 = 2 Y - A21, with A21 formed again
    auto store_g = [&] {
        for (int e = t; e < M * K; e += GT) {
            const int k = e / K, i = e - k * K, r = M + i;
            const double dx = cx[r] - cx[k], dy = cy[r] - cy[k], dz = cz[r] - cz[k];
            F[fl.G + e] = fma(2.0, Y[k * S2 + i], -phs_pow(fma(dz, dz, fma(dy, dy, dx * dx)), half));
        }
        gsync();
    };
    const double *W = P + M;  // W[k * S + r]
    const int EW = kTensor ? st[2] + 1 : 0;
    if (kTensor) {
        // ---- Y = A21 - W A11 / 2 and B = A22 - W Y^T - Y W^T on the tensor cores (split_mma.cuh):
        // W, A11 and Y replaced by their digits, 16 x 8 tiles dealt to the warps
        const int EA = st[3] + 1;
        if (EW >= 0x800 || EA >= 0x800 || !split_scale_ok(EW, EA)) return 1;  // not finite, or out of range
        const unsigned long long zero = 0x8080808080808080ULL;
        unsigned long long *Wd = reinterpret_cast<unsigned long long *>(P + M);
        unsigned long long *Ad = reinterpret_cast<unsigned long long *>(A11);
        unsigned long long *Yd = reinterpret_cast<unsigned long long *>(Y);
        const int tm = (K1 + 15) / 16, g = lane >> 2, c2 = (lane & 3) * 2;
        const float inv = 1.0f / (float)K1;
        // an M x K1 array with column stride ld
        auto to_digits = [&](double *a, int ld, int E) {
            for (int e = t; e < K1 * M; e += GT) {
                const int c = (int)(((float)e + 0.5f) * inv), r = e - c * K1;
                reinterpret_cast<unsigned long long *>(a)[c * ld + r] = digits_of(a[c * ld + r], E);
            }
        };
        to_digits(P + M, S, EW);
        for (int e = t; e < M * (M - 1) / 2; e += GT) Ad[e] = digits_of(A11[e], EA);
        gsync();
        emax = 0;
        {
            const double sc = split_scale(EW, EA);
            for (int tile = warp; tile < tm * ((M + 7) / 8); tile += NW) {
                const int i0 = (tile % tm) * 16, j0 = (tile / tm) * 8, j = j0 + g;
                float acc[kGroups][4] = {};
                for (int k0 = 0; k0 < M; k0 += 16)
                    split_mma(
                        acc, lane,
                        [&](int r, int k) {
                            r += i0;
                            k += k0;
                            return r < K1 && k < M ? Wd[k * S + r] : zero;
                        },
                        [&](int k) {
                            k += k0;
                            return k < M && j < M && k != j ? Ad[k > j ? tri(k - 1) + j : tri(j - 1) + k] : zero;
                        });
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int r = i0 + g + 8 * (u >> 1), c = j0 + c2 + (u & 1);
                    if (r < K1 && c < M) {
                        const double y = fma(split_value(acc, u), -0.5 * sc, Y[c * S2 + r]);
                        Y[c * S2 + r] = y;
                        emax = max(emax, exp_field(y));
                    }
                }
                __syncwarp();
            }
        }
        emax = __reduce_max_sync(0xffffffffu, emax);
        if (lane == 0) atomicMax(&st[4], emax);
        gsync();
        const int EY = st[4] + 1;
        if (EY >= 0x800 || !split_scale_ok(EW, EY)) return 1;
        if (kFactor) store_g();
        to_digits(Y, S2, EY);
        gsync();
        const double sc = split_scale(EW, EY);
        int tile = 0;
        for (int mi = 0; mi < tm; ++mi) {
            for (int ni = 0; ni < 2 * (mi + 1) && 8 * ni < K1; ++ni, ++tile) {
                if (tile % NW != warp) continue;
                const int i0 = 16 * mi, j = 8 * ni + g;
                float acc[kGroups][4] = {};
                for (int k0 = 0; k0 < M; k0 += 16) {
                    auto wd = [&](int r, int k) { return r < K1 && k + k0 < M ? Wd[(k + k0) * S + r] : zero; };
                    auto yd = [&](int r, int k) { return r < K1 && k + k0 < M ? Yd[(k + k0) * S2 + r] : zero; };
                    split_mma(acc, lane, [&](int r, int k) { return wd(i0 + r, k); }, [&](int k) { return yd(j, k); });
                    split_mma(acc, lane, [&](int r, int k) { return yd(i0 + r, k); }, [&](int k) { return wd(j, k); });
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int r = i0 + g + 8 * (u >> 1), c = 8 * ni + c2 + (u & 1);
                    if (r < K1 && c <= r && c < K) B[tri(r) + c] = fma(split_value(acc, u), -sc, B[tri(r) + c]);
                }
                __syncwarp();
            }
        }
    } else {
        // ---- the same on the FP64 pipe, flat element ranges
        const float inv = 1.0f / (float)K1;
        for (int e = t; e < K1 * M; e += GT) {
            const int c = (int)(((float)e + 0.5f) * inv), r = e - c * K1;
            double acc = 0.0;
            for (int k = 0; k < c; ++k) acc = fma(W[k * S + r], A11[tri(c - 1) + k], acc);
            for (int k = c + 1; k < M; ++k) acc = fma(W[k * S + r], A11[tri(k - 1) + c], acc);
            Y[c * S2 + r] = fma(-0.5, acc, Y[c * S2 + r]);
        }
        gsync();
        if (kFactor) store_g();
        // (lower triangle and the point's row; the point's own diagonal entry is unused)
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
    }
    gsync();
    // ---- B = L D L^T without interchanges, panels of kRedPanel columns (U: a panel's columns
    // before scaling, two panels in turn): all warps bring the next panel's columns up to date, then
    // warp 0 factorises them while the others update the columns behind them
    const long long neg = (half & 1) ? 0LL : 1LL;  // sign of B: (-1)^(half + 1)
    // columns [ja, jb) of the trailing triangle, threads th of nt, with the panel [k0, k0 + nb)
    auto trailing = [&](const double *U, int k0, int nb, int ja, int jb, int th, int nt) {
        auto update = [&](int i, int j) {
            const double *li = B + tri(i) + k0;
            double v = li[j - k0];
            if (nb == kRedPanel) {
#pragma unroll
                for (int c = 0; c < kRedPanel; ++c) v = fma(-li[c], U[c * K1 + j], v);
            } else {
                for (int c = 0; c < nb; ++c) v = fma(-li[c], U[c * K1 + j], v);
            }
            B[tri(i) + j] = v;
        };
        if (jb >= K) {  // the whole remaining triangle and the point's row (its corner unused)
            const int E = tri(K1 - ja) - 1;
            for (int e = th; e < E; e += nt) {
                const int q = tri_row(e);
                update(ja + q, ja + (e - tri(q)));
            }
        } else {
            // kRedPanel columns; the few entries above the diagonal are skipped
            for (int e = th; e < (K1 - ja) * kRedPanel; e += nt) {
                const int i = ja + e / kRedPanel, j = ja + e % kRedPanel;
                if (j <= i) update(i, j);
            }
        }
    };
    auto factor = [&](double *U, int k0, int nb) {
        for (int k = k0; k < k0 + nb; ++k) {
            const double d = B[tri(k) + k];
            if (lane == 0 && (zero_or_not_finite(d) ||
                              ((unsigned long long)__double_as_longlong(d) >> 63) != (unsigned long long)neg))
                st[1] = 1;
            double *u = U + (k - k0) * K1;
            for (int i = k + lane; i < K1; i += kWarp) u[i] = B[tri(i) + k];
            const double di = recip_nr(d);
            __syncwarp();
            for (int i = k + 1 + lane; i < K1; i += kWarp) {
                double *bi = B + tri(i);
                const double l = u[i] * di;
                bi[k] = l;
                const int je = i < k0 + nb ? i + 1 : k0 + nb;
                for (int j = k + 1; j < je; ++j) bi[j] = fma(-l, u[j], bi[j]);
            }
            __syncwarp();
        }
    };
    if (warp == 0) factor(Y, 0, K < kRedPanel ? K : kRedPanel);
    gsync();
    for (int k0 = 0, pb = 0; k0 < K; k0 += kRedPanel, pb ^= 1) {
        if (st[1]) return 1;
        const double *U = Y + pb * kRedPanel * K1;
        const int nb = K - k0 < kRedPanel ? K - k0 : kRedPanel, k1 = k0 + nb;
        if (k1 == K) break;
        const int k2 = k1 + kRedPanel < K ? k1 + kRedPanel : K;
        trailing(U, k0, nb, k1, k2, t, GT);
        gsync();
        if (NW == 1) {
            if (k2 < K) trailing(U, k0, nb, k2, K, t, GT);
            __syncwarp();
            factor(Y + (pb ^ 1) * kRedPanel * K1, k1, k2 - k1);
        } else if (warp == 0) {
            factor(Y + (pb ^ 1) * kRedPanel * K1, k1, k2 - k1);
        } else if (k2 < K) {
            trailing(U, k0, nb, k2, K, t - kWarp, GT - kWarp);
        }
        gsync();
    }
    if (kFactor) {
        // ---- L^-1, a thread per column, in place in global memory
        double *T1 = F + fl.T, *T2 = T1 + fl.H * (K + 1);
        for (int c = t; c < K; c += GT) {
            auto at = [&](int i) { return kFactor == kFactorPatch ? i * K + c : fl.fold(i, c); };
            for (int i = 0; i < K; ++i) {
                const double *li = B + tri(i);
                if (i < c) {
                    if (kFactor == kFactorPatch) T1[at(i)] = 0.0;
                    continue;
                }
                double a = i == c ? 1.0 : 0.0;
                for (int j = c; j < i; ++j) a = fma(-li[j], T1[at(j)], a);
                T1[at(i)] = a;
                if (kFactor == kFactorCenter) T2[fl.fold(K - 1 - c, K - 1 - i)] = a;
            }
            if (kFactor == kFactorPatch) {
                F[fl.WT + c] = B[tri(c) + c];
                continue;
            }
            for (int i = c; i < K; ++i) T1[at(i)] /= B[tri(i) + i];
        }
        if (kFactor == kFactorCenter && (K & 1))  // the middle row has a column to itself
            for (int e = fl.H + t; e <= K; e += GT) T1[e * fl.H + fl.H - 1] = T2[e * fl.H + fl.H - 1] = 0.0;
        return RBFSL_OK;
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
        auto w = [&](int i) { return kTensor ? from_digits(wk[i], EW) : wk[i]; };
        double a0 = w(K), a1 = 0.0;  // u
        int i = 0;
        for (; i + 1 < K; i += 2) {
            a0 = fma(-w(i), z[i], a0);
            a1 = fma(-w(i + 1), z[i + 1], a1);
        }
        if (i < K) a0 = fma(-w(i), z[i], a0);
        out[ord[k]] = a0 + a1;
    }
    for (int i = lane; i < K; i += kWarp) out[ord[M + i]] = z[i];
    __syncwarp();
    return RBFSL_OK;
}

// Weights of one point: the reduced form where it serves the system, else (and where it breaks
// down) the pivoted indefinite factorisation. Region and contract of both. kTensor: whether the
// kernel serves systems with the products on the tensor cores (reduced_on_tensor).
template <int NW, bool kTensor = true>
__device__ __forceinline__ int weights_point(double *__restrict__ R, const double *__restrict__ X,
                                             const int32_t *__restrict__ stencil, int n, int m, int ell, int half,
                                             double px, double py, double pz, int t, double *&out) {
    if (reduced_form(n, ell, half)) {
        const int M = m - n;
        const int rc = kTensor && reduced_on_tensor(M)
                           ? weights_point_reduced<NW, kTensor>(R, X, stencil, n, M, ell, half, px, py, pz, t, out)
                           : weights_point_reduced<NW, false>(R, X, stencil, n, M, ell, half, px, py, pz, t, out);
        if (rc <= 0) return rc;
        group_sync<NW>();  // every thread has read the breakdown flag
    }
    return weights_point_ldl<NW>(R, X, stencil, n, m, ell, half, px, py, pz, t, out);
}

// ---- Centre stencils (Sec. 3.3): the point uses the stencil of its nearest node, whose reduced
// factors are kept. Per point u = P1^-T Y(p) by substitution with P1's factor, g = phi_2 - W phi_1 -
// G u, w2 = L^-T (D^-1 L^-1 g) and w1 = u - W^T w2: the last form keeps the weights' polynomial part exact
// whatever the rounding of w2, and the products run without a serial chain across lanes. The inverse of
// B itself, one product of the same size, does not serve: on coarse node sets, where g is small against
// |B| |B^-1| |g|, its weights lost two digits (N = 642, n = 84: 2e-12 against 5e-14 for LU factors; the
// triangles 5e-14). kLanes lanes of a warp per point.
//
// Bound: the FP64 pipe (two thirds of the multiplications of substituting through an LU factor of
// the whole system, and a serial chain of 2 M steps instead of 2 (n + M)), then HBM (8 (n^2 + K (M + 1))
// bytes per point). N = 40,962, n = 84 0.97 ms against 2.33 ms, N = 163,842, n = 31 0.80 ms against
// 1.91 ms for the LU factors, which stay for the systems without the reduced form.

// Shared doubles of one point: P1's factor, phi (later z = D^-1 L^-1 g), Y(p), u, g (later w2) and the weights.
__host__ __device__ inline int center_reduced_doubles(int n, int M) { return M * M + 3 * n + M; }

// Lanes per point: half a warp where the products then leave fewer lanes idle (K <= 32, M <= 16:
// n = 31 has 22 and 9).
__host__ __device__ inline int center_lanes(int n, int M) { return M <= 16 && n - M <= 32 ? 16 : 32; }

// S: the stencil (n), F: its factors, order: pivot order; l: lane within the point's group. The
// other groups of the warp run the same steps. Returns the weights (shared, stencil order).
// kOwnY: whether the group evaluates the harmonics itself; else the caller has left them at
// sm + M * M + n, a barrier before the call.
template <int kLanes, bool kOwnY = true>
__device__ __forceinline__ double *center_point_reduced(const double *__restrict__ X, const int32_t *__restrict__ S,
                                                        const double *__restrict__ F,
                                                        const int32_t *__restrict__ order, int n, int M, int ell,
                                                        int half, double px, double py, double pz,
                                                        double *__restrict__ sm, int l) {
    const int K = n - M;
    const CenterLayout fl(n, M);
    double *LU = sm, *phi = LU + M * M, *y = phi + n, *u = y + M, *g = u + M, *out = g + K;
    for (int e = l; e < M * M; e += kLanes) LU[e] = F[e];
    for (int j = l; j < n; j += kLanes) {
        const int64_t s = S[order[j]];
        const double dx = px - X[3 * s], dy = py - X[3 * s + 1], dz = pz - X[3 * s + 2];
        phi[j] = phs_pow(fma(dz, dz, fma(dy, dy, dx * dx)), half);
    }
    if (kOwnY) sh_eval_lanes(ell, px, py, pz, l, [&](int c, double v) { y[c] = v; });
    __syncwarp();
    for (int k = 0; k < M; ++k) {  // y R^-1
        const double yk = y[k];
        for (int j = k + 1 + l; j < M; j += kLanes) y[j] = fma(-yk, LU[k * M + j], y[j]);
        __syncwarp();
    }
    for (int k = M - 1; k >= 0; --k) {  // then C^-1
        const double uk = y[k] * LU[k * M + k];
        if (l == 0) u[k] = uk;
        for (int j = l; j < k; j += kLanes) y[j] = fma(-uk, LU[k * M + j], y[j]);
        __syncwarp();
    }
    for (int i = l; i < K; i += kLanes) {
        const double *w = F + fl.W + i, *gg = F + fl.G + i;
        double a0 = phi[M + i], a1 = 0.0;
#pragma unroll 8
        for (int k = 0; k < M; ++k) {
            a0 = fma(-w[k * K], phi[k], a0);
            a1 = fma(-gg[k * K], u[k], a1);
        }
        g[i] = a0 + a1;
    }
    __syncwarp();
    // a folded triangle times x, two rows a lane: out(row, value)
    auto triangle = [&](const double *tr, auto x, auto out) {
        for (int c = l; c < fl.H; c += kLanes) {
            const double *p = tr + c;
            double a = 0.0, first = 0.0;
#pragma unroll 8
            for (int e = 0; e <= K; ++e) {
                a = fma(p[e * fl.H], x(e <= c ? e : e - c - 1), a);
                if (e == c) {
                    first = a;
                    a = 0.0;
                }
            }
            out(c, first);
            if (K - 1 - c != c) out(K - 1 - c, a);
        }
        __syncwarp();
    };
    triangle(F + fl.T, [&](int j) { return g[j]; }, [&](int i, double v) { phi[M + i] = v; });
    triangle(F + fl.T + fl.H * (K + 1), [&](int j) { return phi[M + K - 1 - j]; }, [&](int i, double v) {
        g[K - 1 - i] = v;
        out[order[M + K - 1 - i]] = v;
    });
    for (int k = l; k < M; k += kLanes) {
        const double *w = F + fl.WT + k, *z = g;
        double a0 = u[k], a1 = 0.0;
        int i = 0;
#pragma unroll 8
        for (; i + 1 < K; i += 2) {
            a0 = fma(-w[i * M], z[i], a0);
            a1 = fma(-w[(i + 1) * M], z[i + 1], a1);
        }
        if (i < K) a0 = fma(-w[i * M], z[i], a0);
        out[order[k]] = a0 + a1;
    }
    __syncwarp();
    return out;
}

}  // namespace rbfsl
