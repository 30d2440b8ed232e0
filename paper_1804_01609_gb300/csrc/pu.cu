// RBF partition of unity (Sec. 2.3, Eqs. wght_func, bspline, pu_func, PU_interp; Sec. 3.3).
//
// Set-up: patches are the spherical caps |x - omega_l| < R around given centres; members are
// found by a radius query on the node grid and sorted by node index; each patch's augmented
// saddle-point matrix (Eq. rbf_poly_linsys, n_l nodes + (ell+1)^2 harmonics) is factorised
// once in FP64, reduced to the null space of the harmonics (reduced.cuh), or by LU with partial
// pivoting where a patch has no reduced form.
// Per step: (1) the patch coefficients [c; d] = A~_l^-1 [q(X_l); 0] for all tracers, one block
// per patch and 16 tracers; (2) for each evaluation point, the patches that contain it (radius
// query on the centre grid), their interpolants s_l (Eq. rbf_poly) blended with the weights
// phi(|p - omega_l| / R) / sum phi (Eq. pu_func).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "kernels.cuh"
#include "reduced.cuh"
#include "split_mma.cuh"

namespace rbfsl {

constexpr int kPuMaxMembers = RBFSL_MAX_SYSTEM - 16;  // ell = 3 leaves 144 nodes per patch
constexpr int kPuMaxCand = 256;                         // members gathered per patch
constexpr int kPuMaxPatches = 32;                       // patches containing one point

__device__ __forceinline__ double pu_phi(int kind, double r) {
    if (r >= 1.0) return 0.0;
    if (kind == 0) {  // Wendland C2
        const double a = 1.0 - r;
        return a * a * a * a * (4.0 * r + 1.0);
    }
    if (r < 0.5) return 2.0 / 3.0 + 4.0 * (r - 1.0) * r * r;  // cubic B-spline, Eq. bspline
    const double a = r - 1.0;
    return -4.0 / 3.0 * a * a * a;
}

// Patch membership: count (members == nullptr) or gather + sort (members != nullptr).
__global__ void __launch_bounds__(128) pu_members_kernel(KnnGrid g, const double *__restrict__ Om,
                                                         int64_t Mp, double R,
                                                         int32_t *__restrict__ counts,
                                                         const int64_t *__restrict__ mstart,
                                                         int32_t *__restrict__ members) {
    __shared__ int buf[4][kPuMaxCand];
    __shared__ int cnt[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t l = (int64_t)blockIdx.x * 4 + warp;
    if (l >= Mp) return;
    const double ox = Om[3 * l], oy = Om[3 * l + 1], oz = Om[3 * l + 2];
    if (lane == 0) cnt[warp] = 0;
    __syncwarp();
    grid_ball_foreach(g, ox, oy, oz, (float)R, lane, [&](int p, bool on) {
        if (on && sqrt(sqdist_rn(ox, oy, oz, g.sx[p], g.sy[p], g.sz[p])) < R) {
            const int slot = atomicAdd(&cnt[warp], 1);
            if (slot < kPuMaxCand) buf[warp][slot] = g.sid[p];
        }
    });
    __syncwarp();
    const int n = cnt[warp];
    if (!members) {
        if (lane == 0) counts[l] = n;
        return;
    }
    // sort the member indices ascending (bitonic, padded to a power of two)
    const int nn = min(n, kPuMaxCand);
    int P = 1;
    while (P < nn) P <<= 1;
    for (int i = nn + lane; i < P; i += 32) buf[warp][i] = 0x7fffffff;
    __syncwarp();
    for (int len = 2; len <= P; len <<= 1)
        for (int st = len >> 1; st > 0; st >>= 1) {
            for (int i = lane; i < P; i += 32) {
                const int j = i ^ st;
                if (j > i) {
                    const int a = buf[warp][i], b = buf[warp][j];
                    if ((a > b) == ((i & len) == 0)) { buf[warp][i] = b; buf[warp][j] = a; }
                }
            }
            __syncwarp();
        }
    const int64_t base = mstart[l];
    for (int i = lane; i < nn; i += 32) members[base + i] = buf[warp][i];
}

// Factorise patch l's saddle-point matrix (one block of 128 threads per patch).
__global__ void __launch_bounds__(128) pu_factor_kernel(const double *__restrict__ X,
                                                        const int64_t *__restrict__ mstart,
                                                        const int32_t *__restrict__ members,
                                                        const int64_t *__restrict__ lu_off, int M,
                                                        int ell, int half, double *__restrict__ LU,
                                                        int32_t *__restrict__ perm,
                                                        int32_t *__restrict__ status, int colmajor) {
    extern __shared__ double sm[];
    __shared__ int s_p, s_bad;
    __shared__ int order[RBFSL_MAX_SYSTEM];
    const int64_t l = blockIdx.x;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n = (int)(mstart[l + 1] - mstart[l]), m = n + M, ld = m | 1;
    const int32_t *I = members + mstart[l];
    double *A = sm, *cx = A + (size_t)m * ld, *cy = cx + n, *cz = cy + n;
    for (int j = t; j < n; j += 128) {
        const int64_t s = I[j];
        cx[j] = X[3 * s]; cy[j] = X[3 * s + 1]; cz[j] = X[3 * s + 2];
    }
    if (t == 0) s_bad = 0;
    for (int i = t; i < m; i += 128) order[i] = i;
    __syncthreads();
    const int P2 = n * (n - 1) / 2;
    for (int p = t; p < P2; p += 128) {
        const int f = p / (n - 1), e = p - f * (n - 1);
        int r, c;
        if (e < n - 1 - f) { r = f; c = f + 1 + e; } else { r = n - 1 - f; c = e + 1; }
        const double dx = cx[r] - cx[c], dy = cy[r] - cy[c], dz = cz[r] - cz[c];
        const double v = phs_from_d2(dx * dx + dy * dy + dz * dz, half);
        A[r * ld + c] = v;
        A[c * ld + r] = v;
    }
    for (int j = t; j < n; j += 128) {
        A[j * ld + j] = 0.0;
        sh_eval(ell, cx[j], cy[j], cz[j], [&](int c, double v) {
            A[j * ld + n + c] = v;
            A[(n + c) * ld + j] = v;
        });
    }
    for (int e = t; e < M * M; e += 128) A[(n + e / M) * ld + n + e % M] = 0.0;
    __syncthreads();
    for (int k = 0; k < m; ++k) {
        if (warp == 0) {
            long long best = -1;
            int bidx = m;
            for (int r = k + lane; r < m; r += 32) {
                const long long v = __double_as_longlong(A[r * ld + k]) & 0x7fffffffffffffffLL;
                if (v > best) { best = v; bidx = r; }
            }
            for (int off = 16; off > 0; off >>= 1) {
                const long long ob = __shfl_xor_sync(0xffffffffu, best, off);
                const int oi = __shfl_xor_sync(0xffffffffu, bidx, off);
                if (ob > best || (ob == best && oi < bidx)) { best = ob; bidx = oi; }
            }
            if (lane == 0) {
                if (best <= 0 || best >= 0x7ff0000000000000LL) { s_bad = 1; bidx = k; }
                s_p = bidx;
                if (bidx != k) { const int o = order[k]; order[k] = order[bidx]; order[bidx] = o; }
            }
        }
        __syncthreads();
        if (s_bad) break;
        const int p = s_p;
        if (p != k)
            for (int c = t; c < m; c += 128) {
                const double tmp = A[k * ld + c]; A[k * ld + c] = A[p * ld + c]; A[p * ld + c] = tmp;
            }
        __syncthreads();
        const double inv = 1.0 / A[k * ld + k];
        for (int r = k + 1 + t; r < m; r += 128) A[r * ld + k] *= inv;
        __syncthreads();
        const int rows = m - k - 1, cols = m - k - 1;
        for (int e = t; e < rows * cols; e += 128) {
            const int r = k + 1 + e / cols, c = k + 1 + e % cols;
            A[r * ld + c] = fma(-A[r * ld + k], A[k * ld + c], A[r * ld + c]);
        }
        __syncthreads();
    }
    if (s_bad) {
        if (t == 0) atomicAdd(status, 1);
        return;
    }
    double *out = LU + lu_off[l];
    if (!colmajor) {
        for (int e = t; e < m * m; e += 128) out[e] = A[(e / m) * ld + e % m];
    } else {  // column-major, upper columns scaled by the reciprocal diagonal, which is stored on
              // the diagonal (centre stencils: the backward substitution multiplies once per row)
        for (int e = t; e < m * m; e += 128) {
            const int c = e / m, r = e % m;
            const double inv = 1.0 / A[c * ld + c];
            out[e] = r == c ? inv : (r < c ? A[r * ld + c] * inv : A[r * ld + c]);
        }
    }
    int32_t *pr = perm + mstart[l] + l * M;
    for (int i = t; i < m; i += 128) pr[i] = order[i];
}

// One value of a field: FP64 or an FP32 pair.
__device__ __forceinline__ double field_value(double v) { return v; }
__device__ __forceinline__ double field_value(float2 v) { return (double)v.x + (double)v.y; }

// Patch coefficients for all tracers from LU factors (one block per patch): Y = P [q(X_l); 0], L U c = Y.
template <typename In, typename Out>
__global__ void __launch_bounds__(128) pu_coef_kernel(const int64_t *__restrict__ mstart,
                                                      const int32_t *__restrict__ members,
                                                      const int64_t *__restrict__ lu_off, int M,
                                                      const double *__restrict__ LU,
                                                      const int32_t *__restrict__ perm,
                                                      const In *__restrict__ q, int T,
                                                      Out *__restrict__ coef) {
    extern __shared__ double Y[];
    const int64_t l = blockIdx.x;
    const int t = threadIdx.x;
    const int n = (int)(mstart[l + 1] - mstart[l]), m = n + M;
    const int32_t *I = members + mstart[l];
    const int32_t *pr = perm + mstart[l] + l * M;
    const double *F = LU + lu_off[l];
    for (int e = t; e < m * T; e += 128) {
        const int i = e / T, c = e % T;
        const int src = pr[i];
        Y[e] = src < n ? field_value(q[(int64_t)I[src] * T + c]) : 0.0;
    }
    __syncthreads();
    for (int r = 0; r < m - 1; ++r) {  // unit lower
        for (int e = t; e < (m - 1 - r) * T; e += 128) {
            const int s = r + 1 + e / T, c = e % T;
            Y[s * T + c] = fma(-F[s * m + r], Y[r * T + c], Y[s * T + c]);
        }
        __syncthreads();
    }
    for (int r = m - 1; r >= 0; --r) {  // upper
        for (int c = t; c < T; c += 128) Y[r * T + c] /= F[r * m + r];
        __syncthreads();
        for (int e = t; e < r * T; e += 128) {
            const int s = e / T, c = e % T;
            Y[s * T + c] = fma(-F[s * m + r], Y[r * T + c], Y[s * T + c]);
        }
        __syncthreads();
    }
    Out *out = coef + (mstart[l] + l * M) * T;
    for (int e = t; e < m * T; e += 128) out[e] = wcast<Out>(Y[e]);
}

// ---- Coefficients from the reduced factors. With the nodes in pivot order (M pivots, K = n - M
// others), W = P2 P1^-1, G = A21 - W A11 and B = L D L^T the reduced matrix, [[A, P], [P^T, 0]] [c; d] =
// [f; 0] has
//     c2 = L^-T (D^-1 L^-1) (f2 - W f1),   c1 = -W^T c2,   P1 d = f1 - G^T c2,
// products without the 2 (n + M) dependent steps of a substitution, and P^T c = 0 holds by the form of
// c1 whatever the rounding of c2. L^-1 stays a factor: c2 is much smaller than |B^-1| |f2| for a smooth
// f, and a product with B^-1 itself was off by 2e-11 where L's substitutions and L^-1 give 3e-13
// (N = 1,203, n = 100). The five products run on the tensor cores as digit products (split_mma.cuh): the
// matrices are kept as the digits of their rows, each row with its own exponent, the right-hand sides are
// cut column by column, so that neither a row nor a tracer of small values loses digits to a larger one,
// and what is cut off is ~2^-61 of a row times a column.
//
// Bound: the substitution was a chain of 2 m barriers with strided reads of the factor (n = 84, T = 16,
// 1,220 patches: 597 us); now the factors' reads (8 bytes an entry, padded to 16 x 16 tiles
// stored in the order in which the lanes of an MMA take them), the FP64 pipe (the products' last steps, P1's substitution: 40 us) and each block's
// chain of five products: 154 us (n = 100, T = 2, 257 patches: 242, now 48).

// One patch's factors, in 8-byte words: W (K x M), D^-1 L^-1 and L^-T (K x K, the tiles of their
// triangles), G^T and W^T (M x K) in 16 x 16 tiles, the M x M factor of P1 (R above the
// diagonal, C with its columns divided by their diagonal entries below it, their reciprocals on it), the
// rows' exponents (int32, the five matrices in turn).
struct PatchLayout {
    int Kp, Mp, L, LT, G, WT, P1, E, total;  // W at 0
    __host__ __device__ PatchLayout(int n, int M) {
        Kp = (n - M + 15) / 16 * 16;
        Mp = (M + 15) / 16 * 16;
        L = Kp * Mp;
        LT = L + Kp * (Kp + 16) / 2;
        G = LT + Kp * (Kp + 16) / 2;
        WT = G + Kp * Mp;
        P1 = WT + Kp * Mp;
        E = P1 + M * M;
        total = (E + (3 * Kp + 2 * Mp + 1) / 2 + 31) / 32 * 32;
    }
};

constexpr int kPuTracers = 16;  // tracers per block
// the sums of digit products stay below 2^24: at most seven products of full digits (2^14) per weight
// beside two with a leading digit (|digit| <= 32)
static_assert((kPuMaxMembers - 1) * 7 <= 1024, "digit products of a patch exceed the FP32 accumulators");

// Reduced factors of patches l0 + blockIdx.x (CenterLayout, `stride` doubles apart). bad: patches without.
__global__ void __launch_bounds__(128, 4) pu_reduced_factor_kernel(const double *__restrict__ X,
                                                                   const int64_t *__restrict__ mstart,
                                                                   const int32_t *__restrict__ members, int64_t l0,
                                                                   int M, int ell, int half, int64_t stride,
                                                                   double *__restrict__ F, int32_t *__restrict__ perm,
                                                                   int32_t *__restrict__ bad) {
    extern __shared__ double sm[];
    const int64_t l = l0 + blockIdx.x;
    const int n = (int)(mstart[l + 1] - mstart[l]), t = threadIdx.x;
    const int32_t *I = members + mstart[l];
    const int64_t c = I[0];
    double *out = nullptr, *Fl = F + blockIdx.x * stride;
    int32_t *order = perm + mstart[l] + l * M;
    const int rc = reduced_on_tensor(M)
                       ? weights_point_reduced<4, true, kFactorPatch>(sm, X, I, n, M, ell, half, X[3 * c], X[3 * c + 1],
                                                              X[3 * c + 2], t, out, Fl, order)
                       : weights_point_reduced<4, false, kFactorPatch>(sm, X, I, n, M, ell, half, X[3 * c], X[3 * c + 1],
                                                               X[3 * c + 2], t, out, Fl, order);
    if (t == 0 && rc != RBFSL_OK) atomicAdd(bad, 1);
}

// The exponent E of the digits (digits_of: |x| < 2^(E - 1023), E >= 2) from the largest exponent field.
__device__ __forceinline__ int digits_exponent(int field) { return field + 1 < 2 ? 2 : field + 1; }

// Those factors as PatchLayout. bad: patches with an infinity or NaN.
__global__ void __launch_bounds__(128) pu_pack_kernel(const int64_t *__restrict__ mstart, int64_t l0, int M,
                                                      int64_t stride, const double *__restrict__ F,
                                                      const int64_t *__restrict__ off,
                                                      const int32_t *__restrict__ members,
                                                      const int32_t *__restrict__ perm,
                                                      unsigned long long *__restrict__ out,
                                                      int32_t *__restrict__ pmem, int32_t *__restrict__ bad) {
    const int64_t l = l0 + blockIdx.x;
    const int n = (int)(mstart[l + 1] - mstart[l]), K = n - M, t = threadIdx.x;
    const CenterLayout cl(n, M);
    const PatchLayout pl(n, M);
    const double *Fl = F + blockIdx.x * stride;
    unsigned long long *o = out + off[l];
    int32_t *E = reinterpret_cast<int32_t *>(o + pl.E);
    for (int i = t; i < n; i += 128) {
        const int k = perm[mstart[l] + l * M + i];
        pmem[mstart[l] + i] = k >= 0 && k < n ? members[mstart[l] + k] : 0;  // no order where the factors failed
    }
    // the tiles [first(row tile), last(row tile)) of a matrix of rows x cols entries a(r, k)
    auto pack = [&](int rows, int cols, int rows_p, auto first, auto last, unsigned long long *dst, int32_t *Er, auto a) {
        for (int r = t; r < rows_p; r += 128) {
            int f = 0;
            if (r < rows)
                for (int k = 0; k < cols; ++k) f = max(f, exp_field(a(r, k)));
            if (f == 0x7ff) atomicAdd(bad, 1);
            Er[r] = digits_exponent(f);
        }
        __syncthreads();
        for (int rt = 0; rt < rows_p / 16; ++rt) {
            const int kt0 = first(rt), words = (last(rt) - kt0) * 256;
            for (int e = t; e < words; e += 128) {
                // word e: a tile's x[j], x[j + 1] of every lane in turn (split_products)
                const int j = (e >> 6) & 3, lane = (e >> 1) & 31;
                const int r = rt * 16 + (lane >> 2) + 8 * (j >> 1);
                const int k = (kt0 + (e >> 8)) * 16 + (lane & 3) * 2 + 8 * (j & 1) + (e & 1);
                dst[e] = r < rows && k < cols ? digits_of(a(r, k), Er[r]) : kZeroDigits;
            }
            dst += words;
        }
    };
    const int tk = pl.Kp / 16, tm = pl.Mp / 16;
    auto zero = [](int) { return 0; };
    pack(K, M, pl.Kp, zero, [&](int) { return tm; }, o, E, [&](int r, int k) { return Fl[cl.W + k * K + r]; });
    pack(K, K, pl.Kp, zero, [](int rt) { return rt + 1; }, o + pl.L, E + pl.Kp,
         [&](int r, int k) { return Fl[cl.T + r * K + k] / Fl[cl.WT + r]; });
    pack(K, K, pl.Kp, [](int rt) { return rt; }, [&](int) { return tk; }, o + pl.LT, E + 2 * pl.Kp,
         [&](int r, int k) { return Fl[cl.T + k * K + r]; });
    pack(M, K, pl.Mp, zero, [&](int) { return tk; }, o + pl.G, E + 3 * pl.Kp, [&](int r, int k) { return Fl[cl.G + r * K + k]; });
    pack(M, K, pl.Mp, zero, [&](int) { return tk; }, o + pl.WT, E + 3 * pl.Kp + pl.Mp,
         [&](int r, int k) { return Fl[cl.W + r * K + k]; });
    double *P1 = reinterpret_cast<double *>(o + pl.P1);
    for (int e = t; e < M * M; e += 128) {
        const int r = e / M, c = e - r * M;
        P1[e] = r > c ? Fl[e] * Fl[c * M + c] : Fl[e];
    }
}

// Shared bytes of the coefficient kernel: per tracer K and M values twice (strides 8 mod 16 words:
// conflict-free 16-byte loads of the MMA's columns), and four exponents.
__host__ __device__ inline int pu_coef_bytes(int Kp, int Mp, int nc) {
    return nc * (2 * (Kp + 8) + 2 * (Mp + 8)) * 8 + 4 * kPuTracers * 4;
}

template <typename In, typename Out>
__global__ void __launch_bounds__(128, 5) pu_coef_reduced_kernel(const int64_t *__restrict__ mstart,
                                                                 const int32_t *__restrict__ pmem,
                                                                 const int64_t *__restrict__ off, int M,
                                                                 const unsigned long long *__restrict__ factors,
                                                                 const int32_t *__restrict__ perm,
                                                                 const In *__restrict__ q, int T,
                                                                 Out *__restrict__ coef) {
    extern __shared__ __align__(16) double sm[];
    const int64_t l = blockIdx.x;
    const int t0 = blockIdx.y * kPuTracers, tc = min(kPuTracers, T - t0);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int n = (int)(mstart[l + 1] - mstart[l]), K = n - M;
    const PatchLayout pl(n, M);
    const int nt = tc > 8 ? 2 : 1, nc = 8 * nt, S2 = pl.Kp + 8, S1 = pl.Mp + 8;
    const unsigned long long *A = factors + off[l];
    const double *P1 = reinterpret_cast<const double *>(A + pl.P1);
    const int32_t *Er = reinterpret_cast<const int32_t *>(A + pl.E);
    const int32_t *I = pmem + mstart[l], *ord = perm + mstart[l] + l * M;
    double *V = sm, *C2 = V + nc * S2, *H = C2 + nc * S2, *D = H + nc * S1;  // [tracer][row]
    int *E1 = reinterpret_cast<int *>(D + nc * S1), *E2 = E1 + kPuTracers, *E3 = E2 + kPuTracers,
        *E4 = E3 + kPuTracers;
    if (t < 4 * kPuTracers) E1[t] = 0;
    __syncthreads();
    // ---- f in pivot order: f1 in H, f2 in V, zeros for the missing tracers
    for (int e = t; e < n * tc; e += 128) {
        const int i = e / tc, c = e - i * tc;
        const double v = field_value(q[(int64_t)I[i] * T + t0 + c]);
        if (i < M) {
            H[c * S1 + i] = v;
            atomicMax(&E1[c], exp_field(v));
        } else {
            V[c * S2 + i - M] = v;
        }
    }
    for (int c = tc; c < nc; ++c) {
        for (int i = t; i < M; i += 128) H[c * S1 + i] = 0.0;
        for (int i = t; i < K; i += 128) V[c * S2 + i] = 0.0;
    }
    __syncthreads();
    // rows of nc columns at src as digits at dst (may be src), zeros behind them
    auto to_digits = [&](double *dst, const double *src, int S, int rows, int rows_p, const int *E) {
        for (int e = t; e < nc * rows_p; e += 128) {
            const int c = e / rows_p, r = e - c * rows_p;
            reinterpret_cast<unsigned long long *>(dst)[c * S + r] =
                r < rows ? digits_of(src[c * S + r], digits_exponent(E[c])) : kZeroDigits;
        }
    };
    auto pow2 = [](int e) { return __longlong_as_double((long long)(max(e, -1022) + 1023) << 52); };
    // 16 rows (row tile ri, exponents er) x 8 tracers from c0 of the product of the row's tiles at a, `tiles`
    // of them, and the digits at b from its row k0 on: out(row, tracer, value)
    auto product = [&](const unsigned long long *a, int tiles, const int32_t *er, const double *b, int S, int k0,
                       const int *eb, int ri, int c0, auto out) {
        const int g = lane >> 2, tt = (lane & 3) * 2;
        const ulonglong2 *ap = reinterpret_cast<const ulonglong2 *>(a) + lane;
        const double *bp = b + (c0 + g) * S + k0 + tt;
        float acc[kGroups][4] = {};
        ulonglong2 nx[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) nx[j] = ap[32 * j];
        for (int kt = 0; kt < tiles; ++kt) {
            const unsigned long long x[8] = {nx[0].x, nx[0].y, nx[1].x, nx[1].y, nx[2].x, nx[2].y, nx[3].x, nx[3].y};
            if (kt + 1 < tiles) {  // the next tile while this one is multiplied
                ap += 128;
#pragma unroll
                for (int j = 0; j < 4; ++j) nx[j] = ap[32 * j];
            }
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(bp + 16 * kt),
                             b1 = *reinterpret_cast<const ulonglong2 *>(bp + 16 * kt + 8);
            uint32_t bd[kDigits][2];
            digit_frags(bd, b0.x, b0.y, b1.x, b1.y);
            split_products(acc, x, bd);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = ri * 16 + g + 8 * (u >> 1), c = c0 + tt + (u & 1);
            const int ec = digits_exponent(eb[c]), e = er[r] + ec - 2 * 1023 - 34;
            double v = split_value(acc, u);
            if (ec > 0x7ff) v = (double)NAN;                       // an infinity or NaN in the column
            else if (e >= -1022 && e <= 1023) v *= pow2(e);
            else v = v * pow2(e >> 1) * pow2(e - (e >> 1));        // a scale outside a double's range
            out(r, c, v);
        }
    };
    // the largest exponent fields of two columns (this lane's, c0 + tt and the next) into E
    auto column_max = [&](int f0, int f1, int c0, int *E) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            f0 = max(f0, __shfl_xor_sync(0xffffffffu, f0, o));
            f1 = max(f1, __shfl_xor_sync(0xffffffffu, f1, o));
        }
        if (lane < 4) {
            const int c = c0 + 2 * lane;
            atomicMax(&E[c], f0);
            atomicMax(&E[c + 1], f1);
        }
    };
    const int tk = pl.Kp / 16, tm = pl.Mp / 16;
    Out *out = coef + (mstart[l] + l * M) * T + t0;
    // ---- g = f2 - W f1
    to_digits(D, H, S1, M, pl.Mp, E1);
    __syncthreads();
    for (int item = warp; item < tk * nt; item += 4) {
        const int ri = item / nt, c0 = item % nt * 8;
        int f[2] = {0, 0};
        product(A + ri * tm * 256, tm, Er, D, S1, 0, E1, ri, c0, [&](int r, int c, double v) {
            if (r >= K) return;
            const double g = V[c * S2 + r] - v;
            V[c * S2 + r] = g;
            f[c & 1] = max(f[c & 1], exp_field(g));
        });
        column_max(f[0], f[1], c0, E2);
    }
    __syncthreads();
    // ---- z = D^-1 L^-1 g, the longest rows first
    to_digits(V, V, S2, K, pl.Kp, E2);
    __syncthreads();
    for (int item = warp; item < tk * nt; item += 4) {
        const int ri = tk - 1 - item / nt, c0 = item % nt * 8;
        int f[2] = {0, 0};
        product(A + pl.L + ri * (ri + 1) / 2 * 256, ri + 1, Er + pl.Kp, V, S2, 0, E2, ri, c0, [&](int r, int c, double v) {
            if (r >= K) return;
            C2[c * S2 + r] = v;
            f[c & 1] = max(f[c & 1], exp_field(v));
        });
        column_max(f[0], f[1], c0, E3);
    }
    __syncthreads();
    // ---- c2 = L^-T z
    to_digits(C2, C2, S2, K, pl.Kp, E3);
    __syncthreads();
    for (int item = warp; item < tk * nt; item += 4) {
        const int ri = item / nt, c0 = item % nt * 8;
        int f[2] = {0, 0};
        product(A + pl.LT + (ri * tk - ri * (ri - 1) / 2) * 256, tk - ri, Er + 2 * pl.Kp, C2, S2, ri * 16, E3, ri, c0,
                [&](int r, int c, double v) {
                    if (r >= K) return;
                    V[c * S2 + r] = v;
                    f[c & 1] = max(f[c & 1], exp_field(v));
                    if (c < tc) out[(int64_t)ord[M + r] * T + c] = wcast<Out>(v);
                });
        column_max(f[0], f[1], c0, E4);
    }
    __syncthreads();
    // ---- c1 = -W^T c2 and h = f1 - G^T c2
    to_digits(V, V, S2, K, pl.Kp, E4);
    __syncthreads();
    for (int item = warp; item < 2 * tm * nt; item += 4) {
        const int h = item / (tm * nt), it = item - h * tm * nt, ri = it / nt, c0 = it % nt * 8;
        product(A + (h ? pl.WT : pl.G) + ri * tk * 256, tk, Er + 3 * pl.Kp + h * pl.Mp, V, S2, 0, E4, ri, c0,
                [&](int r, int c, double v) {
                    if (r >= M) return;
                    if (h == 0) H[c * S1 + r] -= v;
                    else if (c < tc) out[(int64_t)ord[r] * T + c] = wcast<Out>(-v);
                });
    }
    __syncthreads();
    // ---- P1 d = h by substitution (C, then R), 16 or 32 lanes per tracer
    const int gl = M <= 16 ? 16 : 32, grp = t / gl, j0 = t % gl;
    for (int c0 = 0; c0 < nc; c0 += 128 / gl) {  // 128 / gl divides nc
        double *h = H + (c0 + grp) * S1;
        for (int k = 0; k + 1 < M; ++k) {
            const double z = h[k];
            for (int j = k + 1 + j0; j < M; j += gl) h[j] = fma(-P1[j * M + k], z, h[j]);
            __syncwarp();
        }
        for (int j = j0; j < M; j += gl) h[j] *= P1[j * M + j];
        __syncwarp();
        for (int k = M - 1; k > 0; --k) {
            const double z = h[k];
            for (int j = j0; j < k; j += gl) h[j] = fma(-P1[j * M + k], z, h[j]);
            __syncwarp();
        }
        if (c0 + grp < tc)
            for (int k = j0; k < M; k += gl) out[(int64_t)(n + k) * T + c0 + grp] = wcast<Out>(h[k]);
    }
}

// Members' coordinates patch by patch, at the rows of the coefficients.
__global__ void __launch_bounds__(128) pu_coords_kernel(const double *__restrict__ X, const int64_t *__restrict__ mstart,
                                                        const int32_t *__restrict__ members, int M,
                                                        double *__restrict__ mx) {
    const int64_t l = blockIdx.x, b = mstart[l];
    const int n = (int)(mstart[l + 1] - b);
    for (int e = threadIdx.x; e < 3 * n; e += 128) mx[3 * (b + l * M) + e] = X[3 * (int64_t)members[b + e / 3] + e % 3];
}

// ---- The blend. A term's factor (kernel value or harmonic times the normalised PU weight) and the
// product with the coefficient by type: double throughout; float: FP32 kernel values and sums; float2
// (the mixed step): factors formed in FP64 as in the FP64 blend and split into an FP32 pair, the sums
// pair arithmetic with FP32 operations. The patch sums cancel strongly (sum |c phi| reaches ~3e3 |s|),
// which plain FP32 sums turn into ~1e-4 relative errors; pairs keep ~n 2^-48.
template <typename R>
struct PuTerm;
template <>
struct PuTerm<double> {
    double s = 0.0;
    static __device__ double factor(double dx, double dy, double dz, int half, double w) {
        return phs_pow(fma(dz, dz, fma(dy, dy, dx * dx)), half) * w;
    }
    static __device__ double harmonic(double y, double w) { return y * w; }
    static __device__ double shfl(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
    static __device__ double zero() { return 0.0; }
    static __device__ double nan() { return (double)NAN; }
    __device__ void add(double f, double c) { s = fma(f, c, s); }
    __device__ void down(int o, bool on) {
        const double v = __shfl_down_sync(0xffffffffu, s, o);
        if (on) s += v;
    }
    __device__ void take(const PuTerm &o) { s += o.s; }
    __device__ double value() const { return s; }
};
template <>
struct PuTerm<float> {
    float s = 0.f;
    static __device__ float factor(double dx, double dy, double dz, int half, double w) {
        const float x = (float)dx, y = (float)dy, z = (float)dz, d2 = x * x + y * y + z * z;
        float v = sqrtf(d2);
        for (int h = 0; h < half; ++h) v *= d2;
        return v * (float)w;
    }
    static __device__ float harmonic(double y, double w) { return (float)y * (float)w; }
    static __device__ float shfl(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
    static __device__ float zero() { return 0.f; }
    static __device__ float nan() { return NAN; }
    __device__ void add(float f, float c) { s = fmaf(f, c, s); }
    __device__ void down(int o, bool on) {
        const float v = __shfl_down_sync(0xffffffffu, s, o);
        if (on) s += v;
    }
    __device__ void take(const PuTerm &o) { s += o.s; }
    __device__ float value() const { return s; }
};
template <>
struct PuTerm<float2> {
    float h = 0.f, l = 0.f;
    static __device__ float2 factor(double dx, double dy, double dz, int half, double w) {
        return pair_split<false>(PuTerm<double>::factor(dx, dy, dz, half, w));
    }
    static __device__ float2 harmonic(double y, double w) { return pair_split<false>(y * w); }
    static __device__ float2 shfl(float2 v, int src) {
        return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
    }
    static __device__ float2 zero() { return make_float2(0.f, 0.f); }
    static __device__ float2 nan() { return make_float2(NAN, NAN); }
    __device__ void add(float2 f, float2 c) { pair_fma(f, c, h, l); }
    __device__ void down(int o, bool on) {  // two-sum
        const float oh = __shfl_down_sync(0xffffffffu, h, o), ol = __shfl_down_sync(0xffffffffu, l, o);
        if (!on) return;
        const float s = h + oh, bp = s - h;
        const float e = (h - (s - bp)) + (oh - bp);
        l = l + (ol + e);
        h = s;
    }
    __device__ void take(const PuTerm &o) {
        const float s = h + o.h, bp = s - h;
        const float e = (h - (s - bp)) + (o.h - bp);
        l = l + (o.l + e);
        h = s;
    }
    __device__ float2 value() const { return pair_norm(h, l); }
};

template <typename R, int V>
struct alignas(sizeof(R) * V) PuVec {
    R v[V];
};

// What the blend needs of each of `count` points, a thread per point: the patches whose caps contain it,
// ordered by index (the blend's order of summation; kPuMaxPatches slots of ids and normalised weights) and
// the harmonics. cnt: their number, 0 where no patch contains the point (or all weights vanish), -1 where
// more than kPuMaxPatches do. Point i is P[order[i]] (order null: P[i]).
struct PuPoints {
    int32_t *cnt, *id;
    double *w, *Y;
};
constexpr int64_t kPuMinChunk = 16384, kPuMaxChunk = 65536;  // points per launch of the blend

__global__ void __launch_bounds__(64) pu_points_kernel(KnnGrid cg, double Rr, int wkind, int M, int ell,
                                                       const int32_t *__restrict__ order,
                                                       const double *__restrict__ P, int count, PuPoints o) {
    const int i = blockIdx.x * 64 + threadIdx.x;
    if (i >= count) return;
    const int64_t q = order ? order[i] : i;
    const double px = P[3 * q], py = P[3 * q + 1], pz = P[3 * q + 2];
    int32_t *id = o.id + (int64_t)i * kPuMaxPatches;
    double *w = o.w + (int64_t)i * kPuMaxPatches, *Y = o.Y + (int64_t)i * M;
    sh_eval(ell, px, py, pz, [&](int c, double v) { Y[c] = v; });
    // patches with |p - omega_l| < R: distances squared, the root only where rounding could decide
    const double hi = Rr * Rr * (1.0 + 1e-15), lo = Rr * Rr * (1.0 - 1e-15);
    int n = 0;
    grid_ball_rows(cg, px, py, pz, (float)Rr, [&](int c) {
        const double d2 = sqdist_rn(px, py, pz, cg.sx[c], cg.sy[c], cg.sz[c]);
        if (!(d2 < hi) || (d2 > lo && !(sqrt(d2) < Rr))) return;
        if (n < kPuMaxPatches) {
            const int32_t l = cg.sid[c];
            int s = n;
            for (; s > 0 && id[s - 1] > l; --s) {
                id[s] = id[s - 1];
                w[s] = w[s - 1];
            }
            id[s] = l;
            w[s] = d2;
        }
        ++n;
    });
    if (n > kPuMaxPatches) {
        o.cnt[i] = -1;
        return;
    }
    double wsum = 0.0;
    for (int a = 0; a < n; ++a) wsum += w[a] = pu_phi(wkind, sqrt(w[a]) / Rr);
    if (n == 0 || !(wsum > 0.0)) {
        o.cnt[i] = 0;
        return;
    }
    const double winv = 1.0 / wsum;
    for (int a = 0; a < n; ++a) w[a] *= winv;
    o.cnt[i] = n;
}

// Blend the patch interpolants at `count` points, one warp per point, in the order of pu_points_kernel (the
// order of the node grid's cells keeps a block's points in the same few patches). The terms of all patches
// of a point (members, then harmonics) form one list dealt to the lanes, 32 at a time: a lane forms its
// term's factor, then groups of ceil(tracers / V) lanes take a term each, V neighbouring tracers a lane, so
// that coefficient rows are read whole. Points without patches, or with too many, get NaN and EUNCOVERED
// or EINVAL.
//
// Bound: the FP64 pipe, 12 operations per term's factor (and one per tracer in FP64), where a warp
// instruction costs the same whatever its active lanes: that is why the search, the weights and the
// harmonics are a thread per point in a kernel of their own. N = 40,962, n = 84, 16 tracers in pairs: a
// warp per point for everything, a member per lane with its tracers in turn, pairs split by conversions
// 1,209 us; now 354 (231 of the FP64 pipe at its full rate). N = 10,242, n = 100, two tracers in FP64: 491,
// now 107, and 40 for the points, which run beside the coefficients.
template <typename R, int V>
__global__ void __launch_bounds__(128, 8) pu_eval_kernel(PuPoints pts, const double *__restrict__ mx,
                                                         const int64_t *__restrict__ mstart, int M, int half,
                                                         const R *__restrict__ coef, int T,
                                                         const int32_t *__restrict__ order,
                                                         const double *__restrict__ P, int count,
                                                         R *__restrict__ out, int32_t *__restrict__ status) {
    using Term = PuTerm<R>;
    const int lane = threadIdx.x & 31, pt = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (pt >= count) return;
    const int64_t i = order ? order[pt] : pt;
    const int np = pts.cnt[pt];
    if (np <= 0) {
        for (int c = lane; c < T; c += 32) out[i * T + c] = Term::nan();
        if (status && lane == 0) status[i] = np < 0 ? RBFSL_EINVAL : RBFSL_EUNCOVERED;
        return;
    }
    const double px = P[3 * i], py = P[3 * i + 1], pz = P[3 * i + 2];
    const int32_t *pid = pts.id + (int64_t)pt * kPuMaxPatches;
    const double *w = pts.w + (int64_t)pt * kPuMaxPatches, *Y = pts.Y + (int64_t)pt * M;
    int total = 0;
    for (int a = 0; a < np; ++a) total += (int)(mstart[pid[a] + 1] - mstart[pid[a]]) + M;
    for (int t0 = 0; t0 < T; t0 += 32 * V) {
        const int tv = (min(T - t0, 32 * V) + V - 1) / V, G = 32 / tv, grp = lane / tv, tl = lane - grp * tv;
        const R *C = coef + t0 + tl * V;
        Term acc[V];
        // Pairs: each chunk's terms are added up by themselves first, in chains of 32 / G additions, where
        // a lane has several of them: rounding grows with the length of a chain and its partial sums
        // (one chain over all chunks: error 5.7e-12 instead of 2.9e-12 at N = 40,962, n = 84).
        const bool chunked = std::is_same<R, float2>::value && G <= 16;
        // this lane's term: member or harmonic j of the point's a-th patch, n members from row r0 on.
        // Rows fit 32 bits: the factors of 2^31 of them would not fit the device.
        int a = -1, j = lane, n = -M, r0 = 0;
        double wl = 0.0;
        for (int e0 = 0; e0 < total; e0 += 32, j += 32) {
            const bool on = e0 + lane < total;
            while (on && j >= n + M) {
                j -= n + M;
                const int l = pid[++a];
                const int64_t b = mstart[l];
                n = (int)(mstart[l + 1] - b);
                r0 = (int)(b + (int64_t)l * M);
                wl = w[a];
            }
            R f = Term::zero();
            int row = r0;
            if (on) {
                row += j;
                if (j < n) {
                    const double *x = mx + 3 * (int64_t)row;
                    f = Term::factor(px - x[0], py - x[1], pz - x[2], half, wl);
                } else {
                    f = Term::harmonic(Y[j - n], wl);
                }
            }
            const int live = min(32, total - e0);
            Term part[V];
            if (!chunked) {
#pragma unroll
                for (int v = 0; v < V; ++v) part[v] = acc[v];
            }
#pragma unroll 4
            for (int s0 = 0; s0 < live; s0 += G) {
                const int src = s0 + grp;
                const bool take = grp < G && src < live;
                const R fs = Term::shfl(f, src & 31);
                const int64_t rs = __shfl_sync(0xffffffffu, row, src & 31);
                if (take) {
                    const PuVec<R, V> c = *reinterpret_cast<const PuVec<R, V> *>(C + rs * T);
#pragma unroll
                    for (int v = 0; v < V; ++v) part[v].add(fs, c.v[v]);
                }
            }
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (chunked) acc[v].take(part[v]);
                else acc[v] = part[v];
        }
        int top = 1;
        while (2 * top < G) top *= 2;
#pragma unroll
        for (int v = 0; v < V; ++v)
            for (int s = top; s > 0 && G > 1; s >>= 1) acc[v].down(s * tv, grp < s && grp + s < G);
        if (grp == 0) {
            PuVec<R, V> o;
#pragma unroll
            for (int v = 0; v < V; ++v) o.v[v] = acc[v].value();
            *reinterpret_cast<PuVec<R, V> *>(out + i * T + t0 + tl * V) = o;
        }
    }
    if (status && lane == 0) status[i] = RBFSL_OK;
}

// Factorise Mp stencil / patch systems given in CSR form (used by RBF-PU and by the local
// method's centre stencils). Dynamic shared memory sized for the largest system.
int launch_stencil_factor(const double *X, const int64_t *mstart, const int32_t *members,
                          const int64_t *lu_off, int64_t count, int max_n, int M, int ell,
                          int power, double *LU, int32_t *perm, int32_t *status, cudaStream_t s,
                          int colmajor) {
    int rc = sh_tables_init();
    if (rc) return rc;
    const int mmax = max_n + M;
    const int smem = ((mmax * (mmax | 1)) + 3 * max_n) * (int)sizeof(double);
    RBFSL_CUDA_TRY(cudaFuncSetAttribute(pu_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    pu_factor_kernel<<<(unsigned)count, 128, smem, s>>>(X, mstart, members, lu_off, M, ell, (power - 1) / 2,
                                                        LU, perm, status, colmajor);
    return launch_status("stencil_factor");
}

void pu_free(rbfsl_pu *u) {
    if (u->nodes_ix) rbfsl_knn_index_destroy(u->nodes_ix);
    if (u->centers_ix) rbfsl_knn_index_destroy(u->centers_ix);
    cudaFree(u->X); cudaFree(u->centers); cudaFree(u->mstart); cudaFree(u->members);
    cudaFree(u->lu_off); cudaFree(u->LU); cudaFree(u->perm); cudaFree(u->coef);
    cudaFree(u->mx); cudaFree(u->status);
    cudaFree(u->pmem);
    if (u->side) cudaStreamDestroy(u->side);
    if (u->fork) cudaEventDestroy(u->fork);
    if (u->join) cudaEventDestroy(u->join);
    cudaFree(u->pt_cnt); cudaFree(u->pt_id); cudaFree(u->pt_w); cudaFree(u->pt_Y);
}

constexpr int64_t kPuPackBytes = (int64_t)64 << 20;  // of unpacked factors at a time

// Device bytes of a handle and its set-up for Mp patches of at most `members` nodes each, T tracers.
size_t pu_estimate_bytes(int64_t N, int64_t Mp, int members, int ell, int power, int T) {
    const int M = (ell + 1) * (ell + 1), m = members + M;
    double factor = 8.0 * m * m, scratch = 0.0;  // LU, where a patch has no reduced form
    if (reduced_form(members, ell, (power - 1) / 2)) {
        factor = std::max(factor, 8.0 * PatchLayout(members, M).total);
        scratch = std::min((double)kPuPackBytes, 8.0 * Mp * CenterLayout(members, M).total);
    }
    const double points = (double)std::min(std::max(N, kPuMinChunk), kPuMaxChunk);
    return (size_t)(N * (3 * 8.0 + 28.0) + Mp * (factor + m * (36.0 + 8.0 * T) + 24 + 28 + 24) + scratch +
                    points * (4 + kPuMaxPatches * 12 + M * 8));
}

// Reduced factors of every patch, packed from a scratch buffer of at most kPuPackBytes at a time. Returns 1
// (with nothing kept) where a patch has none: its reduced matrix breaks down or its nodes coincide.
int pu_build_reduced(rbfsl_pu *u, const std::vector<int64_t> &ms, const std::vector<int32_t> &hc, int half,
                     cudaStream_t s) {
    const int M = u->M;
    const int64_t Mp = u->Mp, stride = CenterLayout(u->max_members, M).total;
    const int64_t chunk = std::min<int64_t>(Mp, std::max<int64_t>(1, kPuPackBytes / (stride * 8)));
    std::vector<int64_t> off(Mp);
    int64_t total = 0;
    for (int64_t l = 0; l < Mp; ++l) {
        off[l] = total;
        total += PatchLayout(hc[l], M).total;
    }
    double *F = nullptr;
    auto fail = [&](int code) {
        cudaGetLastError();
        cudaFree(F);
        cudaFree(u->LU);
        cudaFree(u->pmem);
        u->LU = nullptr;
        u->pmem = nullptr;
        if (code < 0) set_error(code == RBFSL_ENOMEM ? "pu_build: out of device memory" : "pu_build: factorisation failed");
        return code;
    };
    if (cudaMalloc(&F, chunk * stride * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&u->LU, total * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&u->pmem, ms[Mp] * sizeof(int32_t)) != cudaSuccess)
        return fail(1);  // the LU factors may still fit
    const int smem = RedLayout(u->max_members, M).total * (int)sizeof(double);
    if (cudaFuncSetAttribute(pu_reduced_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaMemcpyAsync(u->lu_off, off.data(), Mp * sizeof(int64_t), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(u->status, 0, sizeof(int32_t), s) != cudaSuccess)
        return fail(RBFSL_ECUDA);
    for (int64_t l0 = 0; l0 < Mp; l0 += chunk) {
        const unsigned cnt = (unsigned)std::min(chunk, Mp - l0);
        pu_reduced_factor_kernel<<<cnt, 128, smem, s>>>(u->X, u->mstart, u->members, l0, M, u->ell, half, stride, F,
                                                       u->perm, u->status);
        pu_pack_kernel<<<cnt, 128, 0, s>>>(u->mstart, l0, M, stride, F, u->lu_off, u->members, u->perm,
                                           (unsigned long long *)u->LU, u->pmem, u->status);
    }
    int32_t bad = 0;
    if (launch_status("pu_reduced_factor") ||
        cudaMemcpyAsync(&bad, u->status, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return fail(RBFSL_ECUDA);
    if (bad) return fail(1);
    cudaFree(F);
    u->bytes += total * sizeof(double) + ms[Mp] * sizeof(int32_t);
    u->reduced = 1;
    return RBFSL_OK;
}

int pu_build(rbfsl_pu *u, const double *x, int64_t N, const double *centers, int64_t Mp, double R,
             int ell, int power, cudaStream_t s) {
    int rc = sh_tables_init();
    if (rc) return rc;
    RBFSL_CUDA_TRY(cudaStreamCreateWithFlags(&u->side, cudaStreamNonBlocking));
    RBFSL_CUDA_TRY(cudaEventCreateWithFlags(&u->fork, cudaEventDisableTiming));
    RBFSL_CUDA_TRY(cudaEventCreateWithFlags(&u->join, cudaEventDisableTiming));
    u->N = N; u->Mp = Mp; u->R = R; u->ell = ell; u->power = power;
    u->M = (ell + 1) * (ell + 1);
    auto alloc = [&](void **p, size_t b) {
        if (cudaMalloc(p, b ? b : 1) != cudaSuccess) {
            cudaGetLastError();
            set_error("pu_build: out of device memory");
            return RBFSL_ENOMEM;
        }
        u->bytes += b;
        return RBFSL_OK;
    };
    if ((rc = alloc((void **)&u->X, N * 3 * sizeof(double)))) return rc;
    if ((rc = alloc((void **)&u->centers, Mp * 3 * sizeof(double)))) return rc;
    if ((rc = alloc((void **)&u->mstart, (Mp + 1) * sizeof(int64_t)))) return rc;
    if ((rc = alloc((void **)&u->lu_off, Mp * sizeof(int64_t)))) return rc;
    if ((rc = alloc((void **)&u->status, sizeof(int32_t)))) return rc;
    RBFSL_CUDA_TRY(cudaMemcpyAsync(u->X, x, N * 3 * sizeof(double), cudaMemcpyDeviceToDevice, s));
    RBFSL_CUDA_TRY(cudaMemcpyAsync(u->centers, centers, Mp * 3 * sizeof(double), cudaMemcpyDeviceToDevice, s));
    // node grid for membership, centre grid for the evaluation
    const double n_est = N * R * R / 4.0;
    if ((rc = rbfsl_knn_index_create(&u->nodes_ix, u->X, N, std::max(1, (int)n_est), s))) return rc;
    const double a_est = Mp * R * R / 4.0;
    if ((rc = rbfsl_knn_index_create(&u->centers_ix, u->centers, Mp, std::max(1, (int)a_est), s))) return rc;
    u->bytes += u->nodes_ix->bytes + u->centers_ix->bytes;
    // membership counts, host prefix sums
    int32_t *counts = nullptr;
    if ((rc = alloc((void **)&counts, Mp * sizeof(int32_t)))) return rc;
    const unsigned blocks = (unsigned)((Mp + 3) / 4);
    pu_members_kernel<<<blocks, 128, 0, s>>>(grid_view(u->nodes_ix), u->centers, Mp, R, counts, nullptr, nullptr);
    std::vector<int32_t> hc(Mp);
    cudaError_t e = cudaMemcpyAsync(hc.data(), counts, Mp * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(counts);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error(std::string("pu_build: ") + cudaGetErrorString(e));
        return RBFSL_ECUDA;
    }
    std::vector<int64_t> ms(Mp + 1, 0), lo(Mp, 0);
    int min_members = kPuMaxMembers;
    for (int64_t l = 0; l < Mp; ++l) {
        if (hc[l] < 1) { set_error("pu_build: a patch contains no node"); return RBFSL_EINVAL; }
        if (hc[l] > kPuMaxMembers || hc[l] + u->M > RBFSL_MAX_SYSTEM) {
            set_error("pu_build: a patch holds more nodes than RBFSL_MAX_SYSTEM allows");
            return RBFSL_EINVAL;
        }
        u->max_members = std::max(u->max_members, hc[l]);
        min_members = std::min(min_members, hc[l]);
        ms[l + 1] = ms[l] + hc[l];
    }
    u->rows = ms[Mp] + Mp * u->M;
    if ((rc = alloc((void **)&u->members, ms[Mp] * sizeof(int32_t)))) return rc;
    if ((rc = alloc((void **)&u->perm, u->rows * sizeof(int32_t)))) return rc;
    if ((rc = alloc((void **)&u->mx, u->rows * 3 * sizeof(double)))) return rc;
    RBFSL_CUDA_TRY(cudaMemcpyAsync(u->mstart, ms.data(), (Mp + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
    pu_members_kernel<<<blocks, 128, 0, s>>>(grid_view(u->nodes_ix), u->centers, Mp, R, nullptr, u->mstart, u->members);
    // per-point lists of the blend, for as many points as one launch takes
    u->chunk = std::min(std::max(N, kPuMinChunk), kPuMaxChunk);
    if ((rc = alloc((void **)&u->pt_cnt, u->chunk * sizeof(int32_t)))) return rc;
    if ((rc = alloc((void **)&u->pt_id, u->chunk * kPuMaxPatches * sizeof(int32_t)))) return rc;
    if ((rc = alloc((void **)&u->pt_w, u->chunk * kPuMaxPatches * sizeof(double)))) return rc;
    if ((rc = alloc((void **)&u->pt_Y, u->chunk * u->M * sizeof(double)))) return rc;
    pu_coords_kernel<<<(unsigned)Mp, 128, 0, s>>>(u->X, u->mstart, u->members, u->M, u->mx);
    const int half = (power - 1) / 2;
    if (reduced_form(min_members, ell, half)) {
        rc = pu_build_reduced(u, ms, hc, half, s);
        if (rc <= 0) return rc;
    }
    // LU of the whole systems
    int64_t lu_total = 0;
    for (int64_t l = 0; l < Mp; ++l) {
        const int64_t m = hc[l] + u->M;
        lo[l] = lu_total;
        lu_total += m * m;
    }
    if ((rc = alloc((void **)&u->LU, lu_total * sizeof(double)))) return rc;
    RBFSL_CUDA_TRY(cudaMemcpyAsync(u->lu_off, lo.data(), Mp * sizeof(int64_t), cudaMemcpyHostToDevice, s));
    RBFSL_CUDA_TRY(cudaMemsetAsync(u->status, 0, sizeof(int32_t), s));
    if ((rc = launch_stencil_factor(u->X, u->mstart, u->members, u->lu_off, Mp, u->max_members, u->M, ell,
                                    power, u->LU, u->perm, u->status, s, 0)))
        return rc;
    int32_t bad = 0;
    RBFSL_CUDA_TRY(cudaMemcpyAsync(&bad, u->status, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    RBFSL_CUDA_TRY(cudaStreamSynchronize(s));
    if (bad) {
        set_error("pu_build: " + std::to_string(bad) + " singular patch systems");
        return RBFSL_ESINGULAR;
    }
    return RBFSL_OK;
}

namespace {

template <typename In, typename Out>
int launch_pu_coef(rbfsl_pu *u, const In *q, int T, cudaStream_t s) {
    if (u->reduced) {
        auto *kernel = pu_coef_reduced_kernel<In, Out>;
        // the largest patch has the most rows: K grows with n, M does not
        const PatchLayout pl(u->max_members, u->M);
        const int smem = pu_coef_bytes(pl.Kp, pl.Mp, T > 8 ? kPuTracers : 8);
        RBFSL_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        kernel<<<dim3((unsigned)u->Mp, (T + kPuTracers - 1) / kPuTracers), 128, smem, s>>>(
            u->mstart, u->pmem, u->lu_off, u->M, (const unsigned long long *)u->LU, u->perm, q, T, (Out *)u->coef);
    } else {
        auto *kernel = pu_coef_kernel<In, Out>;
        const int smem = (u->max_members + u->M) * T * (int)sizeof(double);
        RBFSL_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        kernel<<<(unsigned)u->Mp, 128, smem, s>>>(u->mstart, u->members, u->lu_off, u->M, u->LU, u->perm, q, T,
                                                  (Out *)u->coef);
    }
    return launch_status("pu_coef");
}

// points of one launch: the chunk from b on, in the order of the node grid's cells where there are as many
// points as nodes (departure points lie near theirs)
struct PuChunk {
    const int32_t *order;
    int64_t base;  // of the arrays by point; 0 with an order, whose entries index them from their start
    int count;
};
PuChunk pu_chunk(const rbfsl_pu *u, int64_t Nq, int64_t b) {
    const int count = (int)std::min(u->chunk, Nq - b);
    return Nq == u->N ? PuChunk{u->nodes_ix->sid + b, 0, count} : PuChunk{nullptr, b, count};
}

PuPoints pu_points(const rbfsl_pu *u) { return PuPoints{u->pt_cnt, u->pt_id, u->pt_w, u->pt_Y}; }

int launch_pu_points(rbfsl_pu *u, const PuChunk &c, const double *p, int wkind, cudaStream_t s) {
    pu_points_kernel<<<(unsigned)((c.count + 63) / 64), 64, 0, s>>>(grid_view(u->centers_ix), u->R, wkind, u->M, u->ell,
                                                                   c.order, p + 3 * c.base, c.count, pu_points(u));
    return launch_status("pu_points");
}

template <typename R>
int launch_pu_eval(rbfsl_pu *u, const PuChunk &c, int T, const double *p, R *out, int32_t *status, cudaStream_t s) {
    auto go = [&](auto *kernel) {
        kernel<<<(unsigned)((c.count + 3) / 4), 128, 0, s>>>(pu_points(u), u->mx, u->mstart, u->M, (u->power - 1) / 2,
                                                            (const R *)u->coef, T, c.order, p + 3 * c.base, c.count,
                                                            out + c.base * T, status ? status + c.base : nullptr);
    };
    // two tracers a lane where rows of coefficients and of the result are aligned for it
    if (T % 2 == 0 && (uintptr_t)out % (2 * sizeof(R)) == 0) go(pu_eval_kernel<R, 2>);
    else go(pu_eval_kernel<R, 1>);
    return launch_status("pu_eval");
}

template <typename In>
int launch_pu_coef_typed(rbfsl_pu *u, const In *q, int T, int dtype, cudaStream_t s) {
    if (dtype == RBFSL_F64) return launch_pu_coef<In, double>(u, q, T, s);
    if (dtype == RBFSL_F32) return launch_pu_coef<In, float>(u, q, T, s);
    return launch_pu_coef<In, float2>(u, q, T, s);
}

}  // namespace

int pu_apply_begin(rbfsl_pu *u, const void *q, int q_dtype, int T, int dtype, cudaStream_t s) {
    RBFSL_CHECK_ARG((size_t)(u->max_members + u->M) * T * sizeof(double) <= 200 * 1024,
                    "pu_apply: too many tracers for one call");
    if (T != u->coef_T) {
        cudaFree(u->coef);
        u->coef = nullptr;
        u->coef_T = 0;
        if (cudaMalloc(&u->coef, u->rows * T * sizeof(double)) != cudaSuccess) {
            cudaGetLastError();
            set_error("pu_apply: out of device memory");
            return RBFSL_ENOMEM;
        }
        u->coef_T = T;
    }
    RBFSL_CUDA_TRY(cudaEventRecord(u->fork, s));
    RBFSL_CUDA_TRY(cudaStreamWaitEvent(u->side, u->fork, 0));
    const int rc = q_dtype == RBFSL_F64 ? launch_pu_coef_typed(u, (const double *)q, T, dtype, u->side)
                                        : launch_pu_coef_typed(u, (const float2 *)q, T, dtype, u->side);
    RBFSL_CUDA_TRY(cudaEventRecord(u->join, u->side));
    if (rc) RBFSL_CUDA_TRY(cudaStreamWaitEvent(s, u->join, 0));
    return rc;
}

int pu_apply_end(rbfsl_pu *u, int T, const double *p, int64_t Nq, int wkind, int dtype, void *out, int32_t *status,
                 cudaStream_t s) {
    int rc = RBFSL_OK;
    for (int64_t b = 0; b < Nq && !rc; b += u->chunk) {
        const PuChunk c = pu_chunk(u, Nq, b);
        rc = launch_pu_points(u, c, p, wkind, s);
        if (b == 0) RBFSL_CUDA_TRY(cudaStreamWaitEvent(s, u->join, 0));
        if (rc) break;
        if (dtype == RBFSL_F64) rc = launch_pu_eval(u, c, T, p, (double *)out, status, s);
        else if (dtype == RBFSL_F32) rc = launch_pu_eval(u, c, T, p, (float *)out, status, s);
        else rc = launch_pu_eval(u, c, T, p, (float2 *)out, status, s);
    }
    if (Nq == 0) RBFSL_CUDA_TRY(cudaStreamWaitEvent(s, u->join, 0));
    return rc;
}

}  // namespace rbfsl

extern "C" int rbfsl_pu_create(rbfsl_pu **out, const double *x, int64_t N, const double *centers,
                               int64_t Mp, double radius, int ell, int kernel, double kparam,
                               void *stream) {
    using namespace rbfsl;
    RBFSL_CHECK_ARG(out && x && centers, "pu_create: null pointer");
    RBFSL_CHECK_ARG(N >= 1 && N < ((int64_t)1 << 31) && Mp >= 1 && Mp < ((int64_t)1 << 31),
                    "pu_create: bad sizes");
    RBFSL_CHECK_ARG(radius > 0 && radius <= 2.0, "pu_create: radius must be in (0, 2]");
    RBFSL_CHECK_ARG(ell >= 0 && ell <= RBFSL_MAX_SH_DEGREE, "pu_create: ell out of range");
    const int pw = (int)kparam;
    RBFSL_CHECK_ARG(kernel == RBFSL_PHS && (double)pw == kparam && pw >= 1 && (pw & 1),
                    "pu_create: only the PHS kernel r^p with odd p is supported");
    auto *u = new rbfsl_pu();
    RBFSL_CUDA_TRY(cudaGetDevice(&u->device));
    const int rc = pu_build(u, x, N, centers, Mp, radius, ell, pw, (cudaStream_t)stream);
    if (rc != RBFSL_OK) {
        pu_free(u);
        delete u;
        return rc;
    }
    *out = u;
    return RBFSL_OK;
}

extern "C" int rbfsl_pu_destroy(rbfsl_pu *u) {
    if (!u) return RBFSL_OK;
    rbfsl::pu_free(u);
    delete u;
    return RBFSL_OK;
}

extern "C" int rbfsl_pu_apply(rbfsl_pu *u, const double *q, int T, const double *p, int64_t Nq,
                              int weight_kind, int dtype, void *out, int32_t *status, void *stream) {
    using namespace rbfsl;
    RBFSL_CHECK_ARG(u != nullptr, "pu_apply: null handle");
    RBFSL_CHECK_ARG(T >= 1 && Nq >= 0, "pu_apply: bad sizes");
    RBFSL_CHECK_ARG(q && (Nq == 0 || (p && out)), "pu_apply: null pointer");
    RBFSL_CHECK_ARG(weight_kind == RBFSL_PU_WENDLAND || weight_kind == RBFSL_PU_BSPLINE, "pu_apply: bad weight kind");
    RBFSL_CHECK_ARG(dtype == RBFSL_F64 || dtype == RBFSL_F32 || dtype == RBFSL_F32X2, "pu_apply: bad dtype");
    const int rc = pu_apply_begin(u, q, RBFSL_F64, T, dtype, (cudaStream_t)stream);
    return rc ? rc : pu_apply_end(u, T, p, Nq, weight_kind, dtype, out, status, (cudaStream_t)stream);
}
