// Stencil weights of the augmented local RBF interpolant (Sec. 2.2, Eqs. rbf_poly and
// rbf_poly_linsys), FP64 throughout.
//
// The weights w solve the symmetric (n + M) x (n + M) saddle-point system (M = (ell+1)^2)
//     [ A    P ] [ w      ]   [ phi(|p - x_j|) ]      A_jk = |x_j - x_k|^pw   (PHS, zero diagonal)
//     [ P^T  0 ] [ lambda ] = [ Y(p)           ]      P_jc = Y_c(x_j)
// Each point's group of warps solves it in shared memory, reduced to the null space of P^T
// (reduced.cuh) or, for exponents above the harmonics' order and n <= M, as a whole by a blocked
// Bunch-Kaufman L D L^T (weights_point_ldl): ~m^3 / 3 flops per point either way (m = n + M), bound
// by GB300's FP64 rate. Small systems take one warp per point (four points per block); larger ones
// two or four warps per point, several points per SM so that one point's serial steps overlap the others'
// products. N = 40,962, reduced form against the indefinite factorisation: m = 109 15.0 ms against
// 30.3 ms, m = 71 (before two warps per point) 6.6 ms against 10.1 ms, m = 40 2.1 ms against 2.9 ms.
#include <vector>

#include "common.cuh"
#include "kernels.cuh"
#include "device_ops.cuh"
#include "reduced.cuh"

namespace rbfsl {

__constant__ ShTables c_sh;

namespace {
bool g_sh_ready[64] = {false};
}

int sh_tables_init() {
    int dev = 0;
    RBFSL_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 64 && g_sh_ready[dev]) return RBFSL_OK;
    ShTables t{};
    const double pi = 3.14159265358979323846;
    for (int m = 0; m <= kMaxL; ++m) {
        double q = 1.0;
        for (int i = 1; i <= m; ++i) q *= (double)(2 * i - 1);
        t.qmm[m] = q;
        for (int l = m; l <= kMaxL; ++l) {
            const int id = l * l + l + m;
            double ratio = 1.0;  // (l-m)! / (l+m)!
            for (int i = l - m + 1; i <= l + m; ++i) ratio /= (double)i;
            t.K[id] = std::sqrt((m == 0 ? 1.0 : 2.0) * (2.0 * l + 1.0) / (4.0 * pi) * ratio);
            if (l == m + 1) {
                t.a[id] = 2.0 * m + 1.0;
                t.b[id] = 0.0;
            } else if (l >= m + 2) {
                t.a[id] = (2.0 * l - 1.0) / (double)(l - m);
                t.b[id] = (double)(l + m - 1) / (double)(l - m);
            }
        }
    }
    RBFSL_CUDA_TRY(cudaMemcpyToSymbol(c_sh, &t, sizeof(t)));
    if (dev < 64) g_sh_ready[dev] = true;
    return RBFSL_OK;
}

struct WeightsArgs {
    const double *X;
    const int32_t *idx;
    int64_t Nq;
    int n, ell, half, m;
    int region_doubles;  // shared-memory doubles per point
    const double *P;
    int32_t *status;
};

// NW warps per point (1, 2 or 4). With NW = 1 a block holds blockDim/32 independent points and
// the group barrier is __syncwarp; with NW > 1 a block is one point and uses __syncthreads. kBlocks:
// the blocks per SM that the registers are bounded for: seven for one warp per point (72 registers);
// with two and four warps, whose digit products want 117 to 128, what shared memory allows (eight points of
// two warps, five or four of four). kReduced: whether the kernel serves the reduced form; without, the
// indefinite factorisation alone, in 72 registers.
template <int NW, int kBlocks, bool kReduced, typename WT>
__global__ void __launch_bounds__(NW == 2 ? 64 : 128, kBlocks) weights_kernel(WeightsArgs a, WT *__restrict__ W) {
    extern __shared__ double smem[];
    constexpr int GT = NW * kWarp;
    const int g = threadIdx.x / GT, t = threadIdx.x % GT;
    const int spb = blockDim.x / GT;
    const int64_t i = (int64_t)blockIdx.x * spb + g;
    if (i >= a.Nq) return;  // NW == 1 only (with NW > 1 the grid has exactly Nq blocks)
    double *R = smem + (size_t)g * a.region_doubles;
    double *w = nullptr;
    int rc;
    if constexpr (kReduced)
        rc = weights_point<NW, NW != 1>(R, a.X, a.idx + i * a.n, a.n, a.m, a.ell, a.half, a.P[3 * i], a.P[3 * i + 1],
                                        a.P[3 * i + 2], t, w);
    else
        rc = weights_point_ldl<NW>(R, a.X, a.idx + i * a.n, a.n, a.m, a.ell, a.half, a.P[3 * i], a.P[3 * i + 1],
                                   a.P[3 * i + 2], t, w);
    if (t >= kWarp) return;
    const int n = a.n, lane = t;
    for (int j = lane; j < n; j += kWarp) W[i * n + j] = wcast<WT>(rc == RBFSL_OK ? w[j] : (double)NAN);
    if (a.status && lane == 0) a.status[i] = rc;
}

template <int NW, int kBlocks, bool kReduced, typename WT>
int launch_weights_nw(const WeightsArgs &a, int spb, void *w, cudaStream_t s) {
    const int smem = spb * a.region_doubles * 8;
    auto *kernel = weights_kernel<NW, kBlocks, kReduced, WT>;
    RBFSL_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    // all of the unified L1 / shared storage as shared memory: as many points per SM as fit
    RBFSL_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    const unsigned blocks = (unsigned)((a.Nq + spb - 1) / spb);
    kernel<<<blocks, spb * NW * kWarp, smem, s>>>(a, (WT *)w);
    return launch_status("stencil_weights");
}

template <int NW, int kBlocks, bool kReduced = true>
int launch_weights_typed(const WeightsArgs &a, int spb, void *w, int w_dtype, cudaStream_t s) {
    if (w_dtype == RBFSL_F64) return launch_weights_nw<NW, kBlocks, kReduced, double>(a, spb, w, s);
    if (w_dtype == RBFSL_F32X2) return launch_weights_nw<NW, kBlocks, kReduced, float2>(a, spb, w, s);
    return launch_weights_nw<NW, kBlocks, kReduced, float>(a, spb, w, s);
}

int launch_weights(const double *x, const int32_t *idx, int64_t Nq, int n, int ell, int power,
                   const double *p, void *w, int w_dtype, int32_t *status, cudaStream_t s) {
    if (Nq == 0) return RBFSL_OK;
    int rc = sh_tables_init();
    if (rc != RBFSL_OK) return rc;
    WeightsArgs a{};
    a.X = x; a.idx = idx; a.Nq = Nq; a.n = n; a.ell = ell; a.half = (power - 1) / 2;
    a.P = p; a.status = status;
    a.m = n + (ell + 1) * (ell + 1);
    a.region_doubles = weights_doubles(n, a.m, ell, a.half);
    const int bytes = a.region_doubles * 8;
    const bool reduced = reduced_form(n, ell, a.half);
    // the indefinite factorisation's steps are all block-wide: four warps per point, and registers for the six or
    // seven points that an SM holds up to 37 KB a point (m = 54 at N = 2,562 488 us, two warps 536; m = 81 at N =
    // 12,347 4.26 ms, bounded for five points 4.72)
    if (!reduced && bytes > kWeightsSmallBytes && bytes <= 37 * 1024)
        return launch_weights_typed<4, 7, false>(a, 1, w, w_dtype, s);
    if (bytes > kWeightsSmallBytes || (reduced && reduced_on_tensor(a.m - n))) {
        // larger systems (m >~ 45, or with the products on the tensor cores), one point per block: two warps
        // per point while eight points fit an SM's 227 KB (more points overlap each other's serial steps:
        // m = 71 at N = 12,347 1.73 ms, four warps and five points 1.90), else four warps; five blocks need
        // 1/5 of it each
        if (bytes <= kWeightsPairBytes) return launch_weights_typed<2, 8>(a, 1, w, w_dtype, s);
        return bytes <= 44 * 1024 ? launch_weights_typed<4, 5>(a, 1, w, w_dtype, s)
                                  : launch_weights_typed<4, 4>(a, 1, w, w_dtype, s);
    }
    return launch_weights_typed<1, 7>(a, 4, w, w_dtype, s);  // four independent points (warps) per block
}

// Centre-stencil weights from LU factors of the whole systems, one warp per point (center_point).
template <typename WT>
__global__ void __launch_bounds__(128) center_weights_kernel(
    const double *__restrict__ X, const int32_t *__restrict__ Kc, const int32_t *__restrict__ Ik,
    const double *__restrict__ LU, const int32_t *__restrict__ perm, int64_t Nq, int n, int ell,
    int half, const double *__restrict__ P, int32_t *__restrict__ I, WT *__restrict__ W,
    int32_t *__restrict__ status) {
    extern __shared__ double sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int M = (ell + 1) * (ell + 1), m = n + M;
    const int64_t i = (int64_t)blockIdx.x * 4 + warp;
    if (i >= Nq) return;
    double *b = sm + (size_t)warp * 2 * m, *y = b + m;
    const int64_t k = Kc[i];
    if (k < 0) {
        for (int j = lane; j < n; j += 32) { W[i * n + j] = wcast<WT>((double)NAN); I[i * n + j] = -1; }
        if (status && lane == 0) status[i] = RBFSL_EKNN;
        return;
    }
    for (int j = lane; j < n; j += 32) I[i * n + j] = Ik[k * n + j];
    center_point(X, Ik + k * n, LU + (size_t)k * m * m, perm + (size_t)k * m, n, m, ell, half,
                 P[3 * i], P[3 * i + 1], P[3 * i + 2], b, y, lane);
    for (int j = lane; j < n; j += 32) W[i * n + j] = wcast<WT>(y[j]);
    if (status && lane == 0) status[i] = RBFSL_OK;
}

// The same from the reduced factors, kLanes lanes per point (center_point_reduced).
template <typename WT, int kLanes>
__global__ void __launch_bounds__(128) center_reduced_kernel(
    const double *__restrict__ X, const int32_t *__restrict__ Kc, const int32_t *__restrict__ Ik,
    const double *__restrict__ F, const int32_t *__restrict__ order, int64_t Nq, int n, int M, int ell, int half,
    const double *__restrict__ P, int32_t *__restrict__ I, WT *__restrict__ W, int32_t *__restrict__ status) {
    extern __shared__ double sm[];
    const int grp = threadIdx.x / kLanes, l = threadIdx.x % kLanes;
    constexpr int kPoints = 128 / kLanes;
    const int64_t b0 = (int64_t)blockIdx.x * kPoints, i0 = b0 + grp;
    // the harmonics of the block's points, a thread per point and order: on the FP64 pipe a warp
    // instruction costs the same whatever its active lanes
    for (int f = threadIdx.x; f < kPoints * (ell + 1); f += 128) {
        const int p = f / (ell + 1);
        const int64_t i = b0 + p < Nq ? b0 + p : Nq - 1;
        double *y = sm + (size_t)p * center_reduced_doubles(n, M) + M * M + n;
        sh_eval_lanes(ell, P[3 * i], P[3 * i + 1], P[3 * i + 2], f - p * (ell + 1), [&](int c, double v) { y[c] = v; });
    }
    __syncthreads();
    if (i0 - grp % (32 / kLanes) >= Nq) return;  // the whole warp past the end
    const bool on = i0 < Nq;                     // a group past the end repeats the last point
    const int64_t i = on ? i0 : Nq - 1;
    const int64_t kc = Kc[i], k = kc < 0 ? 0 : kc;
    const int32_t *S = Ik + k * n;
    double *w = center_point_reduced<kLanes, false>(X, S, F + (size_t)k * CenterLayout(n, M).total, order + (size_t)k * n, n, M,
                                             ell, half, P[3 * i], P[3 * i + 1], P[3 * i + 2],
                                             sm + (size_t)grp * center_reduced_doubles(n, M), l);
    if (!on) return;
    for (int j = l; j < n; j += kLanes) {
        W[i * n + j] = wcast<WT>(kc < 0 ? (double)NAN : w[j]);
        I[i * n + j] = kc < 0 ? -1 : S[j];
    }
    if (status && l == 0) status[i] = kc < 0 ? RBFSL_EKNN : RBFSL_OK;
}

// Reduced factors of every stencil, one block per stencil. bad[0]: stencils without them, bad[1]:
// failed neighbour searches.
__global__ void __launch_bounds__(128, 4) center_factor_kernel(const double *__restrict__ X,
                                                               const int32_t *__restrict__ Ik, int n, int M, int ell,
                                                               int half, double *__restrict__ F,
                                                               int32_t *__restrict__ order, int32_t *__restrict__ bad) {
    extern __shared__ double sm[];
    const int64_t k = blockIdx.x;
    double *out = nullptr, *Fk = F + (size_t)k * CenterLayout(n, M).total;
    const int32_t s0 = Ik[k * n];
    const int64_t c = s0 < 0 ? 0 : s0;
    const int t = threadIdx.x;
    const int rc = reduced_on_tensor(M)
                       ? weights_point_reduced<4, true, kFactorCenter>(sm, X, Ik + k * n, n, M, ell, half, X[3 * c], X[3 * c + 1],
                                                              X[3 * c + 2], t, out, Fk, order + (size_t)k * n)
                       : weights_point_reduced<4, false, kFactorCenter>(sm, X, Ik + k * n, n, M, ell, half, X[3 * c], X[3 * c + 1],
                                                               X[3 * c + 2], t, out, Fk, order + (size_t)k * n);
    if (t == 0 && rc != RBFSL_OK) atomicAdd(&bad[rc == RBFSL_EKNN ? 1 : 0], 1);
}

void center_factors_free(CenterFactors *f) {
    cudaFree(f->F);
    cudaFree(f->order);
    *f = CenterFactors();
}

int center_factors_build(const double *X, const int32_t *Ik, int64_t N, int n, int ell, int power, CenterFactors *out,
                         cudaStream_t s) {
    int rc = sh_tables_init();
    if (rc) return rc;
    const int M = (ell + 1) * (ell + 1), m = n + M, half = (power - 1) / 2;
    int32_t *bad = nullptr, hb[2] = {0, 0};
    int64_t *csr = nullptr;
    auto fail = [&](int code, const char *msg) {
        cudaGetLastError();
        cudaFree(bad);
        cudaFree(csr);
        center_factors_free(out);
        set_error(msg);
        return code;
    };
    auto read_bad = [&] {
        return cudaMemcpyAsync(hb, bad, sizeof(hb), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
               cudaStreamSynchronize(s) == cudaSuccess;
    };
    if (cudaMalloc(&bad, sizeof(hb)) != cudaSuccess) return fail(RBFSL_ENOMEM, "centre factors: out of device memory");
    if (reduced_form(n, ell, half)) {
        const size_t fb = (size_t)N * CenterLayout(n, M).total * sizeof(double), ob = (size_t)N * n * sizeof(int32_t);
        if (cudaMalloc(&out->F, fb) != cudaSuccess || cudaMalloc(&out->order, ob) != cudaSuccess)
            return fail(RBFSL_ENOMEM, "centre factors: out of device memory");
        out->bytes = fb + ob;
        out->reduced = 1;
        const int smem = RedLayout(n, M).total * (int)sizeof(double);
        if (cudaFuncSetAttribute(center_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
            cudaMemsetAsync(bad, 0, sizeof(hb), s) != cudaSuccess)
            return fail(RBFSL_ECUDA, "centre factorisation failed");
        center_factor_kernel<<<(unsigned)N, 128, smem, s>>>(X, Ik, n, M, ell, half, out->F, out->order, bad);
        if (launch_status("center_factor") || !read_bad()) return fail(RBFSL_ECUDA, "centre factorisation failed");
        if (hb[1]) return fail(RBFSL_EKNN, "centre stencils: the neighbour search failed");
        if (!hb[0]) {
            cudaFree(bad);
            return RBFSL_OK;
        }
        center_factors_free(out);
    }
    // LU of the whole systems (partial pivoting, FP64)
    const size_t fb = (size_t)N * m * m * sizeof(double), ob = (size_t)N * m * sizeof(int32_t);
    if (cudaMalloc(&out->F, fb) != cudaSuccess || cudaMalloc(&out->order, ob) != cudaSuccess ||
        cudaMalloc(&csr, (2 * N + 1) * sizeof(int64_t)) != cudaSuccess)
        return fail(RBFSL_ENOMEM, "centre factors: out of device memory");
    out->bytes = fb + ob;
    out->reduced = 0;
    std::vector<int64_t> h(2 * N + 1);
    for (int64_t k = 0; k <= N; ++k) h[k] = k * n;
    for (int64_t k = 0; k < N; ++k) h[N + 1 + k] = k * m * m;
    if (cudaMemcpyAsync(csr, h.data(), h.size() * sizeof(int64_t), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(bad, 0, sizeof(hb), s) != cudaSuccess)
        return fail(RBFSL_ECUDA, "centre factorisation failed");
    rc = launch_stencil_factor(X, csr, Ik, csr + N + 1, N, n, M, ell, power, out->F, out->order, bad, s, 1);
    if (rc != RBFSL_OK || !read_bad()) return fail(rc ? rc : RBFSL_ECUDA, rc ? get_error() : "centre factorisation failed");
    if (hb[0]) return fail(RBFSL_ESINGULAR, (std::to_string(hb[0]) + " singular centre stencils").c_str());
    cudaFree(bad);
    cudaFree(csr);
    return RBFSL_OK;
}

namespace {
template <typename WT>
void launch_center_typed(const double *X, const int32_t *K, const int32_t *Ik, const CenterFactors &f, int64_t Nq, int n,
                         int ell, int half, const double *p, int32_t *I, void *w, int32_t *status, cudaStream_t s) {
    const int M = (ell + 1) * (ell + 1), m = n + M;
    if (!f.reduced) {
        center_weights_kernel<WT><<<(unsigned)((Nq + 3) / 4), 128, 4 * 2 * m * sizeof(double), s>>>(
            X, K, Ik, f.F, f.order, Nq, n, ell, half, p, I, (WT *)w, status);
        return;
    }
    const int lanes = center_lanes(n, M), ppb = 128 / lanes;
    const int smem = ppb * center_reduced_doubles(n, M) * (int)sizeof(double);
    auto go = [&](auto *kernel) {
        if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        kernel<<<(unsigned)((Nq + ppb - 1) / ppb), 128, smem, s>>>(X, K, Ik, f.F, f.order, Nq, n, M, ell, half, p, I,
                                                                  (WT *)w, status);
    };
    if (lanes == 16) go(center_reduced_kernel<WT, 16>);
    else go(center_reduced_kernel<WT, 32>);
}
}  // namespace

int launch_center_weights(const double *X, const int32_t *K, const int32_t *Ik, const CenterFactors &f, int64_t Nq,
                          int n, int ell, int power, const double *p, int32_t *I, void *w, int w_dtype,
                          int32_t *status, cudaStream_t s) {
    if (Nq == 0) return RBFSL_OK;
    int rc = sh_tables_init();
    if (rc) return rc;
    const int half = (power - 1) / 2;
    if (w_dtype == RBFSL_F64) launch_center_typed<double>(X, K, Ik, f, Nq, n, ell, half, p, I, w, status, s);
    else if (w_dtype == RBFSL_F32X2) launch_center_typed<float2>(X, K, Ik, f, Nq, n, ell, half, p, I, w, status, s);
    else launch_center_typed<float>(X, K, Ik, f, Nq, n, ell, half, p, I, w, status, s);
    return launch_status("center_weights");
}

}  // namespace rbfsl

extern "C" int rbfsl_stencil_weights(const double *x, int64_t N, const int32_t *idx, int64_t Nq,
                                     int n, int ell, int kernel, double kparam, const double *p,
                                     void *w, int w_dtype, int32_t *status, void *stream) {
    using namespace rbfsl;
    RBFSL_CHECK_ARG(Nq >= 0 && N >= 1, "stencil_weights: bad sizes");
    RBFSL_CHECK_ARG(n >= 1 && n <= N, "stencil_weights: n out of range");
    RBFSL_CHECK_ARG(ell >= 0 && ell <= RBFSL_MAX_SH_DEGREE, "stencil_weights: ell out of range");
    RBFSL_CHECK_ARG(n + (ell + 1) * (ell + 1) <= RBFSL_MAX_SYSTEM,
                    "stencil_weights: n + (ell+1)^2 exceeds RBFSL_MAX_SYSTEM");
    const int pw = (int)kparam;
    RBFSL_CHECK_ARG(kernel == RBFSL_PHS && (double)pw == kparam && pw >= 1 && (pw & 1),
                    "stencil_weights: only the PHS kernel r^p with odd p is supported");
    RBFSL_CHECK_ARG(w_dtype == RBFSL_F64 || w_dtype == RBFSL_F32 || w_dtype == RBFSL_F32X2,
                    "stencil_weights: bad w_dtype");
    RBFSL_CHECK_ARG(Nq == 0 || (x && idx && p && w), "stencil_weights: null pointer");
    return launch_weights(x, idx, Nq, n, ell, pw, p, w, w_dtype, status, (cudaStream_t)stream);
}
