// Cardinal form of the global interpolant (Sec. 2.1, Eqs. srbfinterp and rbf_linsys).
//
// The interpolant of a field q at a point p is phi(p, X) c with A_X c = q, so at a fixed set of
// points P it is E q with E = Phi(P, X) A_X^-1 (Nq x N), the values of the N cardinal functions
// at the points. Under a steady flow the departure points are the same at every step, so E is
// formed once and each semi-Lagrangian step becomes one dense product q <- E q: the per-step
// triangular solves (2 N^2 T FP64 flops, latency-bound) and the kernel evaluations go away.
//
// Build: A_X is symmetric (phi depends on |x_i - x_j| only, and the assembly forms the same
// squared distance for (i, j) and (j, i)), so E^T = A_X^-1 Phi(P, X)^T. Blocks of kCardChunk
// points are solved with the LU factor of rbfsl_global_factor (forward and backward
// substitution, as the per-step solve) and transposed into E, FP64 or FP32 pairs.
//
// Apply: out = E q on the tensor cores by exact digit products (split_gemm.cu), FP64 or FP32 pairs:
// the cardinal values are O(1) and do not cancel (unlike the coefficients c, which grow as A_X
// becomes singular), so pairs of E and q keep FP64-like accuracy.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "kernels.cuh"
#include "split_gemm.cuh"

namespace rbfsl {

namespace {

constexpr int kCardChunk = 512;  // points per block of right-hand sides in the build

// B[j][ii] = phi(|x_j - p_(i0+ii)|), N x nc row-major: the right-hand sides A_X E^T = Phi^T.
__global__ void cardinal_rhs(const double *__restrict__ X, int64_t N, const double *__restrict__ P,
                             int64_t i0, int nc, int kind, double eps2, double *__restrict__ B) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= N * nc) return;
    const int64_t j = e / nc, ii = e - j * nc;
    const double *p = P + 3 * (i0 + ii);
    const double dx = X[3 * j] - p[0], dy = X[3 * j + 1] - p[1], dz = X[3 * j + 2] - p[2];
    B[e] = global_radial(kind, eps2, dx * dx + dy * dy + dz * dz);
}

// E[i0 + ii][j] = C[j][ii] through a 32 x 32 shared tile (both sides coalesced), converted to
// the storage type (FP64, or an FP32 pair hi = fl(e), lo = fl(e - hi)).
template <typename V>
__global__ void cardinal_store(const double *__restrict__ C, int64_t N, int nc, int64_t i0,
                               V *__restrict__ E) {
    __shared__ double tile[32][33];
    const int64_t j0 = blockIdx.x * 32ll;
    const int ii0 = blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;
    for (int r = ty; r < 32; r += 8) {
        const int64_t j = j0 + r;
        const int ii = ii0 + tx;
        tile[r][tx] = (j < N && ii < nc) ? C[j * nc + ii] : 0.0;
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int ii = ii0 + r;
        const int64_t j = j0 + tx;
        if (ii < nc && j < N) E[(i0 + ii) * N + j] = wcast<V>(tile[tx][r]);
    }
}

}  // namespace

int global_cardinal_build(const double *LU, const int32_t *perm, const double *X, int64_t N, int kind,
                          double eps, const double *P, int64_t Nq, void *E, int e_dtype, cudaStream_t s) {
    if (Nq == 0) return RBFSL_OK;
    const int ncmax = (int)std::min<int64_t>(kCardChunk, Nq);
    double *B = nullptr, *C = nullptr;
    char *ws = nullptr;  // the solve's inverted blocks and scratch, for all blocks of points
    const size_t fb = split_solve_factor_bytes(N);
    RBFSL_CUDA_TRY(cudaMalloc(&B, (size_t)N * ncmax * sizeof(double)));
    if (cudaMalloc(&C, (size_t)N * ncmax * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&ws, fb + split_solve_scratch_bytes(N, ncmax)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(B);
        cudaFree(C);
        set_error("global_cardinal: cudaMalloc failed");
        return RBFSL_ENOMEM;
    }
    int rc = split_solve_prepare(LU, N, ws, s);
    for (int64_t i0 = 0; i0 < Nq && rc == RBFSL_OK; i0 += ncmax) {
        const int nc = (int)std::min<int64_t>(ncmax, Nq - i0);
        const int64_t cnt = N * nc;
        cardinal_rhs<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(X, N, P, i0, nc, kind, eps * eps, B);
        rc = split_solve(LU, perm, N, B, nc, C, ws, ws + fb, s);
        if (rc) break;
        dim3 grid((unsigned)((N + 31) / 32), (unsigned)((nc + 31) / 32)), block(32, 8);
        if (e_dtype == RBFSL_F64) cardinal_store<double><<<grid, block, 0, s>>>(C, N, nc, i0, (double *)E);
        else cardinal_store<float2><<<grid, block, 0, s>>>(C, N, nc, i0, (float2 *)E);
        rc = launch_status("global_cardinal");
    }
    const cudaError_t e = cudaStreamSynchronize(s);
    cudaFree(B);
    cudaFree(C);
    cudaFree(ws);
    if (rc == RBFSL_OK && e != cudaSuccess) {
        set_error(std::string("global_cardinal: ") + cudaGetErrorString(e));
        rc = RBFSL_ECUDA;
    }
    return rc;
}

// Whole fields of partial sums (Nq x T doubles), the digits of q among them.
size_t cardinal_apply_workspace(int64_t Nq, int64_t N, int T) {
    if (Nq == 0) return 0;
    const size_t need = std::max(split_product_bytes(Nq, N, T, RBFSL_F64), split_product_bytes(Nq, N, T, RBFSL_F32X2));
    const size_t field = (size_t)Nq * T * sizeof(double);
    return (need + field - 1) / field * field;
}

int launch_cardinal_apply(const void *E, int64_t Nq, int64_t N, const void *q, int T, int dtype, void *out,
                          void *ws, size_t ws_bytes, cudaStream_t s) {
    if (Nq == 0) return RBFSL_OK;
    if (ws_bytes < cardinal_apply_workspace(Nq, N, T) || !ws) {
        set_error("cardinal_apply: workspace too small");
        return RBFSL_EINVAL;
    }
    return split_apply(E, Nq, N, q, T, dtype, out, ws, s);
}

}  // namespace rbfsl

extern "C" int rbfsl_global_cardinal(const double *LU, const int32_t *perm, const double *x, int64_t N,
                                     int kernel, double eps, const double *p, int64_t Nq, void *E,
                                     int e_dtype, void *stream) {
    using namespace rbfsl;
    RBFSL_CHECK_ARG(N >= 1 && Nq >= 0, "global_cardinal: bad sizes");
    RBFSL_CHECK_ARG(kernel == RBFSL_GAUSS || kernel == RBFSL_IMQ, "global_cardinal: kernel must be GAUSS or IMQ");
    RBFSL_CHECK_ARG(eps > 0 && std::isfinite(eps), "global_cardinal: eps must be positive");
    RBFSL_CHECK_ARG(e_dtype == RBFSL_F64 || e_dtype == RBFSL_F32X2, "global_cardinal: bad e_dtype");
    RBFSL_CHECK_ARG(Nq == 0 || (LU && perm && x && p && E), "global_cardinal: null pointer");
    return global_cardinal_build(LU, perm, x, N, kernel, eps, p, Nq, E, e_dtype, (cudaStream_t)stream);
}

extern "C" size_t rbfsl_cardinal_apply_workspace_bytes(int64_t Nq, int64_t N, int T) {
    if (Nq < 0 || N < 1 || T < 1) return 0;
    return rbfsl::cardinal_apply_workspace(Nq, N, T);
}

extern "C" int rbfsl_cardinal_apply(const void *E, int64_t Nq, int64_t N, const void *q, int T, int dtype,
                                    void *q_out, void *workspace, size_t workspace_bytes, void *stream) {
    using namespace rbfsl;
    RBFSL_CHECK_ARG(Nq >= 0 && N >= 1 && T >= 1, "cardinal_apply: bad sizes");
    RBFSL_CHECK_ARG(dtype == RBFSL_F64 || dtype == RBFSL_F32X2, "cardinal_apply: bad dtype");
    RBFSL_CHECK_ARG(Nq == 0 || (E && q && q_out), "cardinal_apply: null pointer");
    RBFSL_CHECK_ARG(q_out != q, "cardinal_apply: q_out may not alias q");
    return launch_cardinal_apply(E, Nq, N, q, T, dtype, q_out, workspace, workspace_bytes, (cudaStream_t)stream);
}
