// Dense products out = A x to FP64 accuracy on the tensor cores (split_mma.cuh), for the three
// places of the global method that an FP64 product bounds: the trailing updates of the triangular
// solves (A: strips of the factor), the evaluation (A: kernel values formed on the way) and the
// cardinal form (A: the stored cardinal matrix, FP64 or FP32 pairs).
//
// The inner dimension is walked in chunks of 128: up to there the digit sums stay exact in the FP32
// accumulators (128 terms x 8 products x 2^14 = 2^24). Each chunk's sums are scaled by the row's and
// the column's own largest exponent of the chunk and added in FP64. x is cut into digits once
// (x_digits); A's rows are cut by the block that uses them: a warp reads a row's 128 entries, takes
// their largest exponent with one redux and leaves the digits in shared memory.
//
// Blocks of four warps: 16 rows x 32 columns per warp, as 2 x 2 warps (32 rows x 64 columns) or,
// for up to 32 columns, 4 x 1 (64 rows). Bound: the tensor cores' FP16 rate, 43 digit products per
// useful one (43 N^2 T / 304 TMAC/s: 0.95 ms at N = 10,242, T = 64, where the FP64 pipe takes
// 10.7 ms; the cardinal product 1.9 ms there, tensor pipe 45% busy, 612 us at N = 5,003, the rest digit extraction
// between a chunk's barriers); for few columns the digit extraction and the A stream; in the evaluation the FP64
// kernel values (5.4 ms for the same sizes with the Gaussian, 18.0 in FP64; FP64 pipe 78% busy).
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "split_gemm.cuh"
#include "split_mma.cuh"

namespace rbfsl {

namespace {

constexpr int kChunk = kSplitChunk;
constexpr int kLd = 136;  // shared row of a chunk's digits (16-byte loads of eight rows hit all banks)
constexpr int kENan = 0x7ff;

// The common exponent E of a row's or a column's chunk, |x| < 2^(E - 1023), from the largest key of its numbers (a
// key grows with the magnitude): 2 for subnormal numbers, above kENan where one is not finite, in the middle of the
// range for zeros, which are exact at any scale. A key of A's entries is their upper word alone (below 2^-1042 they
// count as zeros), one operation for each.
__device__ __forceinline__ int key_of(double x) {
    return (__double2hiint(x) & 0x7fffffff) | (__double2loint(x) != 0);
}
__device__ __forceinline__ int chunk_exponent(int key) { return key == 0 ? 1024 : max(key >> 20, 1) + 1; }

// ---- sources of A: raw 64-bit words, their keys, their digits, their value
struct SrcF64 {
    const double *A;
    int64_t ld;
    __device__ __forceinline__ unsigned long long raw(int64_t r, int64_t k) const {
        return (unsigned long long)__double_as_longlong(A[r * ld + k]);
    }
    __device__ __forceinline__ static int key(unsigned long long w) { return (int)(w >> 32) & 0x7fffffff; }
    __device__ __forceinline__ static int exponent(int key) { return chunk_exponent(key); }
    __device__ __forceinline__ static unsigned long long digits(unsigned long long w, int E) {
        return digits_of(__longlong_as_double((long long)w), E);
    }
    __device__ __forceinline__ static double value(unsigned long long w) { return __longlong_as_double((long long)w); }
};

// v (a float) as a multiple of 2^(E - 1023 - 61), truncated (no byte bias).
__device__ __forceinline__ long long fixed_of(uint32_t w, int E) {
    const int e = (int)(w >> 23) & 0xff;
    const long long m = (w & 0x7fffff) | (e ? 1u << 23 : 0u);
    // m 2^(e' - 150) with e' = max(e, 1): shift 61 + 1023 - 150 - E + e'
    const int s = (e ? e : 1) + 934 - E;
    const long long v = s >= 0 ? m << (s > 40 ? 40 : s) : (s > -63 ? m >> -s : 0);
    return (int)w < 0 ? -v : v;
}

struct SrcPair {
    const float2 *A;
    int64_t ld;
    __device__ __forceinline__ unsigned long long raw(int64_t r, int64_t k) const {
        const float2 v = A[r * ld + k];
        return (unsigned long long)__float_as_uint(v.x) | (unsigned long long)__float_as_uint(v.y) << 32;
    }
    __device__ __forceinline__ static int key(unsigned long long w) {  // of the larger part
        return max((int)w & 0x7fffffff, (int)(w >> 32) & 0x7fffffff);
    }
    __device__ __forceinline__ static int exponent(int key) {
        return key == 0 ? 1024 : key >= 0x7f800000 ? kENan + 1 : (key >> 23) + 897;
    }
    __device__ __forceinline__ static unsigned long long digits(unsigned long long w, int E) {
        return (unsigned long long)(fixed_of((uint32_t)w, E) + fixed_of((uint32_t)(w >> 32), E)) + 0x8080808080808080ULL;
    }
    __device__ __forceinline__ static double value(unsigned long long w) {
        return (double)__uint_as_float((uint32_t)w) + (double)__uint_as_float((uint32_t)(w >> 32));
    }
};

struct SrcPhi : SrcF64 {
    const double *P, *X;
    int kind;
    double eps2;
    __device__ __forceinline__ unsigned long long raw(int64_t r, int64_t k) const {
        const double dx = P[3 * r] - X[3 * k], dy = P[3 * r + 1] - X[3 * k + 1], dz = P[3 * r + 2] - X[3 * k + 2];
        return (unsigned long long)__double_as_longlong(
            global_radial(kind, eps2, fma(dz, dz, fma(dy, dy, dx * dx))));
    }
};

__device__ __forceinline__ double x_value(const double *x) { return *x; }
__device__ __forceinline__ double x_value(const float2 *x) { return (double)x->x + (double)x->y; }

constexpr int kExtra = 2, kExTop = 4096;  // entries behind a chunk's exponents
__device__ __forceinline__ void column_extremes(int *e, int E) {
    atomicMax(e, E);
    atomicMax(e + 1, kExTop - E);
}

// Digits of x (K x T, row-major), chunk blockIdx.x, columns blockIdx.y * 32 .. + 32: D[chunk][k][t]
// (row length Tp), the columns' exponents Ex[chunk][t] (chunk_exponent), their largest, Ex[chunk][Tp], and
// kExTop less their smallest, Ex[chunk][Tp + 1] (zeroed by the caller).
template <typename V>
__global__ void __launch_bounds__(256) x_digits(const V *__restrict__ x, int64_t K, int T, int Tp,
                                                unsigned long long *__restrict__ D, int *__restrict__ Ex) {
    __shared__ int emax[32];
    const int c = threadIdx.x & 31, w = threadIdx.x >> 5, t = blockIdx.y * 32 + c;
    const int64_t ch = blockIdx.x, k0 = ch * kChunk;
    if (threadIdx.x < 32) emax[threadIdx.x] = 0;
    __syncthreads();
    double v[kChunk / 8];
    int e = 0;
#pragma unroll
    for (int u = 0; u < kChunk / 8; ++u) {
        const int64_t k = k0 + w + 8 * u;
        v[u] = k < K && t < T ? x_value(x + k * T + t) : 0.0;
        e = max(e, key_of(v[u]));
    }
    atomicMax(&emax[c], e);
    __syncthreads();
    const int E = chunk_exponent(emax[c]);
    if (t < Tp) {
#pragma unroll
        for (int u = 0; u < kChunk / 8; ++u) D[(k0 + w + 8 * u) * Tp + t] = digits_of(v[u], E);
        if (w == 0) {
            int *ex = Ex + ch * (Tp + kExtra);
            ex[t] = E;
            column_extremes(ex + Tp, E);
        }
    }
}

// Scale of a chunk's sums, 2^(EA + EX - 2 * 1023 - 34), and whether it is a normal double.
__device__ __forceinline__ bool chunk_tiny(int EA, int EX) { return EA + EX <= 1023 + 34; }
__device__ __forceinline__ double chunk_scale(int EA, int EX) {
    return __longlong_as_double((long long)(EA + EX - 1023 - 34) << 52);
}
// v times that scale for any EA and EX, in two factors (0 for one below the normal doubles: v < 2^62). The
// second of two paths: a warp takes it where one of its scales may not be a normal double.
__device__ __forceinline__ double chunk_scaled(double v, int EA, int EX) {
    const int X = EA + EX - 2 * 1023 - 34, a = X >> 1, b = X - a;
    return v * __longlong_as_double((long long)max(a + 1023, 0) << 52) * __longlong_as_double((long long)max(b + 1023, 0) << 52);
}

// Whether a chunk's sums need plain FP64: rows or columns that are not finite, or results beyond
// the doubles' range.
__device__ __forceinline__ bool chunk_bad(int ea_max, int ex_max) {
    return ea_max > kENan || ex_max > kENan || ea_max + ex_max >= 2047 + 1023 + 34;
}

// To out (row length T) + split * M * T.
template <typename Src, typename V, int kWarpRows>
__global__ void __launch_bounds__(128, 3) split_gemm_kernel(Src A, int64_t M, int64_t K, const V *__restrict__ x, int T,
                                                            int Tp, const unsigned long long *__restrict__ D,
                                                            const int *__restrict__ Ex, int nchunk, int span,
                                                            double *__restrict__ out) {
    constexpr int kRows = 16 * kWarpRows, kWarpCols = 4 / kWarpRows;
    extern __shared__ __align__(16) unsigned long long As[];  // kRows x kLd digits
    __shared__ int Er[kRows];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t2 = (lane & 3) * 2;
    const int64_t r0 = (int64_t)blockIdx.x * kRows;
    const int wr = (warp / kWarpCols) * 16, col0 = (blockIdx.y * kWarpCols + warp % kWarpCols) * 32;
    const int c0 = blockIdx.z * span, c1 = min(nchunk, c0 + span);
    double sum[4][4] = {};
    for (int ch = c0; ch < c1; ++ch) {
        const int64_t k0 = (int64_t)ch * kChunk;
        const int kc = (int)min((int64_t)kChunk, K - k0);
        // ---- digits of the block's rows, four rows of a warp at a time
        bool bad = false;
        const int *ex = Ex + (int64_t)ch * (Tp + kExtra);
        const int exm = ex[Tp], exs = kExTop - ex[Tp + 1];
        for (int q = 0; q < kRows / 4; q += 4) {
            unsigned long long w[4][4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int64_t r = r0 + warp * (kRows / 4) + q + v;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = lane + 32 * u;
                    w[v][u] = r < M && k < kc ? A.raw(r, k0 + k) : 0ULL;
                }
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int row = warp * (kRows / 4) + q + v;
                int e = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) e = max(e, Src::key(w[v][u]));
                const int E = Src::exponent(__reduce_max_sync(0xffffffffu, e));
                if (lane == 0) Er[row] = E;
                bad |= chunk_bad(E, exm);
#pragma unroll
                for (int u = 0; u < 4; ++u) As[row * kLd + lane + 32 * u] = Src::digits(w[v][u], E);
            }
        }
        if (__syncthreads_or(bad)) {
            // not finite, or beyond the doubles' range: this chunk in plain FP64
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t r = r0 + wr + g + 8 * (u >> 1);
                    const int t = col0 + 8 * nt + t2 + (u & 1);
                    if (r < M && t < T)
#pragma unroll 1
                        for (int k = 0; k < kc; ++k)
                            sum[nt][u] = fma(Src::value(A.raw(r, k0 + k)), x_value(x + (k0 + k) * T + t), sum[nt][u]);
                }
        } else {
            const int ea[2] = {Er[wr + g], Er[wr + g + 8]};
            const bool tiny = __any_sync(0xffffffffu, chunk_tiny(min(ea[0], ea[1]), exs));
#pragma unroll
            for (int np = 0; np < 2; ++np) {  // two 8-column tiles at a time
                const int cb = col0 + 16 * np;
                if (cb >= Tp) break;
                const bool two = cb + 8 < Tp;
                float acc[2][kGroups][4] = {};
                for (int ks = 0; ks * 16 < kc; ++ks) {
                    const unsigned long long *a = As + (wr + g) * kLd + ks * 16 + t2;
                    const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(a),
                                     a1 = *reinterpret_cast<const ulonglong2 *>(a + 8 * kLd),
                                     a2 = *reinterpret_cast<const ulonglong2 *>(a + 8),
                                     a3 = *reinterpret_cast<const ulonglong2 *>(a + 8 * kLd + 8);
                    const unsigned long long *d = D + (k0 + ks * 16 + t2) * Tp + cb + g;
                    uint32_t b[2][kDigits][2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1 && !two) break;
                        const unsigned long long b0 = d[8 * h], b1 = d[Tp + 8 * h], b2 = d[8 * Tp + 8 * h],
                                                 b3 = d[9 * Tp + 8 * h];
#pragma unroll
                        for (int s = 0; s < kDigits; ++s) {
                            b[h][s][0] = digit_pair(b0, b1, s);
                            b[h][s][1] = digit_pair(b2, b3, s);
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int s = 0; s < kDigits; ++s) {
                        const uint32_t af[4] = {digit_pair(a0.x, a0.y, s), digit_pair(a1.x, a1.y, s),
                                                digit_pair(a2.x, a2.y, s), digit_pair(a3.x, a3.y, s)};
#pragma unroll
                        for (int q = 0; q < kDigits && s + q < kGroups; ++q) {
                            mma_f16(acc[0][s + q], af, b[0][q]);
                            if (two) mma_f16(acc[1][s + q], af, b[1][q]);
                        }
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (h == 1 && !two) break;
                    const int et[2] = {ex[cb + 8 * h + t2], ex[cb + 8 * h + t2 + 1]};
                    if (!tiny) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            sum[2 * np + h][u] = fma(split_value(acc[h], u), chunk_scale(ea[u >> 1], et[u & 1]),
                                                     sum[2 * np + h][u]);
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            sum[2 * np + h][u] += chunk_scaled(split_value(acc[h], u), ea[u >> 1], et[u & 1]);
                        __syncwarp();
                    }
                }
            }
        }
        __syncthreads();  // the digits are read; the next chunk overwrites them
    }
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t r = r0 + wr + g + 8 * (u >> 1);
            const int t = col0 + 8 * nt + t2 + (u & 1);
            if (r >= M || t >= T) continue;
            out[((int64_t)blockIdx.z * M + r) * T + t] = sum[nt][u];
        }
}

template <typename Src, typename V>
int launch_gemm(const Src &A, int64_t M, int64_t K, const V *x, int T, int Tp, const unsigned long long *D, const int *Ex,
                int splits, double *out, cudaStream_t s) {
    const int nchunk = (int)((K + kChunk - 1) / kChunk), span = (nchunk + splits - 1) / splits;
    auto go = [&](auto *kernel, int rows, int cols) {
        const int smem = rows * kLd * 8;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return;
        dim3 grid((unsigned)((M + rows - 1) / rows), (unsigned)((T + cols - 1) / cols), (unsigned)splits);
        kernel<<<grid, 128, smem, s>>>(A, M, K, x, T, Tp, D, Ex, nchunk, span, out);
    };
    if (T <= 32) go(split_gemm_kernel<Src, V, 4>, 64, 32);
    else go(split_gemm_kernel<Src, V, 2>, 32, 64);
    return launch_status("split_gemm");
}

// ---- triangular solves with diagonal blocks of 128 rows
constexpr int kB = 64;  // inverted triangular blocks (two to a diagonal block)
// Condition of a block above which its inverse's product is corrected (solve_diag). Residuals of whole solves against
// plain substitution's, Gaussian and IMQ factors of 1,000 to 10,242 nodes from well conditioned to flat, sixteen
// fields each: up to 64 the same as with every block corrected (largest 1.9 times, root mean square 1.1), from 256 on 3.0
// and 1.2, from 1,024 2.9 and 2.2, without corrections 202 and 111. A solve at N = 1,000, T = 16: 469 us with every
// block corrected, 415 (from 16 on), 368 (64), 355 without; at N = 10,242, most blocks below 64, 3.17 ms, 2.71, 2.58, 2.51.
constexpr double kSolveCond = 64.0;

// Programmatic dependent launch: the next kernel of the stream may start (its prologue runs beside this
// kernel), and wait until every kernel before this one is complete. What an earlier kernel of the chain
// wrote is read through pointers without __restrict__: loads that the compiler takes for invariant could
// move ahead of the wait.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_dependencies() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A launch whose blocks may start beside the kernel before it in the stream (they wait in the kernel).
template <typename... P, typename... A>
void launch_after_prologue(void (*kernel)(P...), dim3 grid, int threads, int smem, cudaStream_t s, A... a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(a)...);  // errors: launch_status of the caller
}

// Inverses of the 64 x 64 diagonal blocks of the unit lower (blockIdx.y = 0) and the upper factor
// (1), column-major, and the 64 x 64 block that couples a diagonal block's halves (also
// column-major): what the block substitution needs, laid out for its lanes. A block's inverse
// replaces 64 dependent steps by a product. Rows and columns beyond N: the identity. cond: the blocks'
// Skeel condition numbers.
__global__ void __launch_bounds__(64) solve_prepare(const double *__restrict__ LU, int64_t N, double *__restrict__ inv,
                                                    double *__restrict__ off, double *__restrict__ cond) {
    extern __shared__ double sm[];
    __shared__ double z[kB];
    double *F = sm, *V = sm + kB * (kB + 1);  // the block (row-major) and its inverse (column-major), padded
    const int64_t j = blockIdx.x, r0 = j * kB;
    const int c = threadIdx.x, upper = blockIdx.y;
    for (int i = 0; i < kB; ++i)
        F[i * (kB + 1) + c] = r0 + i < N && r0 + c < N ? LU[(r0 + i) * N + r0 + c] : (i == c ? 1.0 : 0.0);
    __syncthreads();
    double *v = V + c * (kB + 1);
    if (!upper) {
        for (int i = 0; i < kB; ++i) {
            const double *f = F + i * (kB + 1);
            double a = i == c ? 1.0 : 0.0, b = 0.0;
            int q = c;
            for (; q + 1 < i; q += 2) {
                a = fma(-f[q], v[q], a);
                b = fma(-f[q + 1], v[q + 1], b);
            }
            if (q < i) a = fma(-f[q], v[q], a);
            v[i] = i < c ? 0.0 : a + b;
        }
    } else {
        for (int i = kB - 1; i >= 0; --i) {
            const double *f = F + i * (kB + 1);
            double a = i == c ? 1.0 : 0.0, b = 0.0;
            int q = i + 1;
            for (; q + 1 <= c; q += 2) {
                a = fma(-f[q], v[q], a);
                b = fma(-f[q + 1], v[q + 1], b);
            }
            if (q <= c) a = fma(-f[q], v[q], a);
            v[i] = i > c ? 0.0 : (a + b) / f[i];
        }
    }
    __syncthreads();
    double *o = inv + (2 * j + upper) * kB * kB;
    for (int q = 0; q < kB; ++q) o[q * kB + c] = V[q * (kB + 1) + c];
    {  // cond(T) = the largest row sum of |T^-1| |T|; a value that is not finite counts as large
        double a = upper ? 0.0 : 1.0;
        for (int q = upper ? c : 0; q < (upper ? kB : c); ++q) a += fabs(F[c * (kB + 1) + q]);
        z[c] = a;
        __syncthreads();
        a = 0.0;
        for (int q = 0; q < kB; ++q) a = fma(fabs(V[q * (kB + 1) + c]), z[q], a);
        __syncthreads();
        z[c] = a;
        __syncthreads();
        if (c == 0) {
            for (int q = 1; q < kB; ++q) a = z[q] <= a ? a : z[q];
            cond[2 * j + upper] = a <= 1e300 ? a : 1e300;
        }
    }
    if (upper ? !(j & 1) : (j & 1)) {  // lower: rows of an odd block, columns before it; upper: the other half
        const int64_t cb = upper ? r0 + kB : r0 - kB;
        double *p = off + (2 * (j >> 1) + upper) * kB * kB;
        __syncthreads();
        for (int i = 0; i < kB; ++i) F[i * (kB + 1) + c] = r0 + i < N && cb + c < N ? LU[(r0 + i) * N + cb + c] : 0.0;
        __syncthreads();
        for (int q = 0; q < kB; ++q) p[q * kB + c] = F[c * (kB + 1) + q];
    }
}

// One diagonal block (128 rows from r0) for one right-hand side per thread block: forward x1 =
// T11^-1 y1, x2 = T22^-1 (y2 - T21 x1), backward the other way round; x replaces y and its digits go
// to the update. A product with a 64 x 64 inverse alone is not backward stable: its residual grows with
// the block's condition, and the blocks of flat kernels are badly conditioned (Gaussian, eps = 3 on 2,562
// nodes: residual 1.8e-9 against substitution's 5e-11). Where cond(T) exceeds kSolveCond the product is
// corrected once, x += T^-1 (y - T x), with the factor's own block T, which brings the residual back to
// substitution's.
// Eight warps: 16 rows and every second pair of columns each, a lane every fourth column; a triangle's empty
// 16 x 16 tiles are left out, with the rows dealt so that the SM's four schedulers have equal work. Bound:
// the FP64 pipe (a warp instruction keeps its scheduler's quarter busy for 64 cycles, which also hides the
// one chain of FMAs a lane has) and latency; a thread's matrix entries are loaded beside the kernel before
// (columns of the padding are the identity's in the inverses and zero in T, where x is zero too).
__global__ void __launch_bounds__(256, 1) solve_diag(const double *__restrict__ LU, const double *__restrict__ inv,
                                                     const double *__restrict__ off, const double *__restrict__ cond,
                                                     int64_t N, int64_t r0, double *Y, int T, int Tp, int upper,
                                                     unsigned long long *D, int *Ex) {
    __shared__ double y[2 * kB], x[kB], res[kB], part[2 * kB];
    __shared__ int emax;
    const int tid = threadIdx.x, w = tid >> 5, t = blockIdx.x;
    const int rt = w < 4 ? w : 7 - w;                                      // row tile; w and w + 4 share a scheduler
    const int i = rt * 16 + (tid & 15), h = 2 * (w >> 2) + ((tid >> 4) & 1);  // row, column class (mod 4)
    const int64_t b = r0 / kB;
    const int f = upper ? kB : 0, s = kB - f;  // first and second half in the order of the substitution
    const int64_t bf = b + (upper ? 1 : 0), bs = b + (upper ? 0 : 1);
    const bool two = r0 + kB < N;  // the block has a second half
    const bool first = !upper || two, second = two || upper;
    const bool c1 = first && cond[2 * bf + upper] > kSolveCond, c2 = second && cond[2 * bs + upper] > kSolveCond;
    launch_dependents();
    constexpr int kQ = kB / 4;  // columns of a thread
    double v1[kQ], t1[kQ], o[kQ], v2[kQ], t2[kQ];
    auto load = [&](double(&m)[kQ], bool on, const double *p) {
#pragma unroll
        for (int q = 0; q < kQ; ++q) m[q] = on ? p[(4 * q + h) * kB + i] : 0.0;
    };
    auto load_t = [&](double(&m)[kQ], bool on, int64_t rb) {  // the triangle at row rb
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const int c = 4 * q + h;
            const bool in = on && (upper ? c >= i : c < i) && rb + i < N && rb + c < N;
            m[q] = in ? LU[(rb + i) * N + rb + c] : (!upper && c == i ? 1.0 : 0.0);
        }
    };
    load(v1, first, inv + (2 * bf + upper) * kB * kB);
    load_t(t1, c1, r0 + f);
    load(o, two, off + (2 * (b >> 1) + upper) * kB * kB);
    load(v2, second, inv + (2 * bs + upper) * kB * kB);
    load_t(t2, c2, r0 + s);
    if (tid == 0) emax = 0;
    wait_dependencies();
    if (tid < 2 * kB) y[tid] = t < T && r0 + tid < N ? Y[(r0 + tid) * T + t] : 0.0;
    __syncthreads();
    // row i of a product over the columns of the tiles [k0, k1); the two warps' parts are added up by the
    // threads of h == 0
    auto product = [&](const double(&m)[kQ], const double *v, int k0, int k1) {
        double a0 = 0.0, a1 = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k < k0 || k >= k1) continue;  // warp-uniform
#pragma unroll
            for (int q = 4 * k; q < 4 * k + 4; q += 2) {
                a0 = fma(m[q], v[4 * q + h], a0);
                a1 = fma(m[q + 1], v[4 * q + 4 + h], a1);
            }
        }
        double a = a0 + a1;
        a += __shfl_xor_sync(0xffffffffu, a, 16);
        if (!(h & 1)) part[(h >> 1) * kB + i] = a;
        __syncthreads();
    };
    auto sum = [&] { return part[i] + part[kB + i]; };
    const int k0 = upper ? rt : 0, k1 = upper ? 4 : rt + 1;  // a triangle's tiles
    auto solve = [&](const double(&v)[kQ], const double(&m)[kQ], double *yh, bool correct) {
        product(v, yh, k0, k1);
        if (h == 0) (correct ? x : yh)[i] = sum();
        __syncthreads();
        if (!correct) return;  // block-uniform
        product(m, x, k0, k1);
        if (h == 0) res[i] = yh[i] - sum();
        __syncthreads();
        product(v, res, k0, k1);
        if (h == 0) yh[i] = x[i] + sum();
        __syncthreads();
    };
    if (first) solve(v1, t1, y + f, c1);
    if (two) {
        product(o, y + f, 0, 4);
        if (h == 0) y[s + i] -= sum();
        __syncthreads();
    }
    if (second) solve(v2, t2, y + s, c2);
    if (tid < 2 * kB) {
        const double v = r0 + tid < N ? y[tid] : 0.0;
        if (t < T && r0 + tid < N) Y[(r0 + tid) * T + t] = v;
        const int e = __reduce_max_sync(0xffffffffu, key_of(v));
        if ((tid & 31) == 0) atomicMax(&emax, e);
    }
    __syncthreads();
    const int E = chunk_exponent(emax);
    if (tid < 2 * kB) D[(int64_t)tid * Tp + t] = digits_of(r0 + tid < N ? y[tid] : 0.0, E);
    if (tid == 0) {
        Ex[t] = E;
        column_extremes(Ex + Tp, E);
    }
}

// The solve's update C[r][t] -= sum over k < kc of A[r][k] x[k][t], 16 rows and 64 / KW columns a block:
// KW warps along k and 4 / KW along the columns (16 each). One launch of a chain of 2 N / 128, each
// waiting for the one before: few rows a block, the factor's digits formed beside the kernel before, and,
// where that leaves SMs idle, the inner dimension split over the warps (launch_update). N = 4,999, T = 9, a step (80 links, evaluation
// 0.83 ms): 64-row blocks with a warp's whole inner dimension, each link after the one before 3.30 ms, now
// 1.85; N = 10,242, T = 64 (160 links) 7.37 ms, with prologues beside the link before 6.89, now 3.99 (4.20 before
// solve_diag left out the triangles' empty tiles).
constexpr int64_t kUpdateBlocks = 4 * 152;

template <int KW>
__global__ void __launch_bounds__(128, 3) solve_update(SrcF64 A, int64_t M, int kc, const double *x, int T, int Tp,
                                                       const unsigned long long *D, const int *Ex, double *C) {
    constexpr int CW = 4 / KW, kCols = 16 * CW, kSteps = 8 / KW;
    __shared__ __align__(16) unsigned long long As[16 * kLd];
    __shared__ double part[KW][16 * kCols];
    __shared__ int Er[16];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t2 = (lane & 3) * 2;
    const int64_t r0 = (int64_t)blockIdx.x * 16;
    const int col0 = blockIdx.y * kCols;
    launch_dependents();
    int ea_max = 0;
    {
        unsigned long long w[4][4];
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t r = r0 + 4 * warp + v;
                const int k = lane + 32 * u;
                w[v][u] = r < M && k < kc ? A.raw(r, k) : 0ULL;
            }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            int e = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) e = max(e, SrcF64::key(w[v][u]));
            const int E = SrcF64::exponent(__reduce_max_sync(0xffffffffu, e));
            if (lane == 0) Er[4 * warp + v] = E;
            ea_max = max(ea_max, E);
#pragma unroll
            for (int u = 0; u < 4; ++u) As[(4 * warp + v) * kLd + lane + 32 * u] = SrcF64::digits(w[v][u], E);
        }
    }
    wait_dependencies();
    const int kw = warp / CW, cb = col0 + 16 * (warp % CW);
    const bool on = cb < Tp, two = cb + 8 < Tp;
    unsigned long long nx[2][2][4];  // x's digits (D has 128 rows, zeros behind kc), a step ahead
    auto load = [&](int q, unsigned long long(&d)[2][4]) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int v = 0; v < 4; ++v)
                d[h][v] = on && (h == 0 || two)
                              ? D[(int64_t)((kw * kSteps + q) * 16 + t2 + (v & 1) + 8 * (v >> 1)) * Tp + cb + 8 * h + g]
                              : kZeroDigits;
    };
    load(0, nx[0]);
    constexpr int kOut = 16 * kCols / 128;  // outputs of a thread: row, then column
    double old[kOut];
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
        const int e = threadIdx.x + 128 * o, r = e / kCols, t = col0 + e % kCols;
        old[o] = r0 + r < M && t < T ? C[(r0 + r) * T + t] : 0.0;
    }
    const bool bad = __syncthreads_or(chunk_bad(ea_max, Ex[Tp]));
    if (!bad && on) {
        float acc[2][kGroups][4] = {};
#pragma unroll
        for (int q = 0; q < kSteps; ++q) {
            if (q + 1 < kSteps) load(q + 1, nx[(q + 1) & 1]);
            const unsigned long long *a = As + g * kLd + (kw * kSteps + q) * 16 + t2;
            const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(a),
                             a1 = *reinterpret_cast<const ulonglong2 *>(a + 8),
                             a2 = *reinterpret_cast<const ulonglong2 *>(a + 8 * kLd),
                             a3 = *reinterpret_cast<const ulonglong2 *>(a + 8 * kLd + 8);
            const unsigned long long av[8] = {a0.x, a0.y, a1.x, a1.y, a2.x, a2.y, a3.x, a3.y};
            uint32_t b[kDigits][2];
            digit_frags(b, nx[q & 1][0][0], nx[q & 1][0][1], nx[q & 1][0][2], nx[q & 1][0][3]);
            split_products(acc[0], av, b);
            if (two) {
                digit_frags(b, nx[q & 1][1][0], nx[q & 1][1][1], nx[q & 1][1][2], nx[q & 1][1][3]);
                split_products(acc[1], av, b);
            }
        }
        const int ea[2] = {Er[g], Er[g + 8]};
        const bool tiny = __any_sync(0xffffffffu, chunk_tiny(min(ea[0], ea[1]), kExTop - Ex[Tp + 1]));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && !two) break;
            const int t = cb + 8 * h + t2, et[2] = {Ex[t], Ex[t + 1]};
            double *o = &part[kw][g * kCols + t - col0];
            if (!tiny) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    o[8 * kCols * (u >> 1) + (u & 1)] = split_value(acc[h], u) * chunk_scale(ea[u >> 1], et[u & 1]);
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    o[8 * kCols * (u >> 1) + (u & 1)] = chunk_scaled(split_value(acc[h], u), ea[u >> 1], et[u & 1]);
                __syncwarp();
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
        const int e = threadIdx.x + 128 * o, r = e / kCols, t = col0 + e % kCols;
        if (r0 + r >= M || t >= T) continue;
        double v = 0.0;
        if (!bad) {
            v = part[0][e];
#pragma unroll
            for (int k = 1; k < KW; ++k) v += part[k][e];
        } else {  // not finite, or beyond the doubles' range: plain FP64
#pragma unroll 1
            for (int k = 0; k < kc; ++k) v = fma(SrcF64::value(A.raw(r0 + r, k)), x[(int64_t)k * T + t], v);
        }
        C[(r0 + r) * T + t] = old[o] - v;
    }
}

// KW by the number of blocks: as many warps along k as keep the blocks to four for each of the 152 SMs
// (N = 10,242, T = 64: two 4.43 ms a step, four 4.20, eight 4.21).
int launch_update(const SrcF64 &A, int64_t M, int kc, const double *x, int T, int Tp, const unsigned long long *D,
                  const int *Ex, double *C, cudaStream_t s) {
    const int64_t rows = (M + 15) / 16;
    auto grid = [&](int kw) { return dim3((unsigned)rows, (unsigned)((T * kw + 63) / 64)); };
    auto fits = [&](int kw) { return rows * ((T * kw + 63) / 64) <= kUpdateBlocks; };
    if (fits(4) || T <= 16) launch_after_prologue(solve_update<4>, grid(4), 128, 0, s, A, M, kc, x, T, Tp, D, Ex, C);
    else if (fits(2) || T <= 32) launch_after_prologue(solve_update<2>, grid(2), 128, 0, s, A, M, kc, x, T, Tp, D, Ex, C);
    else launch_after_prologue(solve_update<1>, grid(1), 128, 0, s, A, M, kc, x, T, Tp, D, Ex, C);
    return launch_status("solve_update");
}

__global__ void solve_gather(const double *__restrict__ Q, const int32_t *__restrict__ perm, int64_t N, int T,
                             double *__restrict__ Y) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= N * T) return;
    const int64_t i = e / T;
    Y[e] = Q[(int64_t)perm[i] * T + (e - i * T)];
}

// out[e] = sum over splits s = 0..S-1 (in that order) of part[s][e], FP64 or an FP32 pair.
template <typename V>
__global__ void split_reduce(const double *__restrict__ part, int64_t cnt, int S, V *__restrict__ out) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= cnt) return;
    double s = part[e];
    for (int k = 1; k < S; ++k) s += part[k * cnt + e];
    out[e] = wcast<V>(s);
}

inline int pad8(int T) { return (T + 7) / 8 * 8; }
inline size_t up256(size_t b) { return (b + 255) & ~(size_t)255; }

struct Plan {
    int splits;
    size_t digits, exps, part;
};

// Splits of the inner dimension: whole rounds of the resident blocks (three per SM), each split as
// long as possible; half a chunk stands for a block's fixed cost.
Plan plan(int64_t M, int64_t K, int T, bool direct) {
    int sms = 152, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        cudaGetLastError();
    const int64_t rows = T <= 32 ? 64 : 32, cols = T <= 32 ? 32 : 64, nchunk = (K + kChunk - 1) / kChunk;
    const int64_t tiles = ((M + rows - 1) / rows) * ((T + cols - 1) / cols);
    Plan p{1, 0, 0, 0};
    double best = 1e300;
    for (int64_t S = 1; S <= 32 && S <= nchunk; ++S) {
        const int64_t span = (nchunk + S - 1) / S;
        if ((nchunk + span - 1) / span != S) continue;
        const int64_t waves = (tiles * S + 3 * sms - 1) / (3 * sms);
        const double cost = (double)waves * ((double)span + 0.5);
        if (cost < 0.97 * best) {
            best = cost;
            p.splits = (int)S;
        }
    }
    p.digits = up256((size_t)nchunk * kChunk * pad8(T) * 8);
    p.exps = up256((size_t)nchunk * (pad8(T) + kExtra) * sizeof(int));
    p.part = p.splits > 1 || !direct ? (size_t)p.splits * M * T * sizeof(double) : 0;
    return p;
}

template <typename Src, typename V, typename O>
int product(const Src &A, int64_t M, int64_t K, const V *x, int T, O *out, void *ws, cudaStream_t s) {
    constexpr bool direct = std::is_same<O, double>::value;
    const Plan p = plan(M, K, T, direct);
    const int Tp = pad8(T), nchunk = (int)((K + kChunk - 1) / kChunk);
    unsigned long long *D = (unsigned long long *)ws;
    int *Ex = (int *)((char *)ws + p.digits);
    double *part = (double *)((char *)ws + p.digits + p.exps);
    RBFSL_CUDA_TRY(cudaMemsetAsync(Ex, 0, p.exps, s));
    x_digits<V><<<dim3((unsigned)nchunk, (unsigned)((Tp + 31) / 32)), 256, 0, s>>>(x, K, T, Tp, D, Ex);
    const int rc = launch_gemm<Src, V>(A, M, K, x, T, Tp, D, Ex, p.splits,
                                              p.part ? part : reinterpret_cast<double *>(out), s);
    if (rc || !p.part) return rc;
    const int64_t cnt = M * T;
    split_reduce<O><<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(part, cnt, p.splits, out);
    return launch_status("split product");
}

}  // namespace

size_t split_product_bytes(int64_t M, int64_t K, int T, int out_dtype) {
    const Plan p = plan(M, K, T, out_dtype == RBFSL_F64);
    return p.digits + p.exps + p.part;
}

int split_apply(const void *E, int64_t M, int64_t K, const void *x, int T, int dtype, void *out, void *ws,
                cudaStream_t s) {
    if (dtype == RBFSL_F64)
        return product(SrcF64{(const double *)E, K}, M, K, (const double *)x, T, (double *)out, ws, s);
    return product(SrcPair{(const float2 *)E, K}, M, K, (const float2 *)x, T, (float2 *)out, ws, s);
}

int split_eval(const double *P, int64_t M, const double *X, int64_t K, int kind, double eps, const double *c, int T,
               int out_dtype, void *out, void *ws, cudaStream_t s) {
    SrcPhi A{};
    A.P = P; A.X = X; A.kind = kind; A.eps2 = eps * eps;
    if (out_dtype == RBFSL_F64) return product(A, M, K, c, T, (double *)out, ws, s);
    return product(A, M, K, c, T, (float2 *)out, ws, s);
}

size_t split_solve_factor_bytes(int64_t N) {
    const int64_t b = (N + kB - 1) / kB;
    return (size_t)(2 * b + 2 * ((b + 1) / 2)) * kB * kB * sizeof(double) + up256((size_t)2 * b * sizeof(double));
}

size_t split_solve_scratch_bytes(int64_t N, int T) {
    const int64_t b = (N + kChunk - 1) / kChunk;
    return up256((size_t)kChunk * pad8(T) * 8) + (size_t)2 * b * (pad8(T) + kExtra) * sizeof(int);
}

int split_solve_prepare(const double *LU, int64_t N, void *factor, cudaStream_t s) {
    const int64_t b = (N + kB - 1) / kB;
    double *inv = (double *)factor, *off = inv + 2 * b * kB * kB, *cond = off + 2 * ((b + 1) / 2) * kB * kB;
    const int smem = 2 * kB * (kB + 1) * (int)sizeof(double);
    RBFSL_CUDA_TRY(cudaFuncSetAttribute(solve_prepare, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    solve_prepare<<<dim3((unsigned)b, 2), kB, smem, s>>>(LU, N, inv, off, cond);
    return launch_status("global_solve prepare");
}

int split_solve(const double *LU, const int32_t *perm, int64_t N, const double *Q, int T, double *C, const void *factor,
                void *scratch, cudaStream_t s) {
    const int64_t b64 = (N + kB - 1) / kB, b = (N + kChunk - 1) / kChunk;
    const double *inv = (const double *)factor, *off = inv + 2 * b64 * kB * kB, *cond = off + 2 * ((b64 + 1) / 2) * kB * kB;
    const int Tp = pad8(T);
    unsigned long long *D = (unsigned long long *)scratch;
    int *Ex = (int *)((char *)scratch + up256((size_t)kChunk * Tp * 8));  // one row per block step
    RBFSL_CUDA_TRY(cudaMemsetAsync(Ex, 0, (size_t)2 * b * (Tp + kExtra) * sizeof(int), s));
    solve_gather<<<(unsigned)((N * T + 255) / 256), 256, 0, s>>>(Q, perm, N, T, C);
    for (int64_t j = 0; j < 2 * b; ++j) {
        const int upper = j >= b;
        const int64_t r0 = (upper ? 2 * b - 1 - j : j) * kChunk, nb = std::min<int64_t>(kChunk, N - r0);
        int *ex = Ex + j * (Tp + kExtra);
        launch_after_prologue(solve_diag, dim3((unsigned)Tp), 256, 0, s, LU, inv, off, cond, N, r0, C, T, Tp, upper, D, ex);
        const int64_t first = upper ? 0 : r0 + nb, rows = upper ? r0 : N - r0 - nb;
        if (rows <= 0) continue;
        const SrcF64 A{LU + first * N + r0, N};
        const int rc = launch_update(A, rows, (int)nb, C + r0 * T, T, Tp, D, ex, C + first * T, s);
        if (rc) return rc;
    }
    return launch_status("global_solve");
}

}  // namespace rbfsl
