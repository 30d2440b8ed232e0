// Products of FP64 matrices on the tensor cores by error-free splitting (Ozaki, Ogita, Oishi and
// Rump): each operand is taken as a 62-bit fixed-point number relative to its matrix' largest
// exponent and cut into eight balanced base-256 digits, every digit exact in FP16. A product of
// two digit matrices has integer entries, summed exactly by the FP32 accumulators while they stay
// below 2^24; the digit products of equal weight (digit positions adding up to g) share one
// accumulator. The 43 products of g <= 8 are kept: what is cut off is ~2^-65 of the largest entry
// product (without g = 8, 2^-57: the weights of n = 84 stencils on 642 nodes then lost a digit).
#pragma once

#include "common.cuh"

namespace rbfsl {

constexpr int kDigits = 8, kGroups = 9;
constexpr unsigned long long kZeroDigits = 0x8080808080808080ULL;  // digits_of(0, E)

// Field of x's exponent (biased, 0 for zero and subnormals, 0x7ff for infinities and NaN).
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x as an integer multiple of 2^(E - 1023 - 61), truncated, for |x| < 2^(E - 1023) (E: the largest
// exponent field + 1), plus 128 in every byte, so that byte s reads digit + 128.
__device__ __forceinline__ unsigned long long digits_of(double x, int E) {
    const long long b = __double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff;
    const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffULL) | (e ? 1ULL << 52 : 0ULL);
    int r = E - 1 - (e ? e : 1);
    r = r > 63 ? 63 : r;
    const long long v = (long long)((m << 8) >> r);
    return (unsigned long long)(b < 0 ? -v : v) + 0x8080808080808080ULL;
}

// The number digits_of made (stored in a double's place), its leading 53 bits: exact for a number
// that lost none.
__device__ __forceinline__ double from_digits(double stored, int E) {
    const long long v = (long long)((unsigned long long)__double_as_longlong(stored) - 0x8080808080808080ULL);
    if (v == 0) return 0.0;
    const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    const int z = __clzll((long long)a);  // the leading bit has weight 2^(63 - z), z >= 2
    const unsigned long long m = (a << z) >> 11;
    const long long e = E - 61 + 63 - z;
    if (e <= 0) return 0.0;
    return __longlong_as_double((long long)((v < 0 ? 1ULL << 63 : 0ULL) | ((unsigned long long)e << 52) | (m & 0xfffffffffffffULL)));
}

// Digit s (0: leading) of two numbers as packed FP16.
__device__ __forceinline__ uint32_t digit_pair(unsigned long long x0, unsigned long long x1, int s) {
    const uint32_t w0 = s < 4 ? (uint32_t)(x0 >> 32) : (uint32_t)x0, w1 = s < 4 ? (uint32_t)(x1 >> 32) : (uint32_t)x1;
    const uint32_t q = 3 - (s & 3);  // byte of the word
    uint32_t v = __byte_perm(w0, w1, q | (q << 4) | ((q + 4) << 8) | ((q + 4) << 12));
    v = (v & 0x00ff00ffu) | 0x64006400u;  // 1024 + (digit + 128), exact in FP16
    asm("sub.rn.f16x2 %0, %0, %1;" : "+r"(v) : "r"(0x64806480u));  // - 1152
    return v;
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// The digits of a lane's part of B (16 x 8): rows t, t + 1, t + 8 and t + 9 of its column as FP16 pairs.
__device__ __forceinline__ void digit_frags(uint32_t (&b)[kDigits][2], unsigned long long b0, unsigned long long b1,
                                            unsigned long long b2, unsigned long long b3) {
#pragma unroll
    for (int s = 0; s < kDigits; ++s) {
        b[s][0] = digit_pair(b0, b1, s);
        b[s][1] = digit_pair(b2, b3, s);
    }
}

// acc[g] += the digit products of weight g of a lane's part of A (16 x 16; x[4 u + v]: row g + 8 u,
// columns t, t + 1, t + 8, t + 9) and of B.
__device__ __forceinline__ void split_products(float (&acc)[kGroups][4], const unsigned long long (&x)[8],
                                               const uint32_t (&b)[kDigits][2]) {
#pragma unroll
    for (int s = 0; s < kDigits; ++s) {
        const uint32_t a[4] = {digit_pair(x[0], x[1], s), digit_pair(x[4], x[5], s), digit_pair(x[2], x[3], s),
                               digit_pair(x[6], x[7], s)};
#pragma unroll
        for (int q = 0; q < kDigits && s + q < kGroups; ++q) mma_f16(acc[s + q], a, b[q]);
    }
}

// acc[g] += the digit products of weight g of A (16 x 16) and B (16 x 8), one warp. A(r, k) for
// r in {g, g + 8}, B(k): this lane's column; both return digits_of a number (0x8080...: zero).
template <typename FA, typename FB>
__device__ __forceinline__ void split_mma(float (&acc)[kGroups][4], int lane, FA A, FB B) {
    const int g = lane >> 2, t = (lane & 3) * 2;
    uint32_t b[kDigits][2];
    digit_frags(b, B(t), B(t + 1), B(t + 8), B(t + 9));
    unsigned long long x[8];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int r = g + 8 * u;
        x[4 * u] = A(r, t);
        x[4 * u + 1] = A(r, t + 1);
        x[4 * u + 2] = A(r, t + 8);
        x[4 * u + 3] = A(r, t + 9);
    }
    __syncwarp();
    split_products(acc, x, b);
}

// hi + lo 2^-32 as a double, rounded to nearest (half an ulp + 2^-11), |hi| < 2^62: the bits put together by
// integer operations, of which the SM runs 32 for one of FP64. A tile's 128 values
// with two additions and a fused multiply-add in FP64 each instead: N = 40,962, n = 84 16.15 ms a step
// against 15.68; n = 55 at N = 12,347 2.11 against 2.07; batch of 24 problems 41.3 against 38.7.
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo) {
    hi += lo >> 32;
    uint32_t l = (uint32_t)lo;
    const bool neg = hi < 0;
    if (neg) {
        l = 0u - l;
        hi = ~hi + (l == 0);
    }
    const bool small = hi == 0;  // the leading bit is in l
    const unsigned long long L = (unsigned long long)l << 32, h = small ? L : (unsigned long long)hi;
    const int z = __clzll((long long)h) & 63;
    const unsigned long long m = (h << z) | (small || z == 0 ? 0 : L >> (64 - z));
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1);  // 53 bits, or 2^53
    const unsigned long long bits = ((unsigned long long)(63 - z - (small ? 64 : 0) + 1022) << 52) + r;
    return __longlong_as_double((long long)(h == 0 ? 0 : bits | ((unsigned long long)neg << 63)));
}

// The sum of the weighted accumulators of one entry, in units of 2^(EA + EB - 2 * 1023 - 34): the
// exact integer hi 2^32 + lo rounded once (times 2^-32), the last group rounded into lo.
__device__ __forceinline__ double split_value(const float (&acc)[kGroups][4], int u) {
    long long hi = 0, lo = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        hi = hi * 256 + __float2int_rn(acc[g][u]);
        lo = lo * 256 + __float2int_rn(acc[g + 4][u]);
    }
    lo += (__float2int_rn(acc[8][u]) + 128) >> 8;
    return fixed_to_double(hi, lo);
}

// 2^(EA + EB - 2 * 1023 - 34) and whether it and its neighbourhood are normal doubles.
__device__ __forceinline__ bool split_scale_ok(int EA, int EB) {
    const int e = EA + EB - 1023 - 34;
    return e > 200 && e < 1846;
}
__device__ __forceinline__ double split_scale(int EA, int EB) {
    return __longlong_as_double((long long)(EA + EB - 1023 - 34) << 52);
}

}  // namespace rbfsl
