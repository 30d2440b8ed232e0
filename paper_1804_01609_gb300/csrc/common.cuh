// Shared device/host helpers of the CUDA library (not shared with any CPU reference code).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <string>

#include "rbfsl.h"

namespace rbfsl {

// Thread-local message of the last failure of a stateless call.
void set_error(const std::string &msg);
const char *get_error();

#define RBFSL_CUDA_TRY(expr)                                                               \
    do {                                                                                   \
        cudaError_t _e = (expr);                                                           \
        if (_e != cudaSuccess) {                                                           \
            cudaGetLastError();                                                            \
            ::rbfsl::set_error(std::string(#expr) + ": " + cudaGetErrorString(_e));        \
            return RBFSL_ECUDA;                                                            \
        }                                                                                  \
    } while (0)

#define RBFSL_CHECK_ARG(cond, msg)                                                         \
    do {                                                                                   \
        if (!(cond)) {                                                                     \
            ::rbfsl::set_error(msg);                                                       \
            return RBFSL_EINVAL;                                                           \
        }                                                                                  \
    } while (0)

inline int launch_status(const char *what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error(std::string(what) + ": " + cudaGetErrorString(e));
        return RBFSL_ECUDA;
    }
    return RBFSL_OK;
}

constexpr int kWarp = 32;

// ---------------------------------------------------------------------------------------
// Real orthonormal spherical harmonics of degree <= ell as polynomials of (x, y, z) on S^2
// (the augmentation basis {p_i} of Sec. 2.2). Index l*l + l + m, m = -l..l.
// With z = cos(theta), x + iy = sin(theta) e^{i phi}, Q_l^m(z) = P_l^m(z) / sin^m(theta):
//   Q_m^m = (2m-1)!!, Q_{m+1}^m = (2m+1) z Q_m^m,
//   Q_l^m = a_lm z Q_{l-1}^m - b_lm Q_{l-2}^m, a_lm = (2l-1)/(l-m), b_lm = (l+m-1)/(l-m),
//   Y_l^0 = K_l0 Q_l^0, Y_l^{+m} = K_lm Q_l^m Re(x+iy)^m, Y_l^{-m} = K_lm Q_l^m Im(x+iy)^m,
//   K_lm = sqrt((2 - delta_m0) (2l+1)/(4 pi) (l-m)!/(l+m)!).
// The coefficient tables live in constant memory, filled once per device by sh_tables_init.
constexpr int kMaxL = RBFSL_MAX_SH_DEGREE;
constexpr int kMaxM = (kMaxL + 1) * (kMaxL + 1);

struct ShTables {
    double K[kMaxM];   // indexed l*l + l + m, m >= 0
    double a[kMaxM];
    double b[kMaxM];
    double qmm[kMaxL + 1];
};

int sh_tables_init();  // host: upload the tables to the current device (idempotent)

extern __constant__ ShTables c_sh;

// Evaluate all (ell+1)^2 harmonics at (x, y, z); out[c * stride] for c = l*l + l + m.
template <typename Out>
__device__ __forceinline__ void sh_eval(int ell, double x, double y, double z, Out out) {
    double cm = 1.0, sm = 0.0;
    for (int m = 0; m <= ell; ++m) {
        if (m > 0) {
            const double c2 = cm * x - sm * y;
            const double s2 = cm * y + sm * x;
            cm = c2;
            sm = s2;
        }
        double q2 = 0.0, q1 = 0.0;
        for (int l = m; l <= ell; ++l) {
            const int id = l * l + l + m;
            double q;
            if (l == m) q = c_sh.qmm[m];
            else q = c_sh.a[id] * z * q1 - c_sh.b[id] * q2;
            const double kq = c_sh.K[id] * q;
            if (m == 0) {
                out(id, kq);
            } else {
                out(id, kq * cm);
                out(l * l + l - m, kq * sm);
            }
            q2 = q1;
            q1 = q;
        }
    }
}

// sh_eval spread over a warp, one lane per order m (lanes 0..ell; the others return at once):
// lane m forms (x + iy)^m by sh_eval's recurrence and then the degrees l = m..ell, so every
// value comes from the same operations as in sh_eval while the serial chain is one order long.
template <typename Out>
__device__ __forceinline__ void sh_eval_lanes(int ell, double x, double y, double z, int lane, Out out) {
    if (lane > ell) return;
    const int m = lane;
    double cm = 1.0, sm = 0.0;
    for (int mm = 1; mm <= m; ++mm) {
        const double c2 = cm * x - sm * y;
        const double s2 = cm * y + sm * x;
        cm = c2;
        sm = s2;
    }
    double q2 = 0.0, q1 = 0.0;
    for (int l = m; l <= ell; ++l) {
        const int id = l * l + l + m;
        double q;
        if (l == m) q = c_sh.qmm[m];
        else q = c_sh.a[id] * z * q1 - c_sh.b[id] * q2;
        const double kq = c_sh.K[id] * q;
        if (m == 0) {
            out(id, kq);
        } else {
            out(id, kq * cm);
            out(l * l + l - m, kq * sm);
        }
        q2 = q1;
        q1 = q;
    }
}

// Polyharmonic spline r^p (p odd) from the squared distance: r * (r^2)^((p-1)/2).
__device__ __forceinline__ double phs_from_d2(double d2, int half) {
    double v = sqrt(d2);
    for (int i = 0; i < half; ++i) v *= d2;
    return v;
}

// Squared distance with every operation rounded separately (the k-NN key).
__device__ __forceinline__ double sqdist_rn(double ax, double ay, double az, double bx,
                                            double by, double bz) {
    const double dx = __dsub_rn(ax, bx), dy = __dsub_rn(ay, by), dz = __dsub_rn(az, bz);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// ---------------------------------------------------------------------------------------
// Mixed-precision storage of fields and weights: each value is an unevaluated pair of FP32
// numbers (hi, lo), value = hi + lo with |lo| <= ulp(hi) / 2, stored interleaved (8 bytes per
// value). The gather-dot sum is formed in pair arithmetic with FP32 operations only: exact
// products of the high parts (FMA error term), the cross terms, and Knuth's two-sum into the
// accumulator, so a step adds ~n 2^-48 relative rounding instead of the ~2^-24 of plain FP32.

// v as a pair: hi = v to nearest, lo = v - hi to nearest, by integer operations on v's bits and one
// conversion of a 32-bit integer, because conversions between FP64 and FP32 run at the FP64 rate.
// v = sign (1 + f) 2^e; 2^e is applied in two factors, which covers subnormal and zero results (a lo below the
// normal range is rounded twice). kStored, for values that are kept or returned: hi is what a conversion gives (ties to
// even), NaN gives (NaN, NaN), an infinity (inf, NaN), a v that rounds beyond FP32's range (inf, -inf), with v's sign.
// Without, for a factor on its way into a sum: ties go away from zero, and lo is NaN for all of these, hi an infinity
// (the four operations less are 3% of the blend of partition-of-unity patches, 625 against 605 us a step at
// N = 40,962, n = 84, T = 16).
template <bool kStored>
__device__ __forceinline__ float2 pair_split(double v) {
    const long long b = __double_as_longlong(v);
    const unsigned long long a = (unsigned long long)b & 0x7fffffffffffffffULL;
    const int field = (int)(a >> 52), e = min(max(field - 1023, -252), 128);
    const int f = (int)((a & 0xfffffffffffffULL) >> 28);          // the fraction's leading 24 bits
    const int up = kStored ? f & ((f >> 1) | ((a & 0xfffffffULL) != 0)) & 1 : f & 1;
    const int top = (f >> 1) + up;                                // 23 bits, rounded
    const int rest = (int)(a & 0x1fffffffULL) - (up << 29);       // the others, units of 2^(e - 52)
    const int sign = (int)(b >> 32) & (int)0x80000000;
    const float s0 = __int_as_float(((e >> 1) + 127) << 23 | sign), s1 = __int_as_float((e - (e >> 1) + 127) << 23);
    float hi = __int_as_float(0x3f800000 + top) * s0 * s1, end = hi - hi;
    if (kStored) {
        if (a > 0x7ff0000000000000ULL) hi = end = __int_as_float(0x7fffffff);
        else if (field < 0x7ff && fabsf(hi) == __int_as_float(0x7f800000)) end = -hi;
    }
    return make_float2(hi, ((float)rest * 0x1p-52f) * s0 * s1 + end);
}
__device__ __forceinline__ float2 pair_from(double v) { return pair_split<true>(v); }

// (sh, sl) += w * q for pairs w and q; w.lo * q.lo (below 2^-48 |w q|) is dropped.
__device__ __forceinline__ void pair_fma(float2 w, float2 q, float &sh, float &sl) {
    const float p = w.x * q.x;
    float pe = fmaf(w.x, q.x, -p);
    pe = fmaf(w.x, q.y, pe);
    pe = fmaf(w.y, q.x, pe);
    const float s = sh + p;
    const float bp = s - sh;
    const float e = (sh - (s - bp)) + (p - bp);
    sl = sl + (e + pe);
    sh = s;
}

// The accumulator as a normalised pair (fast two-sum).
__device__ __forceinline__ float2 pair_norm(float sh, float sl) {
    const float hi = sh + sl;
    return make_float2(hi, sl - (hi - sh));
}

// Weight and field element conversions from FP64 results.
template <typename WT>
__device__ __forceinline__ WT wcast(double v);
template <>
__device__ __forceinline__ double wcast<double>(double v) { return v; }
template <>
__device__ __forceinline__ float wcast<float>(double v) { return (float)v; }
template <>
__device__ __forceinline__ float2 wcast<float2>(double v) { return pair_from(v); }

}  // namespace rbfsl
