// FP64 building blocks of the plain FP64 path, with as few instructions on the FP64 pipe as they can
// do with.
//
// GB300 runs 2 FP64 lane operations per clock and SM against 128 FP32 or integer ones: one FP64
// instruction of a warp takes the pipe as long as 64 other instructions take to issue.  So everything
// that need not be rounded to 53 bits runs elsewhere: exponents, table indices, conversions and
// comparisons on the integer pipe (from the bits of the doubles), reciprocal seeds and the last terms of
// the series, below 2^-27 of the result, in FP32 pairs.  Against the library's exp10, exp2, log and
// division a state-bin of the likelihood takes 59 FP64 instructions instead of 225.
#pragma once

#include <cmath>
#include <cstring>

#include "lisa_math.cuh"

namespace lisa {
namespace m64 {

// Host: the table of exp10_fast, kExpTabDoubles doubles: 2^(j / kExpTab) rounded to FP64, then the relative
// errors of these roundings (what is missing, over the entry) as floats.
inline void fill_exp_table(double* T) {
    float* c = reinterpret_cast<float*>(T + kExpTab);
    for (int j = 0; j < kExpTab; ++j) {
        const long double v = std::exp2((long double)j / kExpTab);
        T[j] = (double)v;
        const float e = (float)(v - (long double)T[j]) / (float)T[j];
        std::memcpy(c + j, &e, sizeof e);
    }
}

__device__ __forceinline__ unsigned hi32(double v) { return (unsigned)__double2hiint(v); }
__device__ __forceinline__ unsigned lo32(double v) { return (unsigned)__double2loint(v); }

// A double truncated to FP32 by its bits (magnitudes below 2^-126 become 0; not for |v| >= 2^128).
__device__ __forceinline__ float to_float(double v) {
    const unsigned h = hi32(v), a = h & 0x7fffffffu;
    const unsigned m = (__funnelshift_l(lo32(v), h, 3) - (896u << 23)) & 0x7fffffffu;
    return __uint_as_float(a >= (897u << 20) ? (m | (h & 0x80000000u)) : 0u);
}
// A normal FP32 number as a double by its bits (0 becomes +-2^-127, which every use here drowns in a
// larger term).
__device__ __forceinline__ double to_double(float f) {
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}
// The order of doubles on integers (NaN excluded; -0 lies below +0): comparisons without the FP64 pipe.  For
// bins against knots: no bin's x is -0 (log10 of 1 Hz is +0), so a knot at a zero of either sign is at or below
// the bin at 1 Hz, as it compares.
__device__ __forceinline__ long long order_key(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
// The same with one key for both zeros, for knots against knots and band edges: a knot at -0 does not lie
// inside a band that ends at +0.  (In the bins' searches too, the further instructions cost the model PSD 0.81 ->
// 0.99 ms, the FP64 likelihood 2 %.)
__device__ __forceinline__ long long position_key(double v) {
    const long long k = order_key(v);
    return k == -1 ? 0 : k;   // (-1 is -0's key alone)
}
// Biased exponent of a double (0: zero or subnormal, 2047: infinite or NaN).
__device__ __forceinline__ int exponent(double v) { return (int)((hi32(v) >> 20) & 0x7ffu); }

__device__ __forceinline__ bool negative(double v) { return (int)hi32(v) < 0; }   // (-0 included)
// Whether |v| lies in [2^-900, 2^900) (false for NaN).
__device__ __forceinline__ bool normal_range(double v) { return (unsigned)(exponent(v) - 123) < 1800u; }
// Whether |v| lies in [2^-480, 2^480): the squares of v and 1 / v are finite.
__device__ __forceinline__ bool square_range(double v) { return (unsigned)(exponent(v) - 543) < 960u; }
// |v| < 100 (false for NaN): the range of exp10_fast.
__device__ __forceinline__ bool small_exponent(double v) { return (hi32(v) & 0x7fffffffu) < 0x40590000u; }

// 10^v for |v| < 100 from the table T of 2^(j / kExpTab) (the table-driven scheme of Tang, ACM TOMS 15,
// 1989): 4 FP64 instructions.  v = k log10(2) / 4096 + r with k chosen in FP32 (|r| <= 0.7 of a step);
// 10^r = 1 + r ln10 + q with q = sum_(n = 2..4) (r ln10)^n / n! <= 2^-27, formed in float-float.  What is
// missing besides is below 2^-50 and collected in one FP32 number: q's low part, k times what log10(2) / 4096
// rounded off, and the table entry's rounding error.  Added to q and r ln10 in FP64, so one rounding is left:
// error at most 0.51 units of the last place, rms 0.29 (the library's exp10 takes about 40 instructions).  With q
// rounded to FP32 and the entries as they are, it was up to 1.7 units, rms 0.41, and the model PSD's error
// against 64 bits half a percent above that of the library's functions.  The tables (48 KB) are read through
// L1, which the kernels that use them leave free (8,192 entries, 96 KB, cost the dense covariance's careful bins
// 2-4 %, entry and error in one 16-byte load small FP64 calls 10 %).
__device__ __forceinline__ double exp10_fast(double v, const double* __restrict__ T) {
    constexpr double C_hi = 0x1.34413509f79ffp-14;    // log10(2) / 4096, rounded to FP64
    constexpr float C_lo = 0x1.9dc1da994fd21p-71 * 2.302585092994045684;   // what that is too large, times ln10
    static_assert(kExpTab == 4096, "constants");
    const float tf = fmaf(to_float(v), 13606.6175f, 12582912.f);   // 4096 / log10(2): k in the low bits
    const int k = __float_as_int(tf) - 0x4b400000, j = k & (kExpTab - 1);
    const double t = __ldg(T + j);
    const float kf = tf - 12582912.f, c = __ldg(reinterpret_cast<const float*>(T + kExpTab) + j);
    const double r = fma(to_double(kf), -C_hi, v);
    // r = rf + rl: its truncation to FP32 and the 29 bits below
    const float rf = to_float(r);
    const unsigned hr = hi32(r), er = (hr >> 20) & 0x7ffu;
    const float sc = er >= 960u ? __uint_as_float((hr & 0x80000000u) | ((er - 948u) << 23)) : 0.f;   // 2^(e - 52)
    const float rl = (float)(lo32(r) & 0x1fffffffu) * sc;
    constexpr float K2 = 2.65094906f, K2l = 5.39269431e-08f, K3 = 2.03467859f, K4 = 1.17125515f;   // ln10^n / n!
    const float h = rf * rf;
    const float l = fmaf(2.f * rf, rl, fmaf(rf, rf, -h));
    const float q0 = K2 * h;
    const dm::ff q = dm::fast_two_sum(q0, fmaf(K2, h, -q0) + fmaf(K2, l, fmaf(rf, fmaf(rf, K4, K3), K2l) * h));
    const double p = fma(r, kLn10, to_double(q.hi) + to_double(fmaf(kf, C_lo, q.lo + c)));
    const double e = fma(t, p, t);
    return __hiloint2double((int)(hi32(e) + (unsigned)((k >> 12) << 20)), (int)lo32(e));
}

// 10^v, any value (A = 10^log10A, and a spline's factor in the wide forms).
__device__ __forceinline__ double amplitude(double v, const double* __restrict__ T) {
    return small_exponent(v) ? exp10_fast(v, T) : exp10(v);
}
// 10^lA 10^p 2^y (the background's factor), any values.
__device__ __forceinline__ double background_wide(double lA, double p, double y, const double* __restrict__ T) {
    constexpr double kLog10_2 = 0.301029995663981195213739;
    const double v = fma(y, kLog10_2, p), A = amplitude(lA, T);
    return small_exponent(v) && normal_range(A) ? A * exp10_fast(v, T) : exp10(lA + p) * exp2(y);
}

// 1 / d to 2^-21 for a normal positive d of exponent within +-900, as a double: an FP32 reciprocal of d's
// mantissa, in (1/2, 1], times 2^-(exponent of d).
__device__ __forceinline__ double reciprocal_seed(double d) {
    const unsigned h = hi32(d);
    const float m = __uint_as_float(0x3f800000u | ((h & 0xfffffu) << 3) | (lo32(d) >> 29));
    const unsigned b = __float_as_uint(dm::rcp_approx(m));
    return __hiloint2double((int)((b >> 3) + (896u << 20) + (1023u << 20) - (h & 0x7ff00000u)), (int)(b << 29));
}
// 1 / d by one cubic step: 3 FP64 instructions, rounded once (error up to half a unit of the last place
// and 2^-64 of the result).
__device__ __forceinline__ double reciprocal(double d) {
    const double r = reciprocal_seed(d), e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
// 1 / d for any d >= 0 (NaN included).
__device__ __forceinline__ double reciprocal_wide(double d) { return normal_range(d) ? reciprocal(d) : 1.0 / d; }
// n / d: a reciprocal to 2^-42, the quotient by it and one correction by the remainder: 5 FP64
// instructions, rounded once.  (n r (1 + e + e^2), 4 instructions, rounds twice: up to 1 unit, 1.2 with a
// seed one unit off.)
__device__ __forceinline__ double divide(double n, double d) {
    const double r0 = reciprocal_seed(d);
    const double r = fma(r0, fma(-d, r0, 1.0), r0);
    const double w = n * r;
    return fma(fma(-d, w, n), r, w);
}

// Running product of normal positive doubles as mantissa and exponent: one FP64 instruction a factor.
// Its logarithm is taken once for many factors (the mantissa grows by less than 2 a factor).
struct LogProduct {
    double m;
    int e;
    __device__ __forceinline__ void reset() {
        m = 1.0;
        e = 0;
    }
    __device__ __forceinline__ void mul(double v) {
        const unsigned h = hi32(v);
        e += (int)(h >> 20) - 1023;
        m *= __hiloint2double((int)((h & 0xfffffu) | 0x3ff00000u), (int)lo32(v));
    }
    __device__ __forceinline__ double log_value() const { return fma((double)e, kLn2, log(m)); }
};

// The calling lane's part of unit u of a plain FP64 likelihood kernel: its state s (sw lanes side by side
// hold different states), and its bins [b0, b0 + nb) of the unit's slot of b64.
struct Unit64 {
    int slot, s, sw, nb;
    int64_t b0;
};

// The calling warp's unit u: its dataset (the last one whose first unit is <= u; empty ones share their
// successor's) and its lanes' parts.  A dataset of up to 16 states splits a unit's bins over 32 / sw rows,
// sw the next power of two of its states: with one lane per state whatever their number, 4 states left 28
// of a warp's lanes idle, and the pipe takes as long for them (figures at loglike_fp64_kernel).
__device__ __forceinline__ const DatasetDev& unit_of(const DatasetDev* __restrict__ ds, int n_ds, int64_t u, int b64,
                                                     const int32_t* __restrict__ sstat, Unit64& w) {
    int lo = 0, hi = n_ds - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (ds[mid].ubase64 <= u) lo = mid; else hi = mid - 1;
    }
    const DatasetDev& D = ds[lo];
    const int groups = (D.ns + 31) >> 5;
    const int lane = (int)(threadIdx.x & 31);
    w.sw = D.ns > 16 ? 32 : 1 << (32 - __clz(D.ns - 1));   // (__clz(0) = 32)
    w.slot = (int)((u - D.ubase64) / groups);
    w.s = D.s0 + 32 * (int)((u - D.ubase64) % groups) + (lane & (w.sw - 1));
    const int64_t first = (int64_t)w.slot * b64;
    const int n = (int)min((int64_t)b64, D.npad - first);
    const int rows = 32 / w.sw, r = lane / w.sw;
    const int a = r * n / rows;
    w.b0 = D.bin0 + first + a;
    w.nb = w.s < D.s0 + D.ns && sstat[w.s] == 0 ? (r + 1) * n / rows - a : 0;
    return D;
}

// The unit's sum of a state over its rows (in a fixed order, by all lanes), stored by the first row.
__device__ __forceinline__ void store_unit(const DatasetDev& D, const Unit64& w, const int32_t* __restrict__ sstat,
                                           double acc, double* __restrict__ partial) {
    for (int o = 16; o >= w.sw; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((int)(threadIdx.x & 31) < w.sw && w.s < D.s0 + D.ns && sstat[w.s] == 0)
        partial[D.pbase64 + (int64_t)(w.s - D.s0) * D.n64 + LISA_IDX(w.slot, D.n64)] = acc;
}

}  // namespace m64
}  // namespace lisa
