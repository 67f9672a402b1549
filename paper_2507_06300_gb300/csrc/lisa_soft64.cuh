// FP64 arithmetic on the integer pipes, for streaming kernels whose few FP64 operations per sample would
// make GB300's FP64 pipe (2 lane operations per clock and SM, against 64 to 128 integer ones) and
// not HBM their bound.  Results are those of IEEE round-to-nearest-even, bit for bit; arguments or
// results outside the normal range are reported to the caller, who takes the hardware's instruction.
#pragma once

#include <cstdint>

namespace lisa {
namespace soft64 {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float rsqrt_seed(float v) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
    return y;
}
__device__ __forceinline__ float bits_float(uint32_t b) { return __uint_as_float(b); }
__device__ __forceinline__ uint32_t float_bits(float f) { return __float_as_uint(f); }
#else
inline float rsqrt_seed(float v) { return 1.0f / __builtin_sqrtf(v); }
inline float bits_float(uint32_t b) { float f; __builtin_memcpy(&f, &b, 4); return f; }
inline uint32_t float_bits(float f) { uint32_t b; __builtin_memcpy(&b, &f, 4); return b; }
#endif

constexpr uint64_t kMant = (1ull << 52) - 1, kOne = 1ull << 52;

#ifdef __CUDACC__
#define LISA_HD __host__ __device__ __forceinline__
#else
#define LISA_HD inline
#endif

// Biased exponent of a double's bits; normal: neither 0 / subnormal nor infinite / NaN.
LISA_HD int exp_of(uint64_t b) { return (int)((b >> 52) & 0x7ff); }
LISA_HD bool is_normal(uint64_t b) { return (unsigned)(exp_of(b) - 1) < 2046u; }

// Bits of sqrt(v / 2) for a normal positive v; false where the rounding is too close to call (about one
// argument in 600) or v / 2 is not normal and positive.
// With m in [1, 4) the scaled argument: an FP32 reciprocal square root y (relative error e ~ 2^-21), then
// twice s += (m - s^2) y / 2 in fixed point, m - s^2 exact: errors 2^-42 and, in the last step's
// correction p (52 + 50 fractional bits), |p| 2^-21 and the truncations, 2^25, which decide whether the
// fraction is safely on one side of one half.
LISA_HD bool sqrt_half(uint64_t v, uint64_t& out) {
    const int E = exp_of(v) - 1024;            // exponent of v / 2
    const unsigned odd = (unsigned)E & 1u;
    const uint64_t F = (v & kMant) | kOne;
    const float mf = bits_float(((127u + odd) << 23) | ((uint32_t)(F >> 29) & 0x7fffffu));
    float y = rsqrt_seed(mf);
    y = y < 0.99999994f ? y : 0.99999994f;
    float g = mf * y;
    g = g > 1.0f ? g : 1.0f;
    g = g < 1.99999988f ? g : 1.99999988f;
    const uint32_t Y = (float_bits(y) & 0x7fffffu) | 0x800000u;           // y 2^24 (y in [1/2, 1))
    const uint32_t G0 = ((float_bits(g) & 0x7fffffu) | 0x800000u) << 8;   // 31 fractional bits
    const int64_t d0 = (int64_t)((F << (10 + odd)) - (uint64_t)G0 * G0);
    const int64_t p0 = (int64_t)(int32_t)(d0 >> 14) * (int32_t)Y;
    const uint64_t G1 = (((uint64_t)G0 << 31) + (uint64_t)(p0 >> 11)) >> 16;   // 46 fractional bits
    const int64_t d1 = (int64_t)((F << (40 + odd)) - G1 * G1);
    const int64_t p = (d1 >> 15) * (int64_t)Y;                            // 56 more fractional bits
    const int64_t frac = p & ((1ll << 50) - 1);
    const uint64_t S = (G1 << 6) + (uint64_t)(p >> 50) + (frac >= (1ll << 49) ? 1u : 0u);
    const int64_t off = frac - (1ll << 49), ap = p < 0 ? -p : p;
    out = ((uint64_t)((E >> 1) + 1023) << 52) + (S - kOne);
    return (off < 0 ? -off : off) > (ap >> 20) + (1ll << 25) && (unsigned)(exp_of(v) - 2) < 2045u && !(v >> 63);
}

// Bits of a x from a's parts (ea: biased exponent, A: its 53-bit significand times 2^11); false where x or
// the product is not normal.
LISA_HD bool mul(int ea, uint64_t A, uint64_t x, uint64_t& out) {
    const uint64_t X = (x & kMant) | kOne;
    const unsigned __int128 P = (unsigned __int128)A * X;
    uint64_t hi = (uint64_t)(P >> 64), lo = (uint64_t)P;    // [2^51, 2^53) and the bits below
    int e = ea + exp_of(x) - 1022;
    if (!(hi >> 52)) {
        hi = (hi << 1) | (lo >> 63);
        lo <<= 1;
        --e;
    }
    const uint64_t inc = (lo >> 63) & (((lo << 1) != 0 ? 1u : 0u) | (hi & 1u));
    out = (x & (1ull << 63)) | (((uint64_t)(uint32_t)e << 52) + (hi - kOne) + inc);
    return is_normal(x) && (unsigned)(e - 1) < 2045u;
}

// Sum of squares in fixed point: (top, acc), 96 bits, times 2^(2 (E - 1023) - 62), E the largest biased
// exponent met.  Each square loses less than two units of its own last bit to its truncation and the sum
// less than one at each shift, so n squares come out at most 3 n units of 2^-62 of the largest one's binade
// too small, never too large.  Additions in FP64 may lose more: 2e5 squares of 2^-61 beside one of 1, 3.6e-14
// here, 7.9e-14 there.
struct SquareSum {
    uint64_t acc;
    uint32_t top;
    int E;
    LISA_HD void reset() {
        acc = 0;
        top = 0;
        E = 0;
    }
    // Makes room for values of biased exponent e.
    LISA_HD void raise(int e) {
        const int sh = 2 * (e - E);
        E = e;
        if (sh >= 96) {
            acc = 0;
            top = 0;
        } else if (sh >= 64) {
            acc = (uint64_t)top >> (sh - 64);
            top = 0;
        } else if (sh > 0) {
            const uint64_t in = sh > 32 ? (uint64_t)top << (64 - sh) : ((uint64_t)top << 32) << (32 - sh);
            acc = (acc >> sh) | in;
            top = sh >= 32 ? 0u : top >> sh;
        }
    }
    // Adds the square of v, finite and of exponent at most E (a subnormal adds nothing: its square is
    // 0 in FP64).
    LISA_HD void add(uint64_t v) {
        const int e = exp_of(v);
        const uint64_t m = (v << 11) | (1ull << 63);
        const uint32_t a1 = (uint32_t)(m >> 32), a0 = (uint32_t)m;
        const uint64_t sq = (uint64_t)a1 * a1 + (((uint64_t)a1 * a0) >> 31);   // m^2 / 2^64 within 2
        const int sh = 2 * (E - e);
        const uint64_t q = (e == 0 || sh > 63) ? 0u : sq >> sh;
        acc += q;
        top += acc < q ? 1u : 0u;
    }
};

}  // namespace soft64
}  // namespace lisa
