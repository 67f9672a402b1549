// The integer-pipe FP64 arithmetic of csrc/lisa_soft64.cuh compiled for the host, for
// tests/test_soft64_host.py.
#include "lisa_soft64.cuh"

using namespace lisa::soft64;

// bits of sqrt(v / 2); ok[i] = 0 where the form leaves it to the hardware's instruction
extern "C" void host_sqrt_half(const uint64_t* v, uint64_t* out, uint8_t* ok, int64_t n) {
    for (int64_t i = 0; i < n; ++i) ok[i] = sqrt_half(v[i], out[i]);
}
// bits of a x for normal positive a
extern "C" void host_mul(const uint64_t* a, const uint64_t* x, uint64_t* out, uint8_t* ok, int64_t n) {
    for (int64_t i = 0; i < n; ++i) ok[i] = mul(exp_of(a[i]), ((a[i] & kMant) | kOne) << 11, x[i], out[i]);
}
// the sum of squares of finite v in the order given: its 96-bit value (top, acc) and exponent E
extern "C" int host_square_sum(const uint64_t* v, int64_t n, uint32_t* top, uint64_t* acc) {
    SquareSum q;
    q.reset();
    for (int64_t i = 0; i < n; ++i) {
        if (exp_of(v[i]) > q.E) q.raise(exp_of(v[i]));
        q.add(v[i]);
    }
    *top = q.top;
    *acc = q.acc;
    return q.E;
}
