// The FP64 building blocks of csrc/lisa_math64.cuh on arrays, for tests/test_gpu_math64.py.
#include "lisa_math64.cuh"

namespace {
__global__ void probe_kernel(int what, const double* a, const double* b, const double* tab, double* out, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (what == 0) out[i] = lisa::m64::exp10_fast(a[i], tab);
    if (what == 1) out[i] = lisa::m64::divide(a[i], b[i]);
    if (what == 2) out[i] = lisa::m64::reciprocal(a[i]);
}
}  // namespace

extern "C" int probe_table_doubles() { return lisa::kExpTabDoubles; }
extern "C" void probe_table(double* host) { lisa::m64::fill_exp_table(host); }
extern "C" int probe_run(int what, const double* a, const double* b, const double* tab, double* out, int64_t n) {
    probe_kernel<<<(unsigned)((n + 255) / 256), 256>>>(what, a, b, tab, out, n);
    return (int)cudaDeviceSynchronize();
}
