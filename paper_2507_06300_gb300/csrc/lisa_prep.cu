// Data preparation (Sec. III.C): synthetic frequency-domain data and the averaged periodogram,
// the inputs of lisa_data_create.  Both are streaming kernels; HBM bounds them only because their FP64
// arithmetic runs on the integer pipes (lisa_soft64.cuh).
#include <cmath>

#include "lisa_internal.cuh"
#include "lisa_soft64.cuh"

namespace lisa {
namespace {

// a v by the integer pipes, or by the FP64 instruction where a factor or the product is not normal.
__device__ __forceinline__ double times(double a, int ea, uint64_t A, bool a_ok, double v) {
    uint64_t r;
    const bool ok = soft64::mul(ea, A, (uint64_t)__double_as_longlong(v), r);
    if (ok && a_ok) return __longlong_as_double((long long)r);
    return a * v;
}

// d = sqrt(S / 2) (z0 + i z1), grid-stride over (channel, sample), 16-byte loads and stores.  The FP64
// pipe took 11 instructions a sample for the square root and the products (2.1 TB/s); about 150
// integer instructions run on pipes 32 to 64 times as wide.  25.2 M samples: 522 us -> 232 us (4.3 TB/s).
__global__ void __launch_bounds__(256) fd_synth_kernel(const double* __restrict__ S, const double2* __restrict__ z,
                                                       int64_t n, double2* __restrict__ d) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const double s = __ldg(S + i);
        const double2 v = __ldg(z + i);
        uint64_t ab;
        double a;
        if (soft64::sqrt_half((uint64_t)__double_as_longlong(s), ab)) {
            a = __longlong_as_double((long long)ab);
        } else {
            a = sqrt(0.5 * s);
            ab = (uint64_t)__double_as_longlong(a);
        }
        const bool a_ok = soft64::is_normal(ab) && !(ab >> 63);
        const uint64_t A = ((ab & soft64::kMant) | soft64::kOne) << 11;
        const int ea = soft64::exp_of(ab);
        d[i] = make_double2(times(a, ea, A, a_ok, v.x), times(a, ea, A, a_ok, v.y));
    }
}

// A lane's sum of squares in fixed point on the integer pipes.
struct LaneSum {
    double fp;   // of batches with an infinity or a NaN only
    soft64::SquareSum q;
    __device__ __forceinline__ void reset() {
        fp = 0.0;
        q.reset();
    }
    // Adds N samples (absent ones as zeros, which add nothing).
    template <int N>
    __device__ __forceinline__ void add(const double2* v) {
        uint64_t b[2 * N];
        int e = 0;
#pragma unroll
        for (int u = 0; u < N; ++u) {
            b[2 * u] = (uint64_t)__double_as_longlong(v[u].x);
            b[2 * u + 1] = (uint64_t)__double_as_longlong(v[u].y);
            e = max(e, max(soft64::exp_of(b[2 * u]), soft64::exp_of(b[2 * u + 1])));
        }
        if (e > q.E) {
            if (e == 2047) {   // an infinity or a NaN: the sum is one too
#pragma unroll
                for (int u = 0; u < N; ++u) fp = fma(v[u].x, v[u].x, fma(v[u].y, v[u].y, fp));
                return;
            }
            q.raise(e);
        }
#pragma unroll
        for (int u = 0; u < 2 * N; ++u) q.add(b[u]);
    }
    __device__ __forceinline__ double value() const {
        // the 96-bit sum rounded to FP64, scaled by 2^(2 (E - 1023) - 62) in two exact halves
        const double m = fma((double)q.top, 18446744073709551616.0, (double)q.acc);
        const int k = 2 * (q.E - 1023) - 62, k1 = k >> 1, k2 = k - k1;
        const double s1 = __longlong_as_double((long long)(k1 + 1023) << 52);
        const double s2 = __longlong_as_double((long long)(k2 + 1023) << 52);
        if (q.E == 0) return fp;
        // (beyond 2^+-800 the halves or the result may leave the normal range)
        return ((unsigned)(q.E - 223) < 1600u ? m * s1 * s2 : scalbn(m, k)) + fp;
    }
};

constexpr int kFixedMin = 12;           // samples from which a bin's sums run in fixed point
constexpr int kFixedBatch = 4;          // samples that a lane adds at once there
constexpr int kSerialThreadsPerSm = 512, kSerialWidths = 4, kLanesPerSm = 2048;

// Averaged periodogram: a group of G lanes per bin (G divides 32), lanes striding over the bin's
// samples with 16-byte loads; the group's partial sums are combined by a butterfly of shuffles (a
// fixed order for a given G), and with G >= 4 its lanes share the epilogue: lane c divides channel
// c's sum, lane 3 writes the bin's centre and nu.  With FP64 multiply-adds the FP64 pipe bounded this
// kernel (two of them per complex sample, 81 us for 25.2 M samples at its rate against 60 us of HBM
// time); the lanes' sums of squares run on the integer pipes (about 40 instructions a sample; at most
// 3 n units of 2^-62 of the largest of a lane's n squares too small, less than FP64 additions may lose) where
// a bin has enough samples to pay for the conversion of the sums, which is the line at kFixedMin.
// 25.2 M samples in 64-sample bins: 125 us -> 92 us.
//
// That takes many bins side by side.  Where the loads of a few lanes are waited for, four of one channel in
// flight instead of four of every channel cost more than the FP64 pipe.  So a bin of up to `serial_max` samples
// takes the channels one after the other, in fixed point from kFixedMin samples on, and a wider one all
// channels together, in FP64; serial_max is kSerialWidths mean widths, or 0 when the bins of 4 or 8 lanes have
// fewer than kSerialThreadsPerSm lanes per SM.  Every bin serial (by its mean width in fixed point): 8,000 bins
// of 1,000 samples (64,000 lanes) 115 us, together 104; 12,000 of 300 (96,000) the same; 20,000 bins of 1 to
// 4,000 samples 402, 298 with this rule; 400 bins of 20,000 samples among 20,000 of one or two 1.89 ms, 1.32.
// With one lane per bin two channels go one after the other (200,000 bins of 4: 16.7 us, together 20.6; of 2 15.5,
// 15.7), three together (of 2 18.7, serial 21.3; of 6 27.7, 30.4; of 8 32.8, 32.3), but for bins of 7 samples
// and more that outnumber the resident lanes (a million of 8: 150, together 161).
template <int C, int G>
__global__ void __launch_bounds__(256)
    avg_periodogram_kernel(const double2* __restrict__ d, int64_t n_freq, double f0, double df,
                           const int64_t* __restrict__ off, int64_t n_bins, double* __restrict__ P,
                           double* __restrict__ f_out, double* __restrict__ nu_out, int n_ch, int serial_min,
                           int64_t serial_max) {
    const int lane = threadIdx.x & (G - 1);
    const int64_t g0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int64_t ng = ((int64_t)gridDim.x * blockDim.x) / G;
    const int64_t n_iter = (n_bins + ng - 1) / ng;   // the same trip count for every lane
    for (int64_t it = 0; it < n_iter; ++it) {
        const int64_t i = g0 + it * ng;
        const bool live = i < n_bins;
        int64_t b0 = 0, b1 = 0;
        if (live) {
            b0 = min(max(__ldg(off + i), (int64_t)0), n_freq);
            b1 = min(max(__ldg(off + i + 1), b0), n_freq);
        }
        const int64_t n = b1 - b0;
        double acc[C];
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = 0.0;
        if (n > serial_max || n < serial_min) {
#pragma unroll 4
            for (int64_t k = b0 + lane; k < b1; k += G) {
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    if (c < n_ch) {
                        const double2 v = __ldg(d + (int64_t)c * n_freq + k);
                        acc[c] = fma(v.x, v.x, fma(v.y, v.y, acc[c]));
                    }
                }
            }
        } else if (G == 1 || n < kFixedMin) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if (c >= n_ch) continue;
                const double2* dc = d + (int64_t)c * n_freq;
#pragma unroll 4
                for (int64_t k = b0 + lane; k < b1; k += G) {
                    const double2 v = __ldg(dc + k);
                    acc[c] = fma(v.x, v.x, fma(v.y, v.y, acc[c]));
                }
            }
        } else {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if (c >= n_ch) continue;
                LaneSum sum;
                sum.reset();
                const double2* dc = d + (int64_t)c * n_freq;
#pragma unroll 1
                for (int64_t k = b0 + lane; k < b1; k += kFixedBatch * G) {
                    double2 v[kFixedBatch];
#pragma unroll
                    for (int u = 0; u < kFixedBatch; ++u)
                        v[u] = k + u * G < b1 ? __ldg(dc + k + u * G) : make_double2(0.0, 0.0);
                    sum.add<kFixedBatch>(v);
                }
                acc[c] = sum.value();
            }
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o, G);
        if (G >= 4) {
            double v = acc[0];
#pragma unroll
            for (int c = 1; c < C; ++c)
                if (lane == c) v = acc[c];
            if (live && lane < n_ch) P[(int64_t)lane * n_bins + i] = n > 0 ? v / (double)n : NAN;
            if (live && lane == 3) {
                f_out[i] = f0 + df * (0.5 * (double)(b0 + b1 - 1));
                nu_out[i] = (double)n;
            }
        } else if (live && lane == 0) {
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (c < n_ch) P[(int64_t)c * n_bins + i] = n > 0 ? acc[c] / (double)n : NAN;
            f_out[i] = f0 + df * (0.5 * (double)(b0 + b1 - 1));
            nu_out[i] = (double)n;
        }
    }
}

template <int C, int G>
cudaError_t launch_avg(const double2* d, int64_t n_freq, double f0, double df, const int64_t* off, int64_t n_bins,
                       double* P, double* f, double* nu, int n_ch, cudaStream_t sm) {
    int dev = 0, n_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int threads = 256;
    const int64_t want = (n_bins * G + threads - 1) / threads;
    const int64_t cap = (int64_t)n_sm * 8;   // persistent: 8 blocks of 256 threads per SM
    const unsigned grid = (unsigned)(want < cap ? (want < 1 ? 1 : want) : cap);
    const bool two = G == 1 && n_ch < 3;
    const bool many = two || n_bins * G >= (int64_t)(G == 1 ? kLanesPerSm : kSerialThreadsPerSm) * n_sm;
    const int64_t serial_max = many ? (int64_t)(kSerialWidths * ((double)n_freq / (double)n_bins)) : 0;
    const int serial_min = G > 1 || two ? 0 : 7;
    avg_periodogram_kernel<C, G><<<grid, threads, 0, sm>>>(d, n_freq, f0, df, off, n_bins, P, f, nu, n_ch, serial_min,
                                                      serial_max);
    return cudaGetLastError();
}

}  // namespace
}  // namespace lisa

using namespace lisa;

extern "C" lisa_status lisa_fd_synthesize(const double* psd, const double* normal, int32_t n_channels, int64_t n_freq,
                                          double* d, lisa_stream_t stream) {
    lisa::NvtxRange nvtx_range("lisa_fd_synthesize");
    if (n_channels < 1 || n_freq < 0) return LISA_ERR_VALUE;
    if (n_freq == 0) return LISA_SUCCESS;
    if (!psd || !normal || !d) return LISA_ERR_NULL;
    if ((reinterpret_cast<uintptr_t>(normal) | reinterpret_cast<uintptr_t>(d)) & 15) return LISA_ERR_VALUE;
    const int64_t n = (int64_t)n_channels * n_freq;
    int dev = 0, n_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (n + 255) / 256, cap = (int64_t)n_sm * 8;
    fd_synth_kernel<<<(unsigned)(want < cap ? want : cap), 256, 0, (cudaStream_t)stream>>>(
        psd, reinterpret_cast<const double2*>(normal), n, reinterpret_cast<double2*>(d));
    return check_cuda(cudaGetLastError());
}

extern "C" lisa_status lisa_averaged_periodogram(const double* d, int32_t n_channels, int64_t n_freq, double f0,
                                                 double df, const int64_t* off, int64_t n_bins, double* P, double* f,
                                                 double* nu, lisa_stream_t stream) {
    lisa::NvtxRange nvtx_range("lisa_averaged_periodogram");
    if (n_channels < 1 || n_channels > 3 || n_freq < 0 || n_bins < 0 || !(df > 0.0) || !std::isfinite(f0))
        return LISA_ERR_VALUE;
    if (n_bins == 0) return LISA_SUCCESS;
    if (!d || !off || !P || !f || !nu) return LISA_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(d) & 15) return LISA_ERR_VALUE;
    const double2* dd = reinterpret_cast<const double2*>(d);
    cudaStream_t sm = (cudaStream_t)stream;
    // lanes per bin from the mean bin width: 8 lanes for bins of hundreds of samples, 4 for tens,
    // one thread for bins of a few samples
    const double width = (double)n_freq / (double)n_bins;
    cudaError_t e;
    if (width >= 256.0)
        e = launch_avg<3, 8>(dd, n_freq, f0, df, off, n_bins, P, f, nu, n_channels, sm);
    else if (width >= 12.0)
        e = launch_avg<3, 4>(dd, n_freq, f0, df, off, n_bins, P, f, nu, n_channels, sm);
    else
        e = launch_avg<3, 1>(dd, n_freq, f0, df, off, n_bins, P, f, nu, n_channels, sm);
    return check_cuda(e);
}

LISA_DEBUG_TU(prep)
