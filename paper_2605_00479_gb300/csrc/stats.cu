// stats.cu -- on-device statistics of trajectory ensembles for the
// validation workloads (the paper's Sec. 4 comparisons: two-sample
// Kolmogorov-Smirnov statistic and Wasserstein-1 distance between the
// ensembles of two precision modes; telegraph OFF-state dwell times).
//
// Definitions (integer-exact; the oracle follows the same ones):
//  * count histogram: h[k] = #{v = k}, k = 0..bins-1; values below 0 or
//    above bins-1 go to the end bins and are counted separately;
//  * KS / W1 from two histograms: C_a, C_b cumulative counts, n_a, n_b
//    totals, diff(k) = |C_a(k) n_b - C_b(k) n_a| in 64-bit integers,
//    D = max diff / (n_a n_b), W1 = sum diff / (n_a n_b), each quotient one
//    binary64 division of the two integers (rounded to binary64 first);
//    NaN when a sample is empty or bins n_a n_b >= 2^63;
//  * dwell histogram: per trajectory of a series s[k] (nonzero = OFF),
//    every completed OFF interval, from the first OFF sample after an ON
//    sample to the first ON sample after it: h[end - start] += 1.
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/ssa.h"

namespace {

// Block-private histograms in shared memory.  What bounds the two histogram
// kernels: not the reads (4 10^6 counts are 16 MB, a few microseconds) but
// equal counts meeting -- lanes of a warp on one shared counter, blocks on one
// global counter.  So a block keeps `copies` copies (lane % copies picks one;
// their stride is odd, so one bin's copies sit in different banks), at most
// kSharedWords words in all, and there are only kBlocksPerSM blocks per SM to
// flush them.  Above kSharedBins bins every count goes to global memory.
// Measured (GB300, kernel time): 4 10^6 int32 counts in 1024 bins 18.5 -> 9.3
// us; OFF intervals of 2 10^5 series of 101 int32 samples 888 -> 36 us (one
// global atomic an interval before).
constexpr int kSharedBins = 8192;
constexpr int kSharedWords = 16384;
constexpr int kThreads = 512;
constexpr int kBlocksPerSM = 2;

// Few values: clearing and adding up the copies would cost more than the
// counts that meet in one (int32 counts, GB300 kernel time: 1001 in 1024 bins
// 2.6 us with the copies, 2.2 with one; 30001 in 251 bins 2.7 and 2.1).
constexpr int64_t kFewValues = 65536;

int histogram_copies(int bins, int64_t n)
{
    if (bins > kSharedBins) return 0;
    if (n < kFewValues) return 1;
    int c = 32;
    while (c > 1 && (int64_t)c * (bins | 1) > kSharedWords) c /= 2;
    return c;
}

size_t histogram_bytes(int bins, int copies) { return (size_t)copies * (size_t)(bins | 1) * 4; }

__device__ __forceinline__ void clear_shared(unsigned int *sh, int bins, int copies)
{
    for (int k = threadIdx.x; k < copies * (bins | 1); k += blockDim.x) sh[k] = 0u;
    __syncthreads();
}

__device__ __forceinline__ void flush_shared(const unsigned int *sh, int bins, int copies, unsigned long long *hist)
{
    __syncthreads();
    if (copies == 1) {   // four reads in flight (1001 counts in 8192 bins: 4.4 -> 2.8 us)
        for (int k = threadIdx.x; k < bins; k += 4 * blockDim.x) {
            unsigned int t[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) t[i] = k + i * (int)blockDim.x < bins ? sh[k + i * (int)blockDim.x] : 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (t[i]) atomicAdd(&hist[k + i * (int)blockDim.x], (unsigned long long)t[i]);
        }
        return;
    }
    for (int k = threadIdx.x; k < bins; k += blockDim.x) {
        unsigned int t = 0;
        for (int c = 0; c < copies; ++c) t += sh[c * (bins | 1) + k];
        if (t) atomicAdd(&hist[k], (unsigned long long)t);
    }
}

// Sixteen bytes of counts a load from the first aligned element on; the
// elements before and after are read one by one.
template <typename T>
__global__ void __launch_bounds__(kThreads) count_hist_kernel(const T *v, int64_t n, int bins, int copies,
                                                              unsigned long long *hist, unsigned long long *clamped)
{
    extern __shared__ unsigned int sh[];
    clear_shared(sh, bins, copies);
    unsigned int *mine = sh + (copies ? (int)(threadIdx.x % (unsigned)copies) * (bins | 1) : 0);
    unsigned int outside = 0;
    auto count = [&](int x) {
        if (x < 0) { x = 0; outside += 1; }
        if (x >= bins) { x = bins - 1; outside += 1; }
        if (copies) atomicAdd(&mine[x], 1u);
        else atomicAdd(&hist[x], 1ull);
    };
    constexpr int kPer = 16 / (int)sizeof(T);
    const uintptr_t addr = reinterpret_cast<uintptr_t>(v);
    int64_t head = (int64_t)(((16u - (unsigned)(addr & 15u)) & 15u) / sizeof(T));
    head = head < n ? head : n;
    const int64_t vectors = (n - head) / kPer;
    const uint4 *p = reinterpret_cast<const uint4 *>(v + head);
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    auto count4 = [&](uint4 q) {
        const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if constexpr (sizeof(T) == 4) {
                count((int)w[i]);
            } else {
                count((int)(short)(w[i] & 0xFFFFu));
                count((int)(short)(w[i] >> 16));
            }
        }
    };
    int64_t i = tid;
    for (; i + step < vectors; i += 2 * step) {   // two loads in flight
        const uint4 a = p[i], b = p[i + step];
        count4(a);
        count4(b);
    }
    if (i < vectors) count4(p[i]);
    const int64_t tail = head + vectors * kPer;
    for (int64_t e = tid; e < head + (n - tail); e += step) count((int)v[e < head ? e : tail + (e - head)]);
    for (int o = 16; o > 0; o >>= 1) outside += __shfl_xor_sync(0xFFFFFFFFu, outside, o);
    if ((threadIdx.x & 31) == 0 && outside) atomicAdd(clamped, (unsigned long long)outside);
    if (copies) flush_shared(sh, bins, copies, hist);
}

// One block of 1024 threads: thread t owns a contiguous run of bins.
__global__ void __launch_bounds__(1024) ks_w1_kernel(const unsigned long long *ha, const unsigned long long *hb,
                                                     int bins, double *out)
{
    __shared__ long long s_a[1024], s_b[1024];
    __shared__ unsigned long long s_max[1024], s_sum[1024];
    const int t = threadIdx.x, T = blockDim.x;
    const int chunk = (bins + T - 1) / T;
    const int lo = t * chunk < bins ? t * chunk : bins, hi = lo + chunk < bins ? lo + chunk : bins;
    long long la = 0, lb = 0;
    for (int k = lo; k < hi; ++k) {
        la += (long long)ha[k];
        lb += (long long)hb[k];
    }
    s_a[t] = la;
    s_b[t] = lb;
    __syncthreads();
    // inclusive scan of the per-thread totals (Hillis-Steele)
    for (int off = 1; off < T; off <<= 1) {
        const long long va = t >= off ? s_a[t - off] : 0, vb = t >= off ? s_b[t - off] : 0;
        __syncthreads();
        s_a[t] += va;
        s_b[t] += vb;
        __syncthreads();
    }
    const long long na = s_a[T - 1], nb = s_b[T - 1];
    long long ca = t > 0 ? s_a[t - 1] : 0, cb = t > 0 ? s_b[t - 1] : 0;
    unsigned long long dmax = 0, dsum = 0;
    for (int k = lo; k < hi; ++k) {
        ca += (long long)ha[k];
        cb += (long long)hb[k];
        const long long d = ca * nb - cb * na;
        const unsigned long long ad = (unsigned long long)(d < 0 ? -d : d);
        dmax = ad > dmax ? ad : dmax;
        dsum += ad;
    }
    __syncthreads();
    s_max[t] = dmax;
    s_sum[t] = dsum;
    __syncthreads();
    for (int off = T / 2; off > 0; off >>= 1) {
        if (t < off) {
            s_max[t] = s_max[t] > s_max[t + off] ? s_max[t] : s_max[t + off];
            s_sum[t] += s_sum[t + off];
        }
        __syncthreads();
    }
    if (t == 0) {
        const double nan = __longlong_as_double(0x7FF8000000000000ll);
        if (na <= 0 || nb <= 0 || (double)bins * (double)na * (double)nb >= 9223372036854775808.0) {
            out[0] = nan;
            out[1] = nan;
        } else {
            const double denom = __ll2double_rn(na * nb);
            out[0] = __ull2double_rn(s_max[0]) / denom;
            out[1] = __ull2double_rn(s_sum[0]) / denom;
        }
    }
}

// One thread a series (neighbouring series in neighbouring lanes), eight
// samples loaded ahead of the state machine that consumes them.
template <typename T>
__global__ void __launch_bounds__(kThreads) dwell_kernel(const T *s, int K, int64_t n, int64_t k_stride, int copies,
                                                         unsigned long long *hist)
{
    extern __shared__ unsigned int sh[];
    clear_shared(sh, K, copies);
    unsigned int *mine = sh + (copies ? (int)(threadIdx.x % (unsigned)copies) * (K | 1) : 0);
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        int start = -1;
        bool prev_off = s[j] != 0;
        for (int k0 = 1; k0 < K; k0 += 8) {
            T v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = k0 + i < K ? s[(int64_t)(k0 + i) * k_stride + j] : T(0);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int k = k0 + i;
                if (k >= K) break;
                const bool off = v[i] != 0;
                if (off && !prev_off) {
                    start = k;
                } else if (!off && prev_off && start >= 0) {
                    if (copies) atomicAdd(&mine[k - start], 1u);
                    else atomicAdd(&hist[k - start], 1ull);
                    start = -1;
                }
                prev_off = off;
            }
        }
    }
    if (copies) flush_shared(sh, K, copies, hist);
}

int device_sms(int *sms)
{
    int dev = 0;
    return cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
}

// Launch of a histogram kernel with its block-private counters (the attribute
// always gets the largest size, so concurrent calls do not lower it).
template <class Kernel, class... Args>
int launch_histogram(Kernel k, int64_t grid, size_t bytes, cudaStream_t s, Args... args)
{
    if (bytes > 48 * 1024 &&
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSharedWords * 4) != cudaSuccess)
        return SSA_ECUDA;
    k<<<(unsigned)grid, kThreads, bytes, s>>>(args...);
    return cudaGetLastError() == cudaSuccess ? SSA_OK : SSA_ECUDA;
}

}  // namespace

extern "C" {

int ssa_count_histogram(const void *values, int elem_bytes, int64_t n, int bins, uint64_t *hist,
                        uint64_t *n_clamped, void *stream)
{
    if (elem_bytes != 2 && elem_bytes != 4) return SSA_EINVAL;
    if (n < 0 || bins < 1 || bins > (1 << 24) || (n > 0 && (!values || !hist || !n_clamped))) return SSA_EINVAL;
    if (n == 0) return SSA_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int sms = 0;
    if (!device_sms(&sms)) return SSA_ECUDA;
    const int64_t per_block = n < kFewValues ? kThreads * 4 : kThreads * 8;
    int64_t grid = (n + per_block - 1) / per_block;
    if (grid > (int64_t)sms * kBlocksPerSM) grid = (int64_t)sms * kBlocksPerSM;
    const int copies = histogram_copies(bins, n);
    auto *h = reinterpret_cast<unsigned long long *>(hist);
    auto *c = reinterpret_cast<unsigned long long *>(n_clamped);
    const size_t bytes = histogram_bytes(bins, copies);
    if (elem_bytes == 4)
        return launch_histogram(count_hist_kernel<int32_t>, grid, bytes, s, static_cast<const int32_t *>(values), n, bins,
                                copies, h, c);
    return launch_histogram(count_hist_kernel<int16_t>, grid, bytes, s, static_cast<const int16_t *>(values), n, bins,
                            copies, h, c);
}

int ssa_hist_ks_w1(const uint64_t *ha, const uint64_t *hb, int bins, double *out, void *stream)
{
    if (!ha || !hb || !out || bins < 1 || bins > (1 << 24)) return SSA_EINVAL;
    ks_w1_kernel<<<1, 1024, 0, static_cast<cudaStream_t>(stream)>>>(
        reinterpret_cast<const unsigned long long *>(ha), reinterpret_cast<const unsigned long long *>(hb), bins, out);
    return cudaGetLastError() == cudaSuccess ? SSA_OK : SSA_ECUDA;
}

int ssa_dwell_histogram(const void *series, int elem_bytes, int K, int64_t n, int64_t k_stride, uint64_t *hist,
                        void *stream)
{
    if (elem_bytes != 2 && elem_bytes != 4) return SSA_EINVAL;
    if (K < 1 || n < 0 || k_stride < n || (n > 0 && (!series || !hist))) return SSA_EINVAL;
    if (n == 0) return SSA_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int sms = 0;
    if (!device_sms(&sms)) return SSA_ECUDA;
    int64_t grid = (n + kThreads - 1) / kThreads;
    if (grid > (int64_t)sms * 4) grid = (int64_t)sms * 4;
    const int copies = histogram_copies(K, n * K);
    auto *h = reinterpret_cast<unsigned long long *>(hist);
    const size_t bytes = histogram_bytes(K, copies);
    if (elem_bytes == 4)
        return launch_histogram(dwell_kernel<int32_t>, grid, bytes, s, static_cast<const int32_t *>(series), K, n, k_stride,
                                copies, h);
    return launch_histogram(dwell_kernel<int16_t>, grid, bytes, s, static_cast<const int16_t *>(series), K, n, k_stride,
                            copies, h);
}

}  // extern "C"
