// Compares the device arithmetic of the step headers with plain IEEE operations
// over all their arguments.  Built and driven by test_gpu_arithmetic.py; each
// entry counts differing results in *bad (device).
#include <cstdint>

#include "ssa_device.cuh"

namespace {

// log of x in binary32 with a plain division: the published operations of the
// library's logarithm (argument reduction to [sqrt(1/2), sqrt(2)], atanh series).
__device__ float plain_log(float x)
{
    const float kLn2Hi = 0x1.62e400p-1f, kLn2Lo = 0x1.7f7d1cp-20f;
    uint32_t ix = __float_as_uint(x);
    int e = (int)(ix >> 23) - 127;
    float m = __uint_as_float((ix & 0x7FFFFFu) | 0x3F800000u);
    if (m > 0x1.6a09e6p+0f) {
        m = m * 0.5f;
        e += 1;
    }
    const float s = (m - 1.0f) / (m + 1.0f);
    const float z = s * s;
    float p = 2.0f / 9.0f;
    p = 2.0f / 7.0f + z * p;
    p = 2.0f / 5.0f + z * p;
    p = 2.0f / 3.0f + z * p;
    const float r = (s + s) + (s * z) * p;
    const float ef = (float)e;
    return ef * kLn2Hi + (ef * kLn2Lo + r);
}

__device__ double plain_log(double x)
{
    const double kLn2Hi = 0x1.62e42fee00000p-1, kLn2Lo = 0x1.a39ef35793c76p-33;
    const uint64_t ix = (uint64_t)__double_as_longlong(x);
    int e = (int)(ix >> 52) - 1023;
    double m = __longlong_as_double((long long)((ix & 0xFFFFFFFFFFFFFull) | 0x3FF0000000000000ull));
    if (m > 0x1.6a09e667f3bccp+0) {
        m = m * 0.5;
        e += 1;
    }
    const double s = (m - 1.0) / (m + 1.0);
    const double z = s * s;
    double p = 2.0 / 23.0;
    p = 2.0 / 21.0 + z * p;
    p = 2.0 / 19.0 + z * p;
    p = 2.0 / 17.0 + z * p;
    p = 2.0 / 15.0 + z * p;
    p = 2.0 / 13.0 + z * p;
    p = 2.0 / 11.0 + z * p;
    p = 2.0 / 9.0 + z * p;
    p = 2.0 / 7.0 + z * p;
    p = 2.0 / 5.0 + z * p;
    p = 2.0 / 3.0 + z * p;
    const double t = (s + s) + (s * z) * p;
    const double ef = (double)e;
    return ef * kLn2Hi + (ef * kLn2Lo + t);
}

__device__ void count(bool wrong, unsigned long long *bad)
{
    if (wrong) atomicAdd(bad, 1ull);
}
__device__ bool differ(float a, float b) { return __float_as_uint(a) != __float_as_uint(b); }

// -log(v 2^-24) for v = 1..2^24, alone and as either half of a pair.
__global__ void logs_24(unsigned long long *bad)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x + 1u;
    const uint32_t w = (v * 0x9E3779B1u >> 8) + 1u;
    const float want = -plain_log((float)v * 0x1p-24f), other = -plain_log((float)w * 0x1p-24f);
    float a, b, c, d;
    ssa::neg_log_u24_pair(v, w, a, b);
    ssa::neg_log_u24_pair(w, v, c, d);
    // -log(1): the sign of zero is free (it is added to a time or divided by a sum)
    count(a != want || d != want || b != other || c != other || ssa::neg_log_u24(v) != want, bad);
}

// log_f32 of every significand at two exponents.
__global__ void logs_32(unsigned long long *bad)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const float x = __uint_as_float(0x3F000000u + i);   // [1/2, 2)
    count(ssa::log_f32(x) != plain_log(x) || ssa::log_f32(x * 0x1p40f) != plain_log(x * 0x1p40f), bad);
}

// -log((w + 1) 2^-32) for all words, with and without the table.
__global__ void logs_64(unsigned long long *bad)
{
    __shared__ double2 ln2[ssa::kLn2Rows];
    for (int k = threadIdx.x; k < ssa::kLn2Rows; k += blockDim.x) ln2[k] = ssa::ln2_row(k);
    __syncthreads();
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < (1ull << 32); w += step) {
        const double want = -plain_log((double)(w + 1) * 0x1p-32);
        count(ssa::neg_log_u32((uint32_t)w, ln2) != want, bad);
        if ((w & 63u) == 0u) count(ssa::neg_log_u32((uint32_t)w, nullptr) != want, bad);
    }
}

// Quotients of two 11-bit significands (those of both 16-bit formats), at the
// exponents' ends.
__global__ void quotients_short(unsigned long long *bad)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;   // 2^20
    const float a = (float)(1024u + (i >> 10)) * 0x1p-10f, b = (float)(1024u + (i & 1023u)) * 0x1p-10f;
    count(differ(ssa::div_short(a, b), a / b), bad);
    const float sa[4] = {0x1p-24f, 0x1p-30f, 0x1p31f, 0x1p-60f}, sb[4] = {0x1p60f, 0x1p-89f, 0x1p60f, 0x1p61f};
    for (int k = 0; k < 4; ++k) count(differ(ssa::div_short(a * sa[k], b * sb[k]), (a * sa[k]) / (b * sb[k])), bad);
}

// For every divisor significand B (24 bits): its reciprocal, dividends drawn at
// random, and those whose quotient lies closest to the middle of two
// neighbours: A 2^s = (2Q + 1) B + rho 2^t with B = 2^t B', rho small and odd,
// i.e. A = rho 2^(t - s) mod B'; s = 25 for A < B, 24 for A >= B.
__global__ void quotients(unsigned long long *bad, unsigned long long *hard)
{
    const uint32_t B = (1u << 23) + blockIdx.x * blockDim.x + threadIdx.x;
    const float b = (float)B;
    const float scale[3] = {1.0f, 0x1p66f, 0x1p-113f};   // b in [2^-90, 2^90]
    for (int k = 0; k < 3; ++k) count(differ(ssa::div_rn(1.0f, b * scale[k]), 1.0f / (b * scale[k])), bad);
    uint32_t x = B * 0x9E3779B1u + 12345u;
    for (int k = 0; k < 16; ++k) {
        x = x * 1664525u + 1013904223u;
        const float a = (float)((x >> 9) | (1u << 23));
        count(differ(ssa::div_rn(a, b), a / b), bad);
        count(differ(ssa::div_rn(a * 0x1p-83f, b), (a * 0x1p-83f) / b), bad);
        count(differ(ssa::div_rn(a * 0x1p66f, b * 0x1p38f), (a * 0x1p66f) / (b * 0x1p38f)), bad);
    }
    const int t = __ffs((int)B) - 1;
    const uint32_t odd = B >> t;
    unsigned long long n = 0;
    for (int s = 24; s <= 25 && odd > 16u; ++s) {
        const uint32_t lo = s == 25 ? 1u << 23 : B, hi = s == 25 ? B : 1u << 24;   // A in [lo, hi)
        for (int rho = -7; rho <= 7; rho += 2) {
            uint32_t A = rho < 0 ? odd - (uint32_t)(-rho) : (uint32_t)rho;
            for (int h = 0; h < s - t; ++h) A = (A & 1u) ? (A + odd) >> 1 : A >> 1;
            uint64_t at = A;
            if (at < lo) at += (lo - at + odd - 1) / odd * odd;
            for (int k = 0; k < 4 && at < hi; ++k, at += odd) {
                const float a = (float)(uint32_t)at;
                count(differ(ssa::div_rn(a, b), a / b), bad);
                count(differ(ssa::div_rn(a * 0x1p-83f, b), (a * 0x1p-83f) / b), bad);
                n += 1;
            }
        }
    }
    if (n) atomicAdd(hard, n);
}

int done(cudaError_t e) { return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e); }

}  // namespace

extern "C" int check_arithmetic(int which, unsigned long long *bad, unsigned long long *hard)
{
    switch (which) {
    case 0: logs_24<<<1 << 16, 256>>>(bad); break;
    case 1: logs_32<<<1 << 16, 256>>>(bad); break;
    case 2: logs_64<<<152 * 8, 256>>>(bad); break;
    case 3: quotients_short<<<1 << 12, 256>>>(bad); break;
    case 4: quotients<<<1 << 15, 256>>>(bad, hard); break;
    default: return -1;
    }
    return done(cudaGetLastError());
}
