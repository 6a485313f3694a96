// tau_device.cuh -- mixed-precision tau-leaping on the GPU.
//
// Explicit tau-leaping (the approximate family of the paper's Table 1; its
// combination with reduced precision is untested there, Sec. 5, and named as
// future work, Sec. 6): with a fixed leap tau, each leap fires k_j ~ Poisson(a_j tau)
// of every channel at once, x += sum_j nu_j k_j.  Contract (shared with the
// oracle, written independently):
//  * leap n covers [n tau, (n+1) tau), L = ceil(t_end / tau) leaps; the leap
//    grid is exact binary64; before leap n every sample s_k < (n+1) tau
//    receives the current state, after the last leap the rest the final one;
//  * a_j by the direct method's propensity contract; lambda_j = a_j * tau in
//    the accumulator type, or rnd16(a_j * rnd16(tau)) in uniform modes (SR
//    slot sr_ops + j); SR slots of leap n come from stream 1 blocks [nB, (n+1)B);
//  * k_j from the Poisson sampler below (binary64 in FP64 mode, binary32
//    otherwise): Knuth's multiplication method for lambda < 10, Hoermann's
//    transformed rejection (PTRS) at 10 and above, uniforms from Philox with
//    counter (word block, leap n, trajectory id, 2 + j);
//  * x += sum_j nu_j k_j in 64-bit integers, negative counts set to 0 with
//    status TAU_CLAMPED (16); the event count is sum_j k_j.
#pragma once

#include <type_traits>

#include "ssa_device.cuh"

namespace ssa {

constexpr uint32_t ST_TAU_CLAMPED = 16;

// e^x for x in [-30, 0]: x = k ln2 + r (Cody-Waite), Taylor series of e^r
// (r^7 in binary32, r^13 in binary64), times 2^k built from its bits.
__device__ __forceinline__ float exp_f32(float x)
{
    const float kLn2Hi = 0x1.62e400p-1f;
    const float kLn2Lo = 0x1.7f7d1cp-20f;
    const float kInvLn2 = 0x1.715476p+0f;
    float kf = x * kInvLn2;
    kf = kf + 0.5f;
    int k = (int)kf;
    if ((float)k > kf) k -= 1;
    const float fk = (float)k;
    float r = x - fk * kLn2Hi;
    r = r - fk * kLn2Lo;
    float p = 1.0f / 5040.0f;
    p = p * r + 1.0f / 720.0f;
    p = p * r + 1.0f / 120.0f;
    p = p * r + 1.0f / 24.0f;
    p = p * r + 1.0f / 6.0f;
    p = p * r + 0.5f;
    p = p * r + 1.0f;
    p = p * r + 1.0f;
    return p * __uint_as_float((uint32_t)(k + 127) << 23);
}

__device__ __forceinline__ double exp_f64(double x)
{
    const double kLn2Hi = 0x1.62e42fee00000p-1;
    const double kLn2Lo = 0x1.a39ef35793c76p-33;
    const double kInvLn2 = 0x1.71547652b82fep+0;
    double kf = x * kInvLn2;
    kf = kf + 0.5;
    int k = (int)kf;
    if ((double)k > kf) k -= 1;
    const double fk = (double)k;
    double r = x - fk * kLn2Hi;
    r = r - fk * kLn2Lo;
    double p = 1.0 / 6227020800.0;
    p = p * r + 1.0 / 479001600.0;
    p = p * r + 1.0 / 39916800.0;
    p = p * r + 1.0 / 3628800.0;
    p = p * r + 1.0 / 362880.0;
    p = p * r + 1.0 / 40320.0;
    p = p * r + 1.0 / 5040.0;
    p = p * r + 1.0 / 720.0;
    p = p * r + 1.0 / 120.0;
    p = p * r + 1.0 / 24.0;
    p = p * r + 1.0 / 6.0;
    p = p * r + 0.5;
    p = p * r + 1.0;
    p = p * r + 1.0;
    return p * __longlong_as_double((long long)((uint64_t)(k + 1023) << 52));
}

// log k!: summed logarithms below 10, Stirling's series at 10 and above.
__device__ __forceinline__ float logfact_f32(float k)
{
    if (k < 10.0f) {
        float s = 0.0f;
        for (int i = 2; (float)i <= k; ++i) s = s + log_f32((float)i);
        return s;
    }
    const float kHalfLn2Pi = 0x1.d67f1cp-1f;
    const float x = k + 1.0f;
    const float lx = log_f32(x);
    float s = (x - 0.5f) * lx;
    s = s - x;
    s = s + kHalfLn2Pi;
    s = s + (1.0f / 12.0f) / x;
    s = s - (1.0f / 360.0f) / (x * x * x);
    return s;
}

__device__ __forceinline__ double logfact_f64(double k)
{
    if (k < 10.0) {
        double s = 0.0;
        for (int i = 2; (double)i <= k; ++i) s = s + log_f64((double)i);
        return s;
    }
    const double kHalfLn2Pi = 0x1.d67f1c864beb5p-1;
    const double x = k + 1.0;
    const double lx = log_f64(x);
    double s = (x - 0.5) * lx;
    s = s - x;
    s = s + kHalfLn2Pi;
    s = s + (1.0 / 12.0) / x;
    s = s - (1.0 / 360.0) / (x * x * x);
    s = s + (1.0 / 1260.0) / (x * x * x * x * x);
    return s;
}

template <class Model, int PREC>
__device__ void tau_finish(const RunArgs &a, Lane<Model, PREC> &L)
{
    while (L.k < a.K) {
        store_state<Model>(a, L.k, L.item, L.x, L.status);
        L.k += 1;
    }
    a.status[L.item] = L.status;
    if (a.n_events) a.n_events[L.item] = L.ev;
    if (a.t_final) a.t_final[L.item] = L.n > 0 ? (double)L.n * a.tau : 0.0;
    L.active = false;
}

// Propensities of a compiled structure: the direct method's chain (the same
// operations and rounding slots as general_propensities), unrolled.
template <class Model, int PREC, int SR>
__device__ __forceinline__ void static_propensities(const RunArgs &a, const Lane<Model, PREC> &L,
                                                    Rounder<PREC, SR> &R, typename ModeTraits<PREC>::P *prop)
{
    using P = typename ModeTraits<PREC>::P;
    unroll<Model::M>([&](auto J) {
        constexpr int j = decltype(J)::value;
        int op = Model::template chain_start<j>(a);
        if (Model::template law<j>(a) == 1) {
            const int reg = Model::template hill_reg<j>(a);
            int xr = 0;
            unroll<Model::N>([&](auto I) {
                constexpr int i = decltype(I)::value;
                if (i == reg) xr = L.x[i];
            });
            const P Pv = R.rnd((P)xr, op++);
            P q = Pv;
            const int h = Model::template hill_h<j>(a);
            for (int m = 1; m < h; ++m) q = R.rnd(q * Pv, op++);
            const P d = R.rnd(P(1) + q, op++);
            const P f = R.rnd(L.h1[j] / d, op++);
            prop[j] = R.rnd(L.h0[j] + f, op++);
        } else {
            P av = L.c[j];
            bool zero = false;
            unroll<Model::N>([&](auto I) {
                constexpr int i = decltype(I)::value;
                const int rr = Model::template order<j, i>(a);
                if (rr > 0 && !Model::template folded<j, i>(a)) {
                    zero = zero || (L.x[i] < rr);
                    for (int m = 0; m < rr; ++m) {
                        const P f = R.rnd((P)(L.x[i] - m), op++);
                        av = R.rnd(av * f, op++);
                    }
                }
            });
            prop[j] = zero ? P(0) : av;
        }
    });
}

// Smallest m >= 0 with fl(m * tau) > s in binary64.  Since fl(m * tau) does
// not decrease with m, "s < fl((n + 1) * tau)" (snapshot s is written before
// leap n) is "n + 1 >= m": the leap loop then needs no binary64 operation.
__device__ inline int64_t first_leap_after(double s, double tau)
{
    const double g = floor(s / tau);
    int64_t m = g < 0.0 ? 0 : (g > 4.0e18 ? (int64_t)4.0e18 : (int64_t)g);
    for (int i = 0; i < 64 && !((double)m * tau > s); ++i) ++m;
    for (int i = 0; i < 64 && m > 0 && (double)(m - 1) * tau > s; ++i) --m;
    return m;
}

// ------------------------------------------------------------------- a leap
// A leap's draws are independent of one another (each channel has its own
// Philox stream), but how long a draw takes differs from lane to lane: the
// multiplication method uses Poisson(lambda) + 1 uniforms, the rejection
// method accepts at once in about 9 of 10 cases and otherwise evaluates three
// logarithms and five quotients.  Run one after the other, the channels of a
// leap each wait for the slowest lane of the warp: 8.8 of 32 lanes were active
// per instruction (Schloegl, tau = 0.005).  So a leap runs in two phases:
//   1. every channel gets one Philox block: four uniforms of the
//      multiplication method, or the rejection method's first quick test.
//      What that does not settle is marked pending (its product, or the
//      candidate left for the slow test, in shared memory);
//   2. every lane works through its own pending channels, one block or
//      rejection round an iteration, so lanes wait only for the largest total
//      of a lane, not for the largest of every channel.
// Quantities that only the slow test reads are computed only there.  Measured
// (GB300, Schloegl fp32, 1.5 10^5 trajectories, 2000 leaps): 51.1 -> 28.4 ms, 23.4
// ms with the slow test decided by hardware logarithms (Rejection::settle).  In
// binary64 every operation costs 64 cycles a warp whatever its lanes, so there
// comparisons and counts are integer, and the first round's candidate is kept
// for the slow test (telegraph 1.97 -> 1.69 ms, Schloegl 2 10^4 240 -> 210 ms;
// before the phases 1.87 and birth-death at lambda = 5000 7.3 against 7.4 now).
// A network without a compiled structure adds its changes up species by species
// in a register (16 reactions, fp32, 4 10^4 trajectories: 6.5 -> 5.3 ms).
template <class R>
struct SamplerMath;
template <>
struct SamplerMath<float> {
    static __device__ __forceinline__ float half_open(uint32_t w) { return (float)(w >> 8) * 0x1p-24f; }
    static __device__ __forceinline__ float positive(uint32_t w) { return (float)((w >> 8) + 1u) * 0x1p-24f; }
    // operands here: x in [0.1, 2^61], y in [2^-48, 2^66]
    static __device__ __forceinline__ float div(float x, float y) { return div_rn(x, y); }
    static __device__ __forceinline__ float exp(float x) { return exp_f32(x); }
    static __device__ __forceinline__ float log(float x) { return log_f32(x); }
    static __device__ __forceinline__ float root(float x) { return sqrtf(x); }
    static __device__ __forceinline__ float down(float x) { return floorf(x); }
    // integral x >= 0; below 2^22 from the sum's bits (the 64-bit conversion is slow)
    static __device__ __forceinline__ int64_t to_int(float x)
    {
        if (x < 0x1p22f) return __float_as_int(x + 0x1.8p23f) - 0x4B400000;
        return (int64_t)x;
    }
    // a settled draw as its column holds it
    static __device__ __forceinline__ float draw(int k) { return (float)k; }
    static __device__ __forceinline__ float draw(float k) { return k; }
    static __device__ __forceinline__ int64_t fired(float d) { return to_int(d); }
    static __device__ __forceinline__ float logfact(float k, const float *small) { return k < 10.0f ? small[(int)k] : logfact_f32(k); }
};
template <>
struct SamplerMath<double> {
    static __device__ __forceinline__ double half_open(uint32_t w) { return u32_scaled(w); }
    static __device__ __forceinline__ double positive(uint32_t w) { return w == 0xFFFFFFFFu ? 1.0 : u32_scaled(w + 1u); }
    static __device__ __forceinline__ double div(double x, double y) { return x / y; }
    static __device__ __forceinline__ double exp(double x) { return exp_f64(x); }
    static __device__ __forceinline__ double log(double x) { return log_f64(x); }
    static __device__ __forceinline__ double root(double x) { return sqrt(x); }
    static __device__ __forceinline__ double down(double x) { return floor(x); }
    static __device__ __forceinline__ int64_t to_int(double x)
    {
        if (later(0x1p30, x)) return __double2loint(x + 0x1.8p52);
        return (int64_t)x;
    }
    // a settled draw as its column holds it: an integer, so that the
    // multiplication method's takes no binary64 operation
    static __device__ __forceinline__ double draw(int k) { return __longlong_as_double((long long)k); }
    static __device__ __forceinline__ double draw(double k) { return __longlong_as_double(to_int(k)); }
    static __device__ __forceinline__ int64_t fired(double d) { return __double_as_longlong(d); }
    static __device__ __forceinline__ double logfact(double k, const double *small) { return k < 10.0 ? small[(int)k] : logfact_f64(k); }
};

// The rejection method's constants of lambda that every round needs.  Positive
// values are compared by later(): in binary64 an integer comparison, where one
// on the binary64 pipe costs 64 cycles a warp.
template <class R>
struct Rejection {
    R slam, b, a;
    __device__ __forceinline__ explicit Rejection(R lam)
    {
        using Q = SamplerMath<R>;
        slam = Q::root(lam);
        b = R(sizeof(R) == 8 ? 0.931 : 0.931f) + R(sizeof(R) == 8 ? 2.53 : 2.53f) * slam;
        a = R(sizeof(R) == 8 ? -0.059 : -0.059f) + R(sizeof(R) == 8 ? 0.02483 : 0.02483f) * b;
    }
    // U of word w0, the distance us of |U| from 1/2 and V of word w1
    __device__ __forceinline__ R point(uint32_t w0, uint32_t w1, R &us, R &V) const
    {
        using Q = SamplerMath<R>;
        const R U = Q::half_open(w0) - R(0.5);
        V = Q::positive(w1);
        us = R(0.5) - (U < R(0) ? -U : U);
        return U;
    }
    // One round on words (w0, w1): true when it settles without the slow
    // test; then kf is the draw, or -1 when the round is rejected.
    __device__ __forceinline__ bool quick(R lam, uint32_t w0, uint32_t w1, R &us, R &V, R &kf) const
    {
        using Q = SamplerMath<R>;
        const R vr = R(sizeof(R) == 8 ? 0.9277 : 0.9277f) - Q::div(R(sizeof(R) == 8 ? 3.6224 : 3.6224f), b - R(2));
        const R U = point(w0, w1, us, V);
        if (!later(us, R(0))) {
            kf = R(-1);
            return true;
        }
        R v = (Q::div(R(2) * a, us) + b) * U;
        v = v + lam;
        v = v + R(sizeof(R) == 8 ? 0.43 : 0.43f);
        kf = Q::down(v);
        if (!later(R(sizeof(R) == 8 ? 0.07 : 0.07f), us) && !later(V, vr)) return true;   // vr >= 0.4 from lambda = 10 on
        const R kmax = lam + R(64) * slam + R(64);
        if (kf < R(0) || (later(R(sizeof(R) == 8 ? 0.013 : 0.013f), us) && later(V, us)) || later(kf, kmax)) {
            kf = R(-1);
            return true;
        }
        return false;
    }
    // The binary32 test decides by hardware logarithms first.  Both sides of the
    // inequality consist of terms of size up to `size`; the contract's operations
    // err by less than 2^-20 of it, the approximate ones (lg2.approx: 2^-22 in
    // log2, absolute for arguments in [1/2, 2] and relative elsewhere) by less
    // than 2^-19, so a difference beyond 2^-17 of it
    // has the contract's sign.  What lies closer (0.2% of the tests at lambda =
    // 20), and lambda above 2000, where the margin would settle little, is
    // evaluated as the contract says.
    __device__ __forceinline__ int settle(float lam, float us, float V, float kf, const float *small) const
    {
        auto ln = [](float x) {
            float y;
            asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
            return y * 0.693147181f;
        };
        const float invalpha = __fmaf_rn(1.1328f, rcp_seed((float)b - 3.4f), 1.1239f);
        const float edge = __fmaf_rn((float)a, rcp_seed(us * us), (float)b);
        const float lhs = ln(V * invalpha) - ln(edge);
        const float x = kf + 1.0f;
        const float llam = kf * ln(lam), lx = (x - 0.5f) * ln(x);
        const float fact = kf < 10.0f ? small[(int)kf] : lx - x + 0.918938533f + 0.0833333333f * rcp_seed(x);
        const float d = (llam - lam - fact) - lhs;
        const float size = lam + llam + lx + x + 64.0f;
        return fabsf(d) > size * 0x1p-17f ? (d > 0.0f ? 1 : -1) : 0;
    }
    __device__ __forceinline__ bool slow(R lam, R us, R V, R kf, const R *small) const
    {
        using Q = SamplerMath<R>;
        if constexpr (sizeof(R) == 4) {
            if (lam < 2000.0f) {
                const int sign = settle(lam, us, V, kf, small);
                if (sign != 0) return sign > 0;
            }
        }
        const R invalpha = R(sizeof(R) == 8 ? 1.1239 : 1.1239f) +
                           Q::div(R(sizeof(R) == 8 ? 1.1328 : 1.1328f), b - R(sizeof(R) == 8 ? 3.4 : 3.4f));
        R lhs = Q::log(V) + Q::log(invalpha);
        lhs = lhs - Q::log(Q::div(a, us * us) + b);
        R rhs = -lam + kf * Q::log(lam);
        rhs = rhs - Q::logfact(kf, small);
        return lhs <= rhs;
    }
};

// (binary32 counts in binary32: 1% faster than in integers)
template <class R>
using CountOf = typename std::conditional<sizeof(R) == 8, int, R>::type;

// Four uniforms of the multiplication method: p *= v; counts the products
// above L.  True when the last one is not (the draw is settled).
template <class R>
__device__ __forceinline__ bool multiply_block(R &p, R L, uint4 u, CountOf<R> &count)
{
    using Q = SamplerMath<R>;
    CountOf<R> c = 0;
    p = p * Q::positive(u.x); if (later(p, L)) c += 1;
    p = p * Q::positive(u.y); if (later(p, L)) c += 1;
    p = p * Q::positive(u.z); if (later(p, L)) c += 1;
    p = p * Q::positive(u.w); if (later(p, L)) c += 1;
    count = c;
    return !later(p, L);
}

// f(j) for every channel: unrolled for compiled structures (j a constant),
// a loop for the general model.
template <class Model, class F>
__device__ __forceinline__ void tau_channels(const RunArgs &a, F &&f)
{
    if constexpr (std::is_same<Model, GeneralModel>::value) {
#pragma unroll 1
        for (int j = 0; j < a.M; ++j) f(j);
    } else {
        unroll<Model::M>([&](auto J) { f((int)decltype(J)::value); });
    }
}

// col: this thread's column of three arrays of a.M values (stride bd):
// lambda; e^-lambda (multiplication method); the pending product, then the
// draw.  small: log k! for k = 0..9.
template <class Model, int PREC, int SR>
__device__ __forceinline__ void tau_leap(const RunArgs &a, Lane<Model, PREC> &L, const uint32_t *m_first, float tau32,
                                              typename ModeTraits<PREC>::P *col, int bd,
                                         const typename ModeTraits<PREC>::P *small)
{
    using Tr = ModeTraits<PREC>;
    using P = typename Tr::P;
    using Q = SamplerMath<P>;
    constexpr bool kGeneral = std::is_same<Model, GeneralModel>::value;
    const int M = kGeneral ? a.M : Model::M;
    const uint32_t n = (uint32_t)L.n;
    while (L.k < a.K && n + 1u >= m_first[L.k]) {
        store_state<Model>(a, L.k, L.item, L.x, L.status);
        L.k += 1;
    }
    uint32_t bad = 0;
    {
        Rounder<PREC, SR> R;
        if constexpr (Tr::k16 && SR) {
            const int sr_total = Model::total_chain_ops(a) + (Tr::kUniform ? Model::last(a) + 1 : 0);
            R.bits.base = (uint64_t)n * (uint64_t)((sr_total + 7) >> 3);
            R.bits.traj = L.traj;
            R.bits.k0 = a.key0;
            R.bits.k1 = a.key1;
            R.bits.cur = -1;
        }
        float tau16 = tau32;
        if constexpr (Tr::k16) tau16 = rn16<Tr::kFmt>(tau32);
        const int lam_op = Model::total_chain_ops(a);
        P prop[Model::M];
        if constexpr (kGeneral) general_propensities<PREC, SR>(a, L, R, prop);
        else static_propensities<Model, PREC, SR>(a, L, R, prop);
        tau_channels<Model>(a, [&](int j) {
            P v;
            if constexpr (Tr::kF64) v = prop[j] * a.tau;
            else if constexpr (Tr::kUniform) v = R.rnd(prop[j] * tau16, lam_op + j);
            else v = prop[j] * tau32;
            if constexpr (Tr::kF64) {
                const uint64_t b = (uint64_t)__double_as_longlong(v), inf = 0x7FF0000000000000ull;
                if ((b & 0x7FFFFFFFFFFFFFFFull) > inf) bad |= ST_NAN;
                else if (b == inf) bad |= ST_OVERFLOW;
            } else {
                if (v != v) bad |= ST_NAN;
                else if (v == P(__int_as_float(0x7F800000))) bad |= ST_OVERFLOW;
            }
            col[j * bd] = v;
        });
    }
    if (bad) {
        L.status |= bad;
        tau_finish<Model, PREC>(a, L);
    } else {
        P *const colL = col + M * bd, *const colK = colL + M * bd;
        TrajPhilox ph;
        {
            const uint64_t p1 = (uint64_t)0xCD9E8D57u * L.traj;
            const uint64_t p0 = (uint64_t)0xD2511F53u * ((uint32_t)(p1 >> 32) ^ n ^ a.key0);
            ph.cx = (uint32_t)p1 ^ (a.key0 + 0x9E3779B9u);
            ph.cz = (uint32_t)(p0 >> 32) ^ (a.key1 + 0xBB67AE85u);
            ph.cw = (uint32_t)p0;
        }
        // phase 1: one block a channel
        uint32_t pend = 0u;
        tau_channels<Model>(a, [&](int j) {
            const P lam = col[j * bd];
            P d = Q::draw(0);
            if (later(lam, P(0))) {
                const uint4 u = ph.block(0u, 2u + (uint32_t)j, a.key0, a.key1);
                if (later(P(10), lam)) {
                    const P e = Q::exp(-lam);
                    P p = P(1);
                    CountOf<P> c;
                    if (multiply_block<P>(p, e, u, c)) {
                        d = Q::draw(c);
                    } else {
                        pend |= 1u << j;
                        colL[j * bd] = e;
                        d = p;
                    }
                } else {
                    const Rejection<P> rej(lam);
                    P us, V, k;
                    if (rej.quick(lam, u.x, u.y, us, V, k) && !later(P(0), k)) {
                        d = Q::draw(k);
                    } else {   // k: the first round's candidate for the slow test, or -1
                        pend |= 1u << j;
                        d = k;
                    }
                }
            }
            colK[j * bd] = d;
        });
        // phase 2: the lane's pending channels.  The first round's candidate is kept
        // in binary64 only; in binary32 another round is cheaper than the branch
        // (Schloegl, 1.5 10^5 trajectories: 23.4 against 23.8 ms).
        constexpr bool kKeep = Tr::kF64;
        int j = 0, it = 0;
        P lam = P(0), e = P(0), p = P(0);
        auto take = [&]() {
            j = __ffs((int)pend) - 1;
            lam = col[j * bd];
            e = colL[j * bd];
            p = colK[j * bd];
            it = later(P(10), lam) || (kKeep && later(P(0), p)) ? 1 : 0;
        };
        if (pend) take();
        while (pend) {
            const bool product = later(P(10), lam);
            const uint4 u = ph.block(product ? (uint32_t)it : (uint32_t)(it >> 1), 2u + (uint32_t)j, a.key0, a.key1);
            bool done;
            P d;
            if (product) {
                CountOf<P> c;
                done = multiply_block<P>(p, e, u, c);
                c += 4 * it;
                if (it == 249 && !done) {   // 1000 uniforms: the bound of the method
                    done = true;
                    c = 999;
                }
                d = Q::draw(c);
            } else {
                const Rejection<P> rej(lam);
                P us, V, k = p;
                const bool second = (it & 1) != 0;
                const uint32_t w0 = second ? u.z : u.x, w1 = second ? u.w : u.y;
                bool settled = false;
                if (kKeep && it == 0) rej.point(w0, w1, us, V);   // its candidate is k
                else settled = rej.quick(lam, w0, w1, us, V, k);
                if (settled) done = !later(P(0), k);
                else done = rej.slow(lam, us, V, k, small);
                if (it == 99 && !done) {    // 100 rounds
                    done = true;
                    k = Q::down(lam);
                }
                d = Q::draw(k);
            }
            it += 1;
            if (done) {
                colK[j * bd] = d;
                pend &= pend - 1u;
                if (pend) take();
            }
        }
        // x += sum_j nu_j k_j
        int64_t fired = 0;
        auto move = [&](int i, int64_t dx) {
            int64_t v = (int64_t)L.x[i] + dx;
            if (v < 0) {
                v = 0;
                L.status |= ST_TAU_CLAMPED;
            }
            if (v > 2147483647) v = 2147483647;
            L.x[i] = (int)v;
        };
        if constexpr (kGeneral) {
            // one species after the other, so that its sum stays in a register;
            // in binary32 from draws narrowed to 32 bits where all of them fit
            int32_t *const narrow = reinterpret_cast<int32_t *>(col);   // lambda is no longer needed
            bool wide = Tr::kF64;
#pragma unroll 1
            for (int c = 0; c < M; ++c) {
                const int64_t k = Q::fired(colK[c * bd]);
                fired += k;
                if constexpr (!Tr::kF64) {
                    narrow[c * bd] = (int32_t)k;
                    wide = wide || k != (int64_t)(int32_t)k;
                }
            }
#pragma unroll 1
            for (int i = 0; i < a.N; ++i) {
                int64_t dx = 0;
                if (wide) {
#pragma unroll 4
                    for (int c = 0; c < M; ++c) dx += Q::fired(colK[c * bd]) * (int64_t)a.stoich[c][i];
                } else {
#pragma unroll 4
                    for (int c = 0; c < M; ++c) dx += (int64_t)narrow[c * bd] * (int64_t)a.stoich[c][i];
                }
                move(i, dx);
            }
        } else {
            int64_t dx[Model::N];
#pragma unroll
            for (int i = 0; i < Model::N; ++i) dx[i] = 0;
            unroll<Model::M>([&](auto J) {
                constexpr int c = decltype(J)::value;
                const int64_t k = Q::fired(colK[c * bd]);
                fired += k;
                unroll<Model::N>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    const int nu = Model::template nu<c, i>(a);
                    if (nu != 0) dx[i] += k * (int64_t)nu;
                });
            });
            unroll<Model::N>([&](auto I) { move(decltype(I)::value, dx[decltype(I)::value]); });
        }
        L.ev += fired;
        L.n += 1;
        if (L.n >= a.n_leaps) tau_finish<Model, PREC>(a, L);
    }
}

// Persistent tau-leaping kernel: lanes refill from the work queue as in the
// direct method; each loop iteration runs one leap.  Model is a compiled
// structure (StaticModel) or the runtime-table GeneralModel.  Dynamic shared
// memory: tau_shared_bytes.
template <class Model, int PREC, int SR>
__global__ void __launch_bounds__(256) tau_kernel(const __grid_constant__ RunArgs a)
{
    using P = typename ModeTraits<PREC>::P;
    extern __shared__ __align__(16) unsigned char tau_smem[];
    __shared__ P small[10];
    if (threadIdx.x < 10) {
        if constexpr (PREC == FP64) small[threadIdx.x] = logfact_f64((double)threadIdx.x);
        else small[threadIdx.x] = logfact_f32((float)threadIdx.x);
    }
    uint32_t *m_first = reinterpret_cast<uint32_t *>(tau_smem);
    P *col = reinterpret_cast<P *>(tau_smem + (((size_t)a.K * 4 + 15) & ~(size_t)15)) + threadIdx.x;
    for (int k = threadIdx.x; k < a.K; k += blockDim.x) {
        const int64_t m = first_leap_after(a.samples[k], a.tau);
        m_first[k] = m > 0xFFFFFFFFll ? 0xFFFFFFFFu : (uint32_t)m;   // leaps are numbered below 2^31
    }
    __syncthreads();
    const float tau32 = (float)a.tau;
    const unsigned lane = threadIdx.x & 31u;
    const P no_samples[1] = {P(0)};
    Lane<Model, PREC> L;
    L.active = false;
    bool drained = false;
    for (;;) {
        const unsigned need = __ballot_sync(0xFFFFFFFFu, !L.active && !drained);
        if (need) {
            const int leader = __ffs(need) - 1;
            unsigned long long base = 0;
            if ((int)lane == leader) base = atomicAdd(a.queue_head, (unsigned long long)__popc(need));
            base = __shfl_sync(0xFFFFFFFFu, base, leader);
            if (!L.active && !drained) {
                const unsigned long long item = base + (unsigned long long)__popc(need & ((1u << lane) - 1u));
                if (item < (unsigned long long)a.n_work) {
                    init_lane<Model, PREC>(a, L, (int64_t)item, no_samples);
                    L.ev = 0;
                    if (a.n_leaps <= 0) tau_finish<Model, PREC>(a, L);
                } else {
                    drained = true;
                }
            }
        }
        if (__ballot_sync(0xFFFFFFFFu, L.active) == 0u) break;
        if (L.active) tau_leap<Model, PREC, SR>(a, L, m_first, tau32, col, (int)blockDim.x, small);
    }
}

inline size_t tau_shared_bytes(const RunArgs &a, int block, int elem_bytes)
{
    return (((size_t)a.K * 4 + 15) & ~(size_t)15) + (size_t)3 * (size_t)a.M * (size_t)block * (size_t)elem_bytes;
}

// Launch of one structure's kernel for (precision, rounding); the grid is
// sized from occupancy (persistent), capped by the work.
template <class Model>
cudaError_t tau_launch_model(const RunArgs &a, int prec, int sr, int block, int blocks_per_sm, cudaStream_t stream,
                             int *grid_out)
{
    using K = void (*)(const RunArgs);
    K k = nullptr;
    switch (prec) {
    case FP64: k = tau_kernel<Model, FP64, 0>; break;
    case FP32: k = tau_kernel<Model, FP32, 0>; break;
    case MIXED_F16: k = sr ? tau_kernel<Model, MIXED_F16, 1> : tau_kernel<Model, MIXED_F16, 0>; break;
    case MIXED_BF16: k = sr ? tau_kernel<Model, MIXED_BF16, 1> : tau_kernel<Model, MIXED_BF16, 0>; break;
    case UNIFORM_F16: k = sr ? tau_kernel<Model, UNIFORM_F16, 1> : tau_kernel<Model, UNIFORM_F16, 0>; break;
    case UNIFORM_BF16: k = sr ? tau_kernel<Model, UNIFORM_BF16, 1> : tau_kernel<Model, UNIFORM_BF16, 0>; break;
    default: return cudaErrorInvalidValue;
    }
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // The attribute gets the same value on every call (the largest a launch can
    // ask for, 100 KB), so calls from several threads do not lower it for each other.
    const size_t smem = tau_shared_bytes(a, block, prec == FP64 ? 8 : 4);
    constexpr int kMost = kMaxK * 4 + 3 * kMaxM * 256 * 8;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, block, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    if (blocks_per_sm > 0 && blocks_per_sm < per_sm) per_sm = blocks_per_sm;
    long long grid = (long long)sms * per_sm;
    const long long need = (a.n_work + block - 1) / block;
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    *grid_out = (int)grid;
    k<<<(unsigned)grid, (unsigned)block, smem, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace ssa
