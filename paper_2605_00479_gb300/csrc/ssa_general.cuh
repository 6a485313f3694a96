// ssa_general.cuh -- the direct-method step of networks without a compiled
// structure (one parameter set per launch).
//
// What bounded ssa_step_general: state, constants, propensities and partial
// sums in local memory, addressed by loops over every (reaction, species)
// pair.  Here the block turns the structure into short lists once -- the
// factors (species, m) of every chain, the counts each reaction changes --
// and keeps them in shared memory; a lane's counts and partial sums are
// columns of shared memory (word index * blockDim + thread: no bank
// conflicts, and the lists' indices are the same for the whole warp).  The
// arithmetic and its shortcuts are those of ssa_fast.cuh; steps outside that
// domain run ssa_step_general, and runs that start outside it (general_plain)
// a kernel of their own.  Measured (GB300, six reactions, three species,
// 10^5 trajectories to t = 50, fp32): 48.8 -> 23.8 ms;
// repressilator with Hill exponent 3 (10^5, t = 5, mixed f16) 135.9 -> 40.9 ms.
#pragma once

namespace ssa {

struct GeneralFactor {
    int offset;      // species * blockDim: the count's place in the lane's column
    float m;
};

struct GeneralChange {
    int offset;
    float nu;
};

// Block-wide lists.  Factors of reaction j: fac[fac_end[j-1] .. fac_end[j]).
template <int PREC>
struct GeneralTables {
    using P = typename ModeTraits<PREC>::P;
    GeneralFactor fac[kMaxM * kMaxN * 3];
    GeneralChange chg[kMaxM][kMaxN];
    int fac_end[kMaxM], slot[kMaxM];   // slot: first rounding operation of the chain
    int hill[kMaxM];                   // 0, or h | regulator offset << 4
    int n_chg[kMaxM];
    P c[kMaxM], h0[kMaxM], h1[kMaxM];
    int max_chg;
    int moving;                        // bit i: species i changes or is read
};

template <int PREC>
__device__ __forceinline__ void build_general_tables(const RunArgs &a, GeneralTables<PREC> *T)
{
    using P = typename ModeTraits<PREC>::P;
    const int bd = (int)blockDim.x;
    if (threadIdx.x == 0) {
        T->max_chg = 0;
        T->moving = 0;
        int n = 0;
        for (int j = 0; j < a.M; ++j) {
            T->slot[j] = a.chain_start[j];
            T->hill[j] = 0;
            T->c[j] = to_prop<PREC>(a.cprime[j]);
            T->h0[j] = P(0);
            T->h1[j] = P(0);
            if (a.law[j] == 1) {
                T->hill[j] = a.hill_h[j] | ((a.hill_reg[j] * bd) << 4);
                T->h0[j] = to_prop<PREC>(a.hill_a0[j]);
                T->h1[j] = to_prop<PREC>(a.hill_a[j]);
                T->moving |= 1 << a.hill_reg[j];
            } else {
                for (int i = 0; i < a.N; ++i) {
                    if (a.order[j][i] == 0 || a.folded[j][i]) continue;
                    T->moving |= 1 << i;
                    for (int m = 0; m < a.order[j][i]; ++m) {
                        T->fac[n].offset = i * bd;
                        T->fac[n].m = (float)m;
                        n += 1;
                    }
                }
            }
            T->fac_end[j] = n;
            int c = 0;
            for (int i = 0; i < a.N; ++i) {
                if (a.stoich[j][i] == 0) continue;
                T->moving |= 1 << i;
                T->chg[j][c].offset = i * bd;
                T->chg[j][c].nu = (float)a.stoich[j][i];
                c += 1;
            }
            T->n_chg[j] = c;
            T->max_chg = c > T->max_chg ? c : T->max_chg;
        }
    }
    __syncthreads();
}

// Bytes of a block's columns: counts, partial sums and, in uniform modes, propensities.
__host__ __device__ inline size_t general_columns(int N, int M, int prec, int block)
{
    return (size_t)block * ((size_t)N * 4 + (size_t)M * (prec == FP64 || prec >= UNIFORM_F16 ? 8 : 4));
}

// Runs that go to the kernel without lists (PLAIN in ssa_device.cuh,
// ssa_step_general for every step): several parameter sets (the lists hold one),
// and one set where run_queue_general's steps would leave its domain anyway --
// changes above 1024 (counts stay below 2^23 + 64 * 2 * |nu| within a slice, and
// must stay exact in binary32), a moving or reactant count that starts at 2^23 or
// more, and in the 16-bit modes a Hill amplitude that, rounded to the format, is
// neither zero nor in [2^-30, 2^31] (div_short; the bounds here are one binade
// inside, and binary16 ends at 65504).
inline bool general_plain(const RunArgs &a, int prec)
{
    if (a.n_sets > 1) return true;
    for (int j = 0; j < a.M; ++j) {
        if (a.law[j] == 1 && prec >= MIXED_F16 && a.hill_a[j] != 0.0) {
            const bool f16 = prec == MIXED_F16 || prec == UNIFORM_F16;
            if (!(a.hill_a[j] >= 0x1p-29 && a.hill_a[j] <= (f16 ? 65504.0 : 0x1p30))) return true;
        }
        for (int i = 0; i < a.N; ++i) {
            const bool read = a.law[j] == 1 ? a.hill_reg[j] == i : a.order[j][i] > 0 && !a.folded[j][i];
            if (a.stoich[j][i] > 1024 || a.stoich[j][i] < -1024) return true;
            if ((read || a.stoich[j][i] != 0) && a.x0[i] >= (1 << 23)) return true;
        }
    }
    return false;
}

template <int PREC, int SR>
struct GeneralLane {
    using P = typename ModeTraits<PREC>::P;
    int *x;                        // column of counts (int between slices, binary32 within)
    P *s;                          // column of partial sums
    P *p;                          // column of propensities (uniform modes)
    int bd;
    P t;
    int64_t n;
    uint32_t traj, status;
    int k;
    bool active;
    TrajPhilox ph;
    __device__ __forceinline__ int64_t item(const RunArgs &a) const { return (int64_t)(uint32_t)(traj - a.traj_offset); }
    __device__ __forceinline__ float *f() const { return reinterpret_cast<float *>(x); }
};

template <int PREC, int SR>
__device__ __forceinline__ void general_init(const RunArgs &a, GeneralLane<PREC, SR> &L, int64_t item)
{
    L.traj = a.traj_offset + (uint32_t)item;
    L.t = 0;
    L.n = 0;
    L.k = 0;
    L.status = 0;
    L.active = true;
    L.ph.init(L.traj, a.key0, a.key1);
#pragma unroll 1
    for (int i = 0; i < a.N; ++i) L.x[i * L.bd] = a.x0_tab ? a.x0_tab[i] : a.x0[i];
}

template <int PREC, int SR>
__device__ __forceinline__ void lane_take(const RunArgs &a, const TailPool<GeneralModel, PREC> *p, int s,
                                          GeneralLane<PREC, SR> &L, const typename ModeTraits<PREC>::P *)
{
    general_init(a, L, p->item[s]);
    L.n = p->n[s];
    L.t = p->t[s];
    L.k = p->k[s];
    L.status = p->status[s];
#pragma unroll 1
    for (int i = 0; i < a.N; ++i) L.x[i * L.bd] = p->x[i][s];
}

template <int PREC, int SR>
__device__ __forceinline__ void lane_give(const RunArgs &a, TailPool<GeneralModel, PREC> *p, int s, GeneralLane<PREC, SR> &L)
{
    p->item[s] = L.item(a);
    p->n[s] = L.n;
    p->t[s] = L.t;
    p->k[s] = L.k;
    p->status[s] = L.status;
#pragma unroll 1
    for (int i = 0; i < a.N; ++i) p->x[i][s] = L.x[i * L.bd];
    L.active = false;
}

// Snapshots from L.k up to the first at or after t_new (all of them at the end).
template <int PREC, int SR>
__device__ __forceinline__ void general_snapshots(const RunArgs &a, const GeneralTables<PREC> &T, GeneralLane<PREC, SR> &L,
                                                  typename ModeTraits<PREC>::P t_new, bool ends, const typename ModeTraits<PREC>::P *smp)
{
    while (L.k < a.K && (ends || later(t_new, smp[L.k]))) {
        int row = 0;
#pragma unroll 1
        for (int i = 0; i < a.N; ++i) {
            if (!((a.out_mask >> i) & 1u)) continue;
            const int64_t idx = ((int64_t)L.k * a.out_N + row) * a.n_traj + L.item(a);
            // a held species outside every chain may lie beyond 2^24: from the initial counts
            int v = (T.moving >> i) & 1 ? __float2int_rn(L.f()[i * L.bd]) : (a.x0_tab ? a.x0_tab[i] : a.x0[i]);
            if (a.state_bytes == 2) {
                if (v > 32767) { v = 32767; L.status |= ST_STATE_RANGE; }
                if (v < -32768) { v = -32768; L.status |= ST_STATE_RANGE; }
                static_cast<int16_t *>(a.out)[idx] = (int16_t)v;
            } else {
                static_cast<int32_t *>(a.out)[idx] = v;
            }
            row += 1;
        }
        L.k += 1;
    }
}

template <int PREC, int SR>
__device__ __forceinline__ void general_end(const RunArgs &a, GeneralLane<PREC, SR> &L, int64_t n, typename ModeTraits<PREC>::P t)
{
    const int64_t it = L.item(a);
    a.status[it] = L.status;
    if (a.n_events) a.n_events[it] = n;
    if (a.t_final) a.t_final[it] = (double)t;
    L.active = false;
}

template <int PREC>
struct GeneralSlice {
    typename ModeTraits<PREC>::P t, lim;
    uint32_t n0;
    bool act, wild;
};

// Partial sums into the lane's column; returns a0.
template <int PREC, int SR>
__device__ __forceinline__ typename ModeTraits<PREC>::P general_sums(const RunArgs &a, const GeneralTables<PREC> &T,
                                                                     const GeneralLane<PREC, SR> &L, StepBits &bits)
{
    using Tr = ModeTraits<PREC>;
    using P = typename Tr::P;
    constexpr int kFmt = Tr::kFmt;
    constexpr bool kNative = Tr::k16 && SR != 1;     // round-to-nearest 16-bit chains
    using H = Native16<kFmt>;
    const float *x = L.f();
    auto rnd = [&](float v, int op) -> float {
        if constexpr (Tr::k16 && SR != 0) return sr16<kFmt>(v, bits.word(op), (op & 1) != 0);
        else return v;
    };
    P S = P(0);
    int q = 0;
#pragma unroll 1
    for (int j = 0; j < a.M; ++j) {
        const int hill = T.hill[j], end = T.fac_end[j];
        P v = T.c[j];
        if (hill == 0) {
            if constexpr (kNative) {
                uint16_t w = H::from_f32((float)v);
                for (; q < end; ++q) w = H::mul(w, H::from_f32(x[T.fac[q].offset] - T.fac[q].m));
                v = H::to_f32(w);
            } else if constexpr (Tr::kF64) {
                bool zero = false;
                for (; q < end; ++q) {
                    const float fx = x[T.fac[q].offset] - T.fac[q].m;
                    zero = zero || fx < 1.0f;
                    v = v * count_f64(fx);
                }
                v = zero ? P(0) : v;
            } else if constexpr (Tr::k16) {
                int op = T.slot[j];
                for (; q < end; ++q, op += 2) {
                    const float f = rnd(x[T.fac[q].offset] - T.fac[q].m, op);
                    v = rnd(v * f, op + 1);
                }
            } else {
                for (; q < end; ++q) v = v * (x[T.fac[q].offset] - T.fac[q].m);
            }
        } else {
            const float xr = x[hill >> 4];
            const int h = hill & 15;
            if constexpr (kNative) {
                const uint16_t Pv = H::from_f32(xr);
                uint16_t w = Pv;
                for (int m = 1; m < h; ++m) w = H::mul(w, Pv);
                float d = H::to_f32(H::add(H::from_f32(1.0f), w));
                if constexpr (kFmt == 0) d = fminf(d, 0x1p60f);
                const uint16_t f = H::from_f32(div_short((float)T.h1[j], d));
                v = H::to_f32(H::add(H::from_f32((float)T.h0[j]), f));
            } else if constexpr (Tr::k16) {
                int op = T.slot[j];
                const float Pv = rnd(xr, op++);
                float w = Pv;
                for (int m = 1; m < h; ++m) w = rnd(w * Pv, op++);
                const float d = rnd(1.0f + w, op++);
                float f = div_short((float)T.h1[j], kFmt == 0 ? fminf(d, 0x1p60f) : d);
                if constexpr (kFmt == 0) f = d > 0x1p60f ? 0.0f : f;
                f = rnd(f, op++);
                v = rnd((float)T.h0[j] + f, op);
            } else {
                P Pv;
                if constexpr (Tr::kF64) Pv = xr >= 1.0f ? count_f64(xr) : 0.0;
                else Pv = xr;
                P w = Pv;
                for (int m = 1; m < h; ++m) w = w * Pv;
                const P d = P(1) + w;
                // P^4 reaches 2^92: beyond the short division's range
                v = T.h0[j] + T.h1[j] / d;
            }
        }
        if (j == 0) S = v;
        else if constexpr (Tr::kUniform && SR == 0) S = rn16<kFmt>(S + v);
        else if constexpr (Tr::kUniform) S = rnd(S + v, (SR == 2 ? 0 : a.sr_ops) + j - 1);
        else S = S + v;
        L.s[j * L.bd] = S;
        if constexpr (Tr::kUniform) L.p[j * L.bd] = v;
    }
    return S;
}

template <int PREC, int SR>
__device__ __forceinline__ void general_step(const RunArgs &a, const GeneralTables<PREC> &T, GeneralLane<PREC, SR> &L,
                                             GeneralSlice<PREC> &W, typename ModeTraits<PREC>::P E, uint32_t w1, uint32_t n,
                                             int blocks, const typename ModeTraits<PREC>::P *smp,
                                             typename ModeTraits<PREC>::P t_end)
{
    using Tr = ModeTraits<PREC>;
    using P = typename Tr::P;
    constexpr int kFmt = Tr::kFmt;
    const int M = a.M;
    StepBits bits;
    if constexpr (Tr::k16 && SR) {
        bits.g0 = n * (uint32_t)blocks;
        bits.k0 = a.key0;
        bits.k1 = a.key1;
        bits.ph = L.ph;
        bits.cur = -1;
    }
    auto sr = [&](float v, int op) { return sr16<kFmt>(v, bits.word(op), (op & 1) != 0); };
    const P a0 = general_sums<PREC, SR>(a, T, L, bits);
    P target, t_new;
    if constexpr (Tr::kF64) {
        target = u32_scaled(w1) * a0;
        t_new = W.t + E / a0;
    } else {
        const float u2 = (float)(w1 >> 8) * 0x1p-24f;
        if constexpr (Tr::kUniform) {
            if constexpr (SR == 1) {
                const int op = a.sr_ops + M - 1;
                const float Er = sr(E, op);
                const float U2 = sr(u2, op + 1);
                const float tau = sr(div_short(Er, a0), op + 2);
                target = sr(U2 * a0, op + 3);
                t_new = sr(W.t + tau, op + 4);
            } else {
                const uint32_t eu = pack16<kFmt>(u2, E);
                const float tau = rn16<kFmt>(div_short(low16<kFmt>(eu), a0));
                target = rn16<kFmt>(high16<kFmt>(eu) * a0);
                t_new = SR == 2 ? sr(W.t + tau, M - 1) : rn16<kFmt>(W.t + tau);
            }
        } else {
            target = u2 * a0;
            t_new = W.t + div_rn(E, a0);
        }
    }
    uint32_t ab;
    constexpr uint32_t kLow = Tr::kF64 ? 0x07B00000u : 0x12800000u;
    constexpr uint32_t kSpan = Tr::kF64 ? 0x70800000u : 0x5A000000u;
    if constexpr (Tr::kF64) ab = (uint32_t)__double2hiint(a0);
    else ab = __float_as_uint(a0);
    const bool wild = ab - kLow > kSpan;
    const bool due = later(t_new, W.lim);
    if ((wild || due) && W.act) {
        if (wild) {
            W.wild = true;
            W.act = false;
            L.n = (int64_t)n;
            L.t = W.t;
        } else {
            const bool ends = later(t_new, t_end);
            general_snapshots(a, T, L, t_new, ends, smp);
            if (ends) {
                general_end(a, L, (int64_t)n, W.t);
                W.act = false;
            }
            const P s_next = L.k < a.K ? smp[L.k] : t_end;
            W.lim = later(s_next, t_end) ? t_end : s_next;
        }
    }
    if (W.act) {
        // the partial sums never decrease: the channel is the number of them
        // at or below the target
        int mu = 0;
#pragma unroll 4
        for (int j = 0; j < M - 1; ++j) mu += later(L.s[j * L.bd], target) ? 0 : 1;
        if constexpr (Tr::kUniform) {
            if (!(a0 > target)) {   // the last channel with a positive propensity fires
                mu = M - 1;
                while (mu > 0 && !(L.p[mu * L.bd] > P(0))) mu -= 1;
            }
        }
        bool negative = false;
        const int nc = T.n_chg[mu];
#pragma unroll 1
        for (int c = 0; c < T.max_chg; ++c) {
            if (c < nc) {
                float *xp = L.f() + T.chg[mu][c].offset;
                const float v = *xp + T.chg[mu][c].nu;
                *xp = v;
                negative = negative || v < 0.0f;
            }
        }
        W.t = t_new;
        if (negative) {
            L.status |= ST_STATE_RANGE;
            general_snapshots(a, T, L, t_new, true, smp);
            general_end(a, L, (int64_t)n + 1, t_new);
            W.act = false;
        }
    }
}

// run_queue_fast's loop (ssa_fast.cuh) on columns of shared memory.
template <int PREC, int SR>
__device__ __forceinline__ void run_queue_general(const RunArgs &a, const typename ModeTraits<PREC>::P *smp,
                                                  typename ModeTraits<PREC>::P t_end, const double2 *ln2,
                                                  const GeneralTables<PREC> &T, unsigned char *columns,
                                                  TailPool<GeneralModel, PREC> *pool)
{
    using Tr = ModeTraits<PREC>;
    using P = typename Tr::P;
    const int slots = !Tr::k16 || SR == 0 ? 0 : SR == 2 ? a.M : a.sr_ops + (Tr::kUniform ? a.M + 4 : 0);
    const int blocks = (slots + 7) >> 3;
    const int64_t max_fast = (blocks > 2 ? 0xFFFFFFFFll / blocks : 0x7FFFFFFFll) - 256;
    const unsigned lane = threadIdx.x & 31u;
    GeneralLane<PREC, SR> L;
    L.bd = (int)blockDim.x;
    L.s = reinterpret_cast<P *>(columns) + threadIdx.x;
    L.p = L.s + (Tr::kUniform ? a.M * L.bd : 0);
    L.x = reinterpret_cast<int *>(columns + (size_t)(Tr::kUniform ? 2 : 1) * a.M * blockDim.x * sizeof(P)) + threadIdx.x;
    L.active = false;
    L.n = 0;
    L.k = a.K;
    L.t = P(0);
    for (int i = 0; i < a.N; ++i) L.x[i * L.bd] = 0;
    bool drained = false;
    const int slice = a.slice_pairs > 0 ? a.slice_pairs : 1;
    for (;;) {
        const unsigned need = __ballot_sync(0xFFFFFFFFu, !L.active && !drained);
        if (need) {
            const int leader = __ffs(need) - 1;
            unsigned long long base = 0;
            if ((int)lane == leader) base = atomicAdd(a.queue_head, (unsigned long long)__popc(need));
            base = __shfl_sync(0xFFFFFFFFu, base, leader);
            if (!L.active && !drained) {
                const unsigned long long item = base + (unsigned long long)__popc(need & ((1u << lane) - 1u));
                if (a.resume_order) {
                    if (item < *a.resume_count) {
                        const int64_t it = a.resume_order[item];
                        general_init(a, L, it);
                        L.n = a.resume_events;
                        L.t = (P)a.park_t[it];
                        L.k = a.park_k[it];
                        L.status = a.park_status[it];
#pragma unroll 1
                        for (int i = 0; i < a.N; ++i) L.x[i * L.bd] = a.park_x[(int64_t)i * a.n_work + it];
                    } else {
                        drained = true;
                    }
                } else if (item < (unsigned long long)a.n_work) {
                    general_init(a, L, (int64_t)item);
                } else {
                    drained = true;
                }
            }
        }
        if (pool && __any_sync(0xFFFFFFFFu, drained || *(volatile int *)&pool->count > 0)) {
            if (pool_visit<GeneralModel, PREC>(a, pool, L, smp)) break;
        }
        if (__ballot_sync(0xFFFFFFFFu, L.active) == 0u) break;

        const int64_t room = a.max_events - L.n;
        bool outside = room < 2 || L.n > max_fast;
#pragma unroll 1
        for (int i = 0; i < a.N; ++i)
            if ((T.moving >> i) & 1) outside = outside || L.x[i * L.bd] >= (1 << 23);
        GeneralSlice<PREC> W;
        W.act = L.active && !outside;
        W.wild = L.active && outside;
        const int reach = !W.act ? slice : (room < 2 * (int64_t)slice ? (int)(room >> 1) : slice);
        const int pairs = __reduce_min_sync(0xFFFFFFFFu, reach);
        const bool floats = W.act;           // this lane's column holds binary32 until the slice ends
        if (floats) {
#pragma unroll 1
            for (int i = 0; i < a.N; ++i) L.f()[i * L.bd] = (float)L.x[i * L.bd];
        }
        W.t = L.t;
        W.n0 = (uint32_t)L.n;
        {
            const P s_next = L.k < a.K ? smp[L.k] : t_end;
            W.lim = later(s_next, t_end) ? t_end : s_next;
        }
        for (int s = 0; s < pairs; ++s) {
            if (W.act) {
                const uint32_t n = W.n0 + 2u * (uint32_t)s;
                const uint4 u = L.ph.block(n >> 1, 0u, a.key0, a.key1);
#pragma unroll 1
                for (uint32_t h = 0; h < 2; ++h) {
                    P E;
                    if constexpr (Tr::kF64) E = neg_log_u32(h ? u.z : u.x, ln2);
                    else E = neg_log_u24(((h ? u.z : u.x) >> 8) + 1u);
                    general_step<PREC, SR>(a, T, L, W, E, h ? u.w : u.y, n + h, blocks, smp, t_end);
                }
            }
            if (__ballot_sync(0xFFFFFFFFu, W.act) == 0u) break;
        }
        if (floats) {
#pragma unroll 1
            for (int i = 0; i < a.N; ++i) {
                if ((T.moving >> i) & 1) L.x[i * L.bd] = __float2int_rn(L.f()[i * L.bd]);
                else L.x[i * L.bd] = a.x0_tab ? a.x0_tab[i] : a.x0[i];
            }
        }
        if (W.act) {
            L.t = W.t;
            L.n += 2 * (int64_t)pairs;
        }
        if (W.wild) {   // the length of a slice through ssa_step_general, ending between pairs
            Lane<GeneralModel, PREC> G;
            init_lane<GeneralModel, PREC>(a, G, L.item(a), smp);
            G.t = L.t;
            G.n = L.n;
            G.k = L.k;
            G.status = L.status;
            G.s_next = G.k < a.K ? smp[G.k] : P(__int_as_float(0x7F800000));
#pragma unroll 1
            for (int i = 0; i < a.N; ++i) G.x[i] = L.x[i * L.bd];
#pragma unroll 1
            for (int s = 0; s < slice && G.active; ++s) {
                const uint64_t blk = (uint64_t)(G.n >> 1);
                const uint4 u = philox4x32_10(make_uint4((uint32_t)blk, (uint32_t)(blk >> 32), G.traj, 0u), a.key0, a.key1);
                if ((G.n & 1) == 0) ssa_step_general<PREC, SR, false>(a, G, u.x, u.y, smp, t_end);
                if (G.active && (G.n & 1)) ssa_step_general<PREC, SR, false>(a, G, u.z, u.w, smp, t_end);
            }
            L.t = G.t;
            L.n = G.n;
            L.k = G.k;
            L.status = G.status;
            L.active = G.active;
#pragma unroll 1
            for (int i = 0; i < a.N; ++i) L.x[i * L.bd] = G.x[i];
        }
    }
}

}  // namespace ssa
