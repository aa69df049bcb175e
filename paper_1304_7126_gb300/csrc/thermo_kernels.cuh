// Thermochemistry kernels (first pass, and the two stages of the
// team-per-cell kernel) and their launch sequence, templated on the group count G, the
// photon storage type P (double: RT_FP64; float: RT_MIXED), FP32 rate
// transcendentals R32 (RT_MIXED32) and smoothed RT SM (Sec. 3.4).  Each
// launcher translation unit instantiates one (P, R32) family, so the
// families compile in parallel.
//
// Smoothed RT: on entry N, F hold the result N', F' of injection and
// transport and Npre, Fpre the state before them.  A cell starts from
// N^t = Npre with Ndot = (N' - N^t)/dt per group; its flux is kept as
// F = Fs Fpre + Fb Fdot, Fdot = (F' - Fpre)/dt, with Fs = prod 1/(1 + h D),
// Fb = sum h prod 1/(1 + h D) over its accepted sub-steps.
//
// A cell handed to a queue keeps its N in FP64 beside its flux scales (N
// itself is rounded to P once, when the cell finishes), and N', F', Npre,
// Fpre stay as they are until then: which kernel runs which of its attempts
// depends on timing and must not show in the result.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "rates.cuh"
#include "rt_internal.h"
#include "thermo_step.cuh"

namespace rtgb {
namespace {

using namespace thermo_detail;

constexpr int kPass1Block = 128;
constexpr double kLongSteps = 32.0; // sub-steps ahead from which a queued cell is taken early
constexpr double kHandSteps = 8.0;  // ... from which it moves to the second stage

// a queued cell's N in Queue::N; else (RT_FP64 without smoothing) in N, exactly
template <typename P, bool SM>
__host__ __device__ constexpr bool queue_keeps_N()
{
    return SM || !std::is_same<P, double>::value;
}

// first: the cell's first load in this RT step (thermo_pass1).  PT: 1, or the
// lanes of the cell's team, each of which loads and stores its own groups
template <int G, int PT, typename P, bool R32, bool SM>
__device__ __forceinline__ void load_cell(const ThermoParams &p, long long c, bool first, const double *xHII,
                                          const double *xHeII, const double *xHeIII, const double *T,
                                          const P *N, const P *Npre, const Queue &q,
                                          CellState<lane_groups<>(G, PT)> &st, IsoRates<> &iso, CoolCache<> &cc)
{
    st.x = xHII[c];
    st.y2 = xHeII[c];
    st.y3 = xHeIII[c];
    st.T = T[c];
#pragma unroll
    for (int r = 0; r < lane_groups<>(G, PT); ++r) {
        const int i = r * PT + team_lane<PT>();
        st.N[r] = 0.0;
        st.Fs[r] = 1.0;
        if constexpr (SM) st.Nd[r] = st.Fb[r] = 0.0;
        if (PT > 1 && i >= G) continue;
        const long long k = (long long)i * p.nc + c;
        if constexpr (SM) {
            const double n0 = (double)Npre[k];
            st.Nd[r] = ((double)N[k] - n0) / p.dt;   // Eq. (smoothrate1)
            st.N[r] = first ? n0 : q.N[k];
            st.Fb[r] = first ? 0.0 : q.fscale[(long long)(G + i) * p.nc + c];
        } else if constexpr (queue_keeps_N<P, SM>()) {
            st.N[r] = first ? (double)N[k] : q.N[k];
        } else {
            st.N[r] = (double)N[k];
        }
        st.Fs[r] = first ? 1.0 : q.fscale[k];
    }
    cc.valid = false;
    cc.rvalid = false;
    if (p.isothermal) {
        TLevel L;
        dfm::Exact e;
        t_level(st.T, L, e);
        h_rates<PT, R32>(L, 0.0, p.case_b, iso.h, e);
        if (p.helium) he_rates<PT, R32>(L, 0.0, p.case_b, iso.he, e);
    }
}

// handoff: the cell goes to a queue unfinished.  Its N, flux scale and (smoothed
// RT) Fdot weight then go to the queue's arrays, and the flux is formed once,
// when the cell finishes, so neither depends on where it sub-cycled.
template <int G, int PT, typename P, bool SM>
__device__ __forceinline__ void store_cell(const ThermoParams &p, long long c, bool handoff, double *xHII,
                                           double *xHeII, double *xHeIII, double *T, P *N, P *F, const P *Fpre,
                                           const Queue &q, const CellState<lane_groups<>(G, PT)> &st,
                                           unsigned *status)
{
    if (team_lane<PT>() == 0) {
        xHII[c] = st.x;
        xHeII[c] = st.y2;
        xHeIII[c] = st.y3;
        T[c] = st.T;
    }
    bool bad = !isfinite(st.x) || !isfinite(st.T);
#pragma unroll
    for (int r = 0; r < lane_groups<>(G, PT); ++r) {
        const int i = r * PT + team_lane<PT>();
        if (PT > 1 && i >= G) continue;
        const long long k = (long long)i * p.nc + c;
        bad |= !isfinite(st.N[r]);
        if (handoff) {
            if constexpr (queue_keeps_N<P, SM>()) q.N[k] = st.N[r];
            else N[k] = st.N[r];
            q.fscale[k] = st.Fs[r];
            if constexpr (SM) q.fscale[(long long)(G + i) * p.nc + c] = st.Fb[r];
            continue;
        }
        N[k] = (P)st.N[r];
        if constexpr (SM) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const long long b = (3LL * i + d) * p.nc + c;
                const double base = (double)Fpre[b];
                const double fd = ((double)F[b] - base) / p.dt;   // Eq. (smoothrate2)
                F[b] = (P)(st.Fs[r] * base + st.Fb[r] * fd);
            }
        } else if (st.Fs[r] != 1.0) {
            long long b = 3LL * i * p.nc + c;
            const P f = (P)st.Fs[r];
            F[b] *= f;
            F[b + p.nc] *= f;
            F[b + 2 * p.nc] *= f;
        }
    }
    if (bad) atomicOr(status, kStatusNonFinite);
}

__device__ __forceinline__ void push_item(const QueueArrays &a, unsigned long long slot, long long cap, uint32_t c,
                                          double t_left, double dt_tc, int att, unsigned *status)
{
    if (slot < (unsigned long long)cap) {
        a.cell[slot] = c;
        a.t_left[slot] = t_left;
        a.dt_tc[slot] = dt_tc;
        a.attempts[slot] = att;
    } else {
        atomicOr(status, kStatusQueue);
    }
}

// Four blocks per SM (128 registers, some spilled): 128^3 x 3 groups 1.18,
// 1.08 and 1.14 ms with three, four and five.  The more groups, the more is
// spilled and the less the fourth block gives: 96^3, three against four blocks,
// 1, 3, 5 and 8 groups 0.39, 0.84, 0.99 and 1.39 against 0.36, 0.76, 0.91 and 1.39
// ms; smoothed 0.57, 0.95, 1.33 and 1.99 against 0.54, 0.92, 1.37 and 2.00 ms.
template <int G, typename P, bool R32, bool SM>
__global__ void __launch_bounds__(kPass1Block, 4)
thermo_pass1(ThermoParams p, const double *__restrict__ nH, double *xHII, double *xHeII, double *xHeIII,
             double *T, P *N, P *F, const P *Npre, const P *Fpre, int32_t *subcycles, Queue q, unsigned *status)
{
    long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    bool valid = c < p.nc;
    bool push = false;
    double t_left = p.dt, dt_tc = p.dt;
    int att = 0;
    if (valid) {
        CellState<G> st;
        IsoRates<> iso;
        CoolCache<> cc;
        load_cell<G, 1, P, R32, SM>(p, c, true, xHII, xHeII, xHeIII, T, N, Npre, q, st, iso, cc);
        double n = nH[c];
        cell_constants(p, n, iso);
        bool done = false;
        const int lim = p.pass1_attempts < p.max_sub ? p.pass1_attempts : p.max_sub;
        for (int k = 0; k < lim && !done; ++k)
            done = subcycle_once<G, 1, R32, double, SM>(p, n, st, t_left, dt_tc, att, iso, cc);
        if (!done && att >= p.max_sub) {
            atomicOr(status, kStatusSubcycle);
            done = true;
        }
        store_cell<G, 1, P, SM>(p, c, !done, xHII, xHeII, xHeIII, T, N, F, Fpre, q, st, status);
        if (done) subcycles[c] = att;
        else push = true;
    }
    // warp-aggregated append of unfinished cells to queue A: the ones with
    // the most sub-steps ahead (at the present step length) from its front,
    // to be taken first, the others from its back
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const bool mine = push && (t_left > kLongSteps * dt_tc) == (e == 0);
        const unsigned m = __ballot_sync(0xffffffffu, mine);
        if (!m) continue;
        const int leader = __ffs(m) - 1;
        unsigned long long base = 0;
        if (lane == leader) base = atomicAdd(&q.counters[e], (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, leader) + __popc(m & ((1u << lane) - 1u));
        if (mine)
            push_item(q.a, e ? (unsigned long long)q.capacity - 1ULL - base : base, q.capacity, (uint32_t)c, t_left,
                      dt_tc, att, status);
    }
}

// Item `it` of queue A: front items first, then those at the back
struct QueueView {
    unsigned long long front, total;
    __device__ __forceinline__ explicit QueueView(const Queue &q)
        : front(q.counters[0]), total(q.counters[0] + q.counters[1])
    {
    }
    __device__ __forceinline__ unsigned long long slot(const Queue &q, unsigned long long it) const
    {
        return it < front ? it : (unsigned long long)q.capacity - 1ULL - (it - front);
    }
};

// A team of TS lanes per queued cell, 32 / TS cells per warp: the team's
// lanes share the cell's rate functions and photon groups and, where they
// can, its FP64 terms (one FP64 instruction with a term per lane).  An
// attempt is a chain of dependent FP32 pair and FP64 operations; on a warp
// alone it takes 7.0 us with teams of four (7.9 before the FP64 terms were
// shared), whether the warp holds one cell or eight, and two warps per SM
// sub-partition come close to filling the FP64 pipe.  (A pair of warps per
// cell was no shorter and spent sixteen times the issue slots and FP64
// instructions per cell.)  The first items go to different
// warps, spread over the SMs, then each team takes the next one.
//
// It runs twice.  Stage 1, for queues of more than bulk_min cells, fills the
// SMs and is bound by the FP64 pipe, of which a team of two needs half as
// much per cell as a team of four and takes longer per attempt.  Once the
// queue has run empty its warps hold a few long cells each, whose attempts
// cost a warp as much as full ones, so every 16th attempt (bulk_budget) a
// cell with many sub-steps ahead then moves to queue B.  Stage 2, teams of
// four, takes those, or a queue that was short, on few warps.
// Two stages instead of teams of four alone: 256^3 48.1 -> 39.7 ms, 128^3 with
// grown fronts 21.1 -> 17.9 ms; a queue that stage 2 holds at once gains
// nothing from stage 1.  Stage 1 at 128 registers and four blocks per SM,
// stage 2 at up to 255 (both at 128: 256^3 39.7 instead of 37.6 ms).  From five
// groups on stage 1 spills (340 bytes at eight): 96^3 with fronts in progress and
// 24000 to 31000 queued cells, both stages: 17.2 ms at three groups, 22.1 at five,
// 22.3 at eight.
template <int G, int TS, typename P, bool R32, bool SM>
__global__ void __launch_bounds__(128, TS == 2 ? 4 : 2)
thermo_team(ThermoParams p, const double *__restrict__ nH, double *xHII, double *xHeII, double *xHeIII,
            double *T, P *N, P *F, const P *Npre, const P *Fpre, int32_t *subcycles, Queue q, unsigned *status,
            unsigned few_blocks)
{
    constexpr int stage = TS == 2 ? 1 : 2;
    const QueueView qv(q);
    const bool bulk = (long long)qv.total > p.bulk_min;
    if (stage == 1 && !bulk) return;
    const bool left = stage == 2 && bulk;   // queue B
    unsigned long long count = left ? q.counters[3] : qv.total;
    if (count > (unsigned long long)q.capacity) count = (unsigned long long)q.capacity;
    const QueueArrays src = left ? q.b : q.a;
    unsigned long long *taken = &q.counters[stage == 1 ? 2 : 4];
    const unsigned per_block = blockDim.x / TS;
    // stage 2 runs on one block per SM (few_blocks) for as many cells as those
    // hold, else on two (more made the longest chains longer)
    const unsigned blocks =
        (stage == 2 && count <= (unsigned long long)few_blocks * per_block && few_blocks < gridDim.x) ? few_blocks
                                                                                                      : gridDim.x;
    if (blockIdx.x >= blocks) return;
    const unsigned mask = team_mask<TS>();
    const int t = team_lane<TS>();
    // item order of the first round: warp 0 of every block, warp 1, ...
    const unsigned long long warps = (unsigned long long)blocks * (blockDim.x >> 5);
    const unsigned long long teams = (unsigned long long)blocks * per_block;
    unsigned long long it = ((threadIdx.x & 31) / TS) * warps + (threadIdx.x >> 5) * blocks + blockIdx.x;
    CellState<lane_groups<>(G, TS)> st{};
    IsoRates<> iso{};
    CoolCache<> cc{};
    double t_left = 0.0, dt_tc = 0.0, n = 0.0;
    int att = 0, used = 0;
    long long c = -1;
    auto load = [&]() {
        if (it >= count) return false;
        const unsigned long long sl = left ? it : qv.slot(q, it);
        c = src.cell[sl];
        t_left = src.t_left[sl];
        dt_tc = src.dt_tc[sl];
        att = src.attempts[sl];
        used = 0;
        n = nH[c];
        load_cell<G, TS, P, R32, SM>(p, c, false, xHII, xHeII, xHeIII, T, N, Npre, q, st, iso, cc);
        cell_constants(p, n, iso);
        return true;
    };
    bool have = load();
    while (whole_warp<TS>() ? __any_sync(0xffffffffu, have) : have) {
        bool done = subcycle_once<G, TS, R32, double, SM>(p, n, st, t_left, dt_tc, att, iso, cc, have);
        if (!have) continue;
        if (!done && att >= p.max_sub) {
            if (t == 0) atomicOr(status, kStatusSubcycle);
            done = true;
        }
        bool hand = false;
        if (stage == 1 && !done && ++used >= p.bulk_budget) {
            used = 0;
            unsigned long long k = 0;
            if (t == 0) k = teams + *(volatile unsigned long long *)taken;
            k = __shfl_sync(mask, k, 0, TS);
            hand = k >= count && t_left > kHandSteps * dt_tc;   // the queue is empty
        }
        if (done || hand) {
            store_cell<G, TS, P, SM>(p, c, hand, xHII, xHeII, xHeIII, T, N, F, Fpre, q, st, status);
            if (t == 0) {
                if (done) subcycles[c] = att;
                else push_item(q.b, atomicAdd(&q.counters[3], 1ULL), q.capacity, (uint32_t)c, t_left, dt_tc, att, status);
            }
            it = count;
            if (count > teams) {
                if (t == 0) it = teams + atomicAdd(taken, 1ULL);
                it = __shfl_sync(mask, it, 0, TS);
            }
            have = load();
        }
    }
}

template <int G, typename P, bool R32, bool SM>
cudaError_t launch_g(const ThermoParams &tp, const double *nH, double *xHII, double *xHeII, double *xHeIII,
                     double *T, P *N, P *F, P *Npre, P *Fpre, int32_t *sub, Queue q, unsigned *status, int n_sm,
                     cudaStream_t s, cudaEvent_t *ev)
{
    const int B = kPass1Block;
    long long nb = (tp.nc + B - 1) / B;
    if (ev) cudaEventRecord(ev[0], s);
    thermo_pass1<G, P, R32, SM><<<(unsigned)nb, B, 0, s>>>(tp, nH, xHII, xHeII, xHeIII, T, N, F, Npre, Fpre, sub, q,
                                                          status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    static int per_sm = 0;
    if (per_sm == 0) {
        int k = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, thermo_team<G, 2, P, R32, SM>, 128, 0);
        per_sm = k < 1 ? 1 : k;
    }
    if (ev) { cudaEventRecord(ev[1], s); cudaEventRecord(ev[2], s); }
    ThermoParams p = tp;
    // a queue that fits two blocks per SM needs no first stage
    if (p.bulk_min < 0) p.bulk_min = 2LL * n_sm * (128 / 4);
    if (p.nc > p.bulk_min) {   // (otherwise the queue cannot hold that many)
        thermo_team<G, 2, P, R32, SM><<<(unsigned)(per_sm * n_sm), 128, 0, s>>>(p, nH, xHII, xHeII, xHeIII, T, N, F,
                                                                              Npre, Fpre, sub, q, status, 0u);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const long long g = 2LL * n_sm, need = (p.nc + 128 / 4 - 1) / (128 / 4);
    thermo_team<G, 4, P, R32, SM><<<(unsigned)(g < need ? g : need), 128, 0, s>>>(p, nH, xHII, xHeII, xHeIII, T, N, F,
                                                                                Npre, Fpre, sub, q, status,
                                                                                (unsigned)n_sm);
    if (ev) cudaEventRecord(ev[3], s);
    return cudaGetLastError();
}

template <typename P, bool R32, bool SM>
cudaError_t dispatch_g(const ThermoParams &tp, int G, const double *nH, double *xHII, double *xHeII, double *xHeIII,
                       double *T, P *N, P *F, P *Npre, P *Fpre, int32_t *sub, Queue q, unsigned *status, int n_sm,
                       cudaStream_t s, cudaEvent_t *ev)
{
#define RTGB_G(GG)                                                                                                 \
    case GG:                                                                                                       \
        return launch_g<GG, P, R32, SM>(tp, nH, xHII, xHeII, xHeIII, T, N, F, Npre, Fpre, sub, q, status, n_sm, s, \
                                        ev);
    switch (G) {
        RTGB_G(1)
        RTGB_G(2)
        RTGB_G(3)
        RTGB_G(4)
        RTGB_G(5)
        RTGB_G(6)
        RTGB_G(7)
        RTGB_G(8)
    default: return cudaErrorInvalidValue;
    }
#undef RTGB_G
}

}  // namespace
}  // namespace rtgb
