// Thermochemistry kernels (first pass, lane-per-cell drain, team-per-cell
// kernel) and their launch sequence, templated on the group count G, the
// photon storage type P (double: RT_FP64; float: RT_MIXED), FP32 rate
// transcendentals R32 (RT_MIXED32) and smoothed RT SM (Sec. 3.4).  Each
// launcher translation unit instantiates one (P, R32) family, so the
// families compile in parallel.
//
// Smoothed RT: on entry N, F hold the result N', F' of injection and
// transport and Npre, Fpre the state before them.  The first pass loads
// N^t = Npre and Ndot = (N' - N^t)/dt per group; a cell's flux is kept as
// F = Fs F_base + Fb Fdot with Fs = prod 1/(1 + h D), Fb = sum h prod
// 1/(1 + h D) over its accepted sub-steps.  A cell handed to a queue
// leaves its partial N, F in N, F and its Ndot, Fdot in Npre, Fpre.
#pragma once

#include <cuda_runtime.h>

#include "rates.cuh"
#include "rt_internal.h"
#include "thermo_step.cuh"

namespace rtgb {
namespace {

using namespace thermo_detail;

constexpr int kPass1Block = 128;
constexpr int kTeam = 4;            // lanes per cell of thermo_team
constexpr double kLongSteps = 32.0; // sub-steps ahead from which a queued cell is taken early

// first: the cell's first load in this RT step (thermo_pass1).  PT: 1, or the
// lanes of the cell's team, each of which loads and stores its own groups
template <int G, int PT, typename P, bool R32, bool SM>
__device__ __forceinline__ void load_cell(const ThermoParams &p, long long c, bool first, const double *xHII,
                                          const double *xHeII, const double *xHeIII, const double *T,
                                          const P *N, const P *Npre, const double *fscale,
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
            if (first) {
                const double n0 = (double)Npre[k];
                st.Nd[r] = ((double)N[k] - n0) / p.dt;   // Eq. (smoothrate1)
                st.N[r] = n0;
            } else {
                st.N[r] = (double)N[k];
                st.Nd[r] = (double)Npre[k];
            }
            st.Fb[r] = first ? 0.0 : fscale[(long long)(G + i) * p.nc + c];
        } else {
            st.N[r] = (double)N[k];
        }
        st.Fs[r] = first ? 1.0 : fscale[k];
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

// handoff: the cell goes to a queue unfinished.  Its flux scale (and Fdot
// weight) then goes to fscale and F keeps F_base: the flux is formed once,
// when the cell finishes, so it does not depend on where it sub-cycled.
template <int G, int PT, typename P, bool SM>
__device__ __forceinline__ void store_cell(const ThermoParams &p, long long c, bool first, bool handoff,
                                           double *xHII, double *xHeII, double *xHeIII, double *T, P *N, P *F,
                                           P *Npre, P *Fpre, double *fscale,
                                           const CellState<lane_groups<>(G, PT)> &st, unsigned *status)
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
        N[(long long)i * p.nc + c] = (P)st.N[r];
        bad |= !isfinite(st.N[r]);
        if (handoff) {
            fscale[(long long)i * p.nc + c] = st.Fs[r];
            if constexpr (SM) fscale[(long long)(G + i) * p.nc + c] = st.Fb[r];
        }
        if constexpr (SM) {
            if (handoff && !first) continue;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const long long b = (3LL * i + d) * p.nc + c;
                double base, fd;
                if (first) {
                    base = (double)Fpre[b];
                    fd = ((double)F[b] - base) / p.dt;   // Eq. (smoothrate2)
                } else {
                    base = (double)F[b];
                    fd = (double)Fpre[b];
                }
                if (handoff) {
                    F[b] = Fpre[b];
                    Fpre[b] = (P)fd;
                } else {
                    F[b] = (P)(st.Fs[r] * base + st.Fb[r] * fd);
                }
            }
            if (handoff) Npre[(long long)i * p.nc + c] = (P)st.Nd[r];
        } else if (!handoff && st.Fs[r] != 1.0) {
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

template <int G, typename P, bool R32, bool SM>
__global__ void __launch_bounds__(kPass1Block)
thermo_pass1(ThermoParams p, const double *__restrict__ nH, double *xHII, double *xHeII, double *xHeIII,
             double *T, P *N, P *F, P *Npre, P *Fpre, int32_t *subcycles, Queue q, unsigned *status)
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
        load_cell<G, 1, P, R32, SM>(p, c, true, xHII, xHeII, xHeIII, T, N, Npre, q.fscale, st, iso, cc);
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
        store_cell<G, 1, P, SM>(p, c, true, !done, xHII, xHeII, xHeIII, T, N, F, Npre, Fpre, q.fscale, st, status);
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

// The lane-per-cell drain, for long queues only (more than lane_min cells):
// cells of queue A sub-cycle here for at most lane_budget attempts, every
// lane taking items one at a time; a cell still unfinished moves to queue B.
template <int G, typename P, bool R32, bool SM>
__global__ void __launch_bounds__(128)
thermo_drain(ThermoParams p, const double *__restrict__ nH, double *xHII, double *xHeII, double *xHeIII,
             double *T, P *N, P *F, P *Npre, P *Fpre, int32_t *subcycles, Queue q, unsigned *status)
{
    const QueueView qv(q);
    if ((long long)qv.total <= p.lane_min) return;
    CellState<G> st;
    IsoRates<> iso;
    CoolCache<> cc;
    double t_left = 0.0, dt_tc = 0.0, n = 0.0;
    int att = 0, used = 0;
    long long c = -1;
    bool have = false;
    auto fetch = [&]() {
        const unsigned long long it = atomicAdd(&q.counters[2], 1ULL);
        have = it < qv.total;
        if (have) {
            const unsigned long long sl = qv.slot(q, it);
            c = q.a.cell[sl];
            t_left = q.a.t_left[sl];
            dt_tc = q.a.dt_tc[sl];
            att = q.a.attempts[sl];
            n = nH[c];
            used = 0;
            load_cell<G, 1, P, R32, SM>(p, c, false, xHII, xHeII, xHeIII, T, N, Npre, q.fscale, st, iso, cc);
            cell_constants(p, n, iso);
        }
    };
    fetch();
    while (have) {
        bool done = subcycle_once<G, 1, R32, double, SM>(p, n, st, t_left, dt_tc, att, iso, cc);
        if (!done && att >= p.max_sub) {
            atomicOr(status, kStatusSubcycle);
            done = true;
        }
        if (done) {
            store_cell<G, 1, P, SM>(p, c, false, false, xHII, xHeII, xHeIII, T, N, F, Npre, Fpre, q.fscale, st, status);
            subcycles[c] = att;
            fetch();
        } else if (++used >= p.lane_budget) {
            // long sub-cycler: hand it to the team kernel
            store_cell<G, 1, P, SM>(p, c, false, true, xHII, xHeII, xHeIII, T, N, F, Npre, Fpre, q.fscale, st, status);
            const unsigned long long slot = atomicAdd(&q.counters[3], 1ULL);
            push_item(q.b, slot, q.capacity, (uint32_t)c, t_left, dt_tc, att, status);
            fetch();
        }
    }
}

// A team of four lanes per queued cell, eight cells per warp: the team's
// lanes share the cell's rate functions (one softplus and exponential each
// instead of four to eleven) and photon groups.  Bound by the length of an
// attempt, a chain of dependent FP32 pair and FP64 operations in which a warp
// of one cell and a warp of eight take the same time; a pair of warps per
// cell, the kernel before, was no shorter and spent sixteen times the issue
// slots and FP64 instructions per cell.  The first items go to different
// warps, spread over the SMs, then each team takes the next one.
template <int G, typename P, bool R32, bool SM>
__global__ void __launch_bounds__(128)
thermo_team(ThermoParams p, const double *__restrict__ nH, double *xHII, double *xHeII, double *xHeIII,
            double *T, P *N, P *F, P *Npre, P *Fpre, int32_t *subcycles, Queue q, unsigned *status)
{
    const QueueView qv(q);
    const bool drained = (long long)qv.total > p.lane_min;   // the cells left are in queue B
    unsigned long long count = drained ? q.counters[3] : qv.total;
    if (count > (unsigned long long)q.capacity) count = (unsigned long long)q.capacity;
    const QueueArrays src = drained ? q.b : q.a;
    const unsigned mask = team_mask<kTeam>();
    const int t = team_lane<kTeam>();
    // item order of the first round: warp 0 of every block, warp 1, ...
    const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    const unsigned long long first = ((threadIdx.x & 31) / kTeam) * warps + (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const unsigned long long teams = warps * (32 / kTeam);
    CellState<lane_groups<>(G, kTeam)> st;
    IsoRates<> iso;
    CoolCache<> cc;
    double t_left = 0.0, dt_tc = 0.0, n = 0.0;
    int att = 0;
    long long c = -1;
    unsigned long long it = first;
    auto load = [&]() {
        if (it >= count) return false;
        const unsigned long long sl = drained ? it : qv.slot(q, it);
        c = src.cell[sl];
        t_left = src.t_left[sl];
        dt_tc = src.dt_tc[sl];
        att = src.attempts[sl];
        n = nH[c];
        load_cell<G, kTeam, P, R32, SM>(p, c, false, xHII, xHeII, xHeIII, T, N, Npre, q.fscale, st, iso, cc);
        cell_constants(p, n, iso);
        return true;
    };
    bool have = load();
    while (have) {
        bool done = subcycle_once<G, kTeam, R32, double, SM>(p, n, st, t_left, dt_tc, att, iso, cc);
        if (!done && att >= p.max_sub) {
            if (t == 0) atomicOr(status, kStatusSubcycle);
            done = true;
        }
        if (done) {
            store_cell<G, kTeam, P, SM>(p, c, false, false, xHII, xHeII, xHeIII, T, N, F, Npre, Fpre, q.fscale, st,
                                        status);
            if (t == 0) subcycles[c] = att;
            it = count;
            if (count > teams) {
                if (t == 0) it = teams + atomicAdd(&q.counters[4], 1ULL);
                it = __shfl_sync(mask, it, 0, kTeam);
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
    static int per_sm[2] = {0, 0};
    if (per_sm[0] == 0) {
        int a = 0, b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, thermo_drain<G, P, R32, SM>, 128, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, thermo_team<G, P, R32, SM>, 128, 0);
        per_sm[1] = b < 1 ? 1 : b;
        per_sm[0] = a < 1 ? 1 : a;
    }
    auto grid = [&](int k, long long cells_per_block) {
        const long long g = (long long)per_sm[k] * n_sm, need = (tp.nc + cells_per_block - 1) / cells_per_block;
        return (unsigned)(g < need ? g : need);
    };
    if (ev) { cudaEventRecord(ev[1], s); cudaEventRecord(ev[2], s); }
    if (tp.nc > tp.lane_min) {   // (otherwise the queue cannot hold that many)
        thermo_drain<G, P, R32, SM><<<grid(0, 128), 128, 0, s>>>(tp, nH, xHII, xHeII, xHeIII, T, N, F, Npre, Fpre, sub,
                                                                q, status);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    thermo_team<G, P, R32, SM><<<grid(1, 128 / kTeam), 128, 0, s>>>(tp, nH, xHII, xHeII, xHeIII, T, N, F, Npre, Fpre,
                                                                   sub, q, status);
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
