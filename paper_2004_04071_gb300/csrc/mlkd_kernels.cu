// mlkd_kernels.cu -- the correlated-pair kernel and its reductions.
//
// One lane simulates one pair at a time: the fine path of Alg. 1 at dt_l and,
// on levels l >= 1, the coarse path at dt_{l-1} = M dt_l built on the fly from
// the fine path's random numbers (Alg. 2 with the mapping of Sec. 3.1 and the
// aggregation of Sec. 3.2).  All pair state lives in registers; the only
// memory traffic is one row of block partial sums, and the histogram flush.
//
// Work distribution: each warp owns a contiguous chunk of pairs; a lane whose
// pair has finished takes the next pair of the chunk (ballot + popc), so lanes
// stay busy although pairs need different numbers of KD events.  The
// assignment depends only on the event counts, so results are reproducible.
#include <cfloat>

#include "mlkd_hetero.cuh"
#include "mlkd_internal.h"
#include "mlkd_pair.cuh"
#include "mlkd_warp_pair.cuh"

namespace mlkd {

template <typename Real> __device__ __forceinline__ const BgParams<Real> &level_params(const PairLaunch &P);
template <> __device__ __forceinline__ const BgParams<float> &level_params<float>(const PairLaunch &P) { return P.bf; }
template <> __device__ __forceinline__ const BgParams<double> &level_params<double>(const PairLaunch &P) { return P.bd; }

// Blocks per SM the register allocation must allow: FP32 state of the
// homogeneous background fits 64 registers (8 blocks of 128 threads); the
// heterogeneous pair state does not, and at 64 registers its kernel kept the
// FP64 pipe 21-83 % busy (ncu) without a line of FP64 arithmetic, so it gets
// 128 (4 blocks).  FP64 state takes what it needs (118 registers, 4 blocks).
template <typename Real, int PHYS> struct MinBlocks { static constexpr int value = PHYS == 1 ? 4 : 8; };
template <int PHYS> struct MinBlocks<double, PHYS> { static constexpr int value = 1; };

// Pair state of the two physics: the homogeneous background (PHYS 0) and the
// heterogeneous backgrounds B1/B2 of Sec. 5 (PHYS 1).
template <typename Real, int PHYS> struct PhysState { typedef PairState<Real> type; };
template <typename Real> struct PhysState<Real, 1> { typedef HetPairState<Real> type; };

// Per warp: pairs started 32 at a time, and a ring of finished pairs that are
// summed 32 at a time, so that neither path runs for only the few lanes that
// fell idle together, and lanes wait less.  For coupled homogeneous pairs, with
// a loop that holds nothing but the event (what the two gave when they came in,
// 2^20 pairs of level 8 of the periodic problem: FP32 1.37 -> 1.20 ms, FP64
// 9.16 -> 8.54; 1000 FP32 pairs of level 10 at eps = 1e-3, whose chains are all
// there is: 1.15 -> 0.86 ms).  Uncoupled
// pairs have so few events that the queues cost more than they save (5e6 paths
// of level 0: FP32 0.18 ms without, 0.21 with them), and the heterogeneous
// event is long enough (level 10 of B1: 2.39 and 2.43 ms).
template <typename Real> struct StartedPairs {
    Real x0[32], v0[32], q0[32];
    int32_t off[32];                 // pair number - the first started one's
};
template <typename Real> struct FinishedPairs {
    Real xf[64], xc[64];             // both paths at T
    uint32_t kf[64], kc[64];         // fine and coarse events
};

// Counts this block in; true in the launch's last of `blocks` to come here.
__device__ __forceinline__ bool last_to_arrive(unsigned long long *counter, unsigned long long ticket, unsigned blocks)
{
    atomicMax(counter, ticket << kTicketShift);
    return (atomicAdd(counter, 1ull) & ((1ull << kTicketShift) - 1ull)) == blocks - 1u;
}

// Sums `count` block rows, `stride` rows apart, in a fixed order; every thread
// of the block calls it.  Word j of the sum is left in s_red[0][j].
__device__ __forceinline__ void sum_rows(double *rows, int stride, int count, double (*s_red)[kPartialWords])
{
    const int t = threadIdx.x, part = t & 3;
    constexpr int kGroups = kThreads / 4, kAhead = 6;            // loads in flight per thread
    double v0 = 0.0, v1 = 0.0;
    for (int b0 = t >> 2; b0 < count; b0 += kGroups * kAhead) {
        double2 r[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int b = b0 + j * kGroups;
            r[j] = b < count ? __ldcg((const double2 *)(rows + (size_t)b * stride * kPartialWords) + part)
                             : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            v0 += r[j].x;
            v1 += r[j].y;
        }
    }
#pragma unroll
    for (int off = 16; off >= 4; off >>= 1) {
        v0 += __shfl_down_sync(kFullMask, v0, off);
        v1 += __shfl_down_sync(kFullMask, v1, off);
    }
    __syncthreads();
    if ((t & 31) < 4) {
        s_red[t >> 5][2 * part] = v0;
        s_red[t >> 5][2 * part + 1] = v1;
    }
    __syncthreads();
    if (t < kPartialWords) {
        double w = s_red[0][t];
        for (int k = 1; k < kWarpsPerBlock; ++k) w += s_red[k][t];
        s_red[0][t] = w;                                         // no other thread reads it before the next barrier
    }
    __syncthreads();
}

// Run by the last block of a launch: the summed rows into the launch's sums.
// Folding this into the pair kernel saves a launch and, in an estimate, the
// launch that accumulated the histogram, and one copy brings both results
// to the host (when it came in: 2000 FP64 pairs with 20 bins 88 -> 78 us, 300
// paths with 128 bins 50 -> 41 us, a small adaptive estimate with 64 bins
// 0.81 -> 0.70 ms).
__device__ __forceinline__ void finish_launch(const PairLaunch &P, const double *w)
{
    const int t = threadIdx.x;
    if (t == 0) {
        DevLevelStats s;
        s.n = (long long)P.n_pairs;
        s.sy = w[0];
        s.sy2 = w[1];
        s.sqf = w[2];
        s.sqf2 = w[3];
        s.sqc = w[4];
        s.sqc2 = w[5];
        s.events_f = (unsigned long long)llrint(w[6]);
        s.events_c = (unsigned long long)llrint(w[7]);
        if (P.stats) *P.stats = s;
        if (P.acc) {
            DevLevelStats &a = *P.acc;
            a.n += s.n;
            a.sy += s.sy;
            a.sy2 += s.sy2;
            a.sqf += s.sqf;
            a.sqf2 += s.sqf2;
            a.sqc += s.sqc;
            a.sqc2 += s.sqc2;
            a.events_f += s.events_f;
            a.events_c += s.events_c;
        }
    }
}

// The end of a launch.  The last block to arrive sums the rows and finishes it.
// Rows of large grids are first summed in groups, each by the group's last
// block into its first row: one block alone would wait for the FP64 pipe and the
// loads of all, and one counter for the arrivals of all (300 377 FP32 paths of
// five events, 1216 blocks: a call takes 47 us, 71 without groups).
__device__ __noinline__ void close_launch(const PairLaunch &P, double (*s_red)[kPartialWords])
{
    __shared__ bool s_last;
    const int groups = (int)gridDim.x > kOneGroup ? kArrivals - 1 : 1;
    const int per = ((int)gridDim.x + groups - 1) / groups;
    const int group = (int)blockIdx.x / per, group_first = group * per;
    const int group_size = min(per, (int)gridDim.x - group_first);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = last_to_arrive(P.arrived + 1 + group, P.ticket, (unsigned)group_size);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double *first_row = P.partials + (size_t)group_first * kPartialWords;
    sum_rows(first_row, 1, group_size, s_red);
    if (groups > 1) {
        const int used = ((int)gridDim.x + per - 1) / per;
        if (threadIdx.x < kPartialWords) first_row[threadIdx.x] = s_red[0][threadIdx.x];
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_last = last_to_arrive(P.arrived, P.ticket, (unsigned)used);
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        sum_rows(P.partials, per, used, s_red);
    }
    finish_launch(P, s_red[0]);
}

template <typename Real, int MODE, bool COUPLED, int PHYS, bool WARP = false>
__global__ void __launch_bounds__(kThreads, (MinBlocks<Real, PHYS>::value))
pair_kernel(const __grid_constant__ PairLaunch P)
{
    constexpr int CPL = COUPLED ? 1 : 0;
    constexpr int RECIPE = ModeRecipe<MODE>::value;
    extern __shared__ unsigned int s_hist[];          // [3][nbins]
    __shared__ double s_red[kWarpsPerBlock][kPartialWords];

    init_draw_tables<Real>();
    const int nbins = P.nbins;
    for (int i = threadIdx.x; i < 3 * nbins; i += blockDim.x) s_hist[i] = 0u;
    if (nbins > 0) __syncthreads();

    const BgParams<Real> &bp = level_params<Real>(P);
    LevelCtx<Real> L;
    L.bg.R = bp.R;
    L.bg.invR = bp.invR;
    L.bg.mu = bp.mu;
    L.bg.sigma = bp.sigma;
    L.bg.two_c2 = bp.two_c2;
    L.bg.dt = bp.dt;
    L.bg.Rdt = bp.Rdt;
    L.bg.inv_Rdt = bp.inv_Rdt;
    L.bg.c = bp.c;
    L.bg.c_lo = bp.c_lo;
    L.n = P.n;
    L.M = P.M;
    L.divM.init(P.M);
    L.init = P.init == 1 ? 1 : 0;          // a point start is set after pair_start
    L.word2 = P.word2;
    L.request = P.request;
    HetLevel<Real> H;
    if constexpr (PHYS == 1) {
        H.bg.b = (Real)P.bg_b;
        H.bg.a_left = (Real)P.bg_a_left;
        H.bg.a_right = (Real)P.bg_a_right;
        H.bg.dt = bp.dt;
        H.n = P.n;
        H.M = P.M;
        H.divM = L.divM;
        H.x0 = (Real)P.x0;
        H.word2 = P.word2;
        H.request = P.request;
    }

    Bins bins;
    bins.lo = P.lo;
    bins.hi = P.hi;
    bins.h = P.h;
    bins.inv_h = P.bd.inv_h;
    bins.lo_f = P.bf.lo;
    bins.hi_f = P.bf.hi;
    bins.inv_h_f = P.bf.inv_h;
    bins.nbins = nbins;
    bins.periodic = P.periodic != 0;

    const int lane = threadIdx.x & 31;
    const unsigned long long warp_id =
        (unsigned long long)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    const unsigned long long end_all = P.first_pair + P.n_pairs;
    unsigned long long w_begin = P.first_pair + warp_id * P.pairs_per_warp;
    if (w_begin > end_all) w_begin = end_all;
    unsigned long long w_end = w_begin + P.pairs_per_warp;
    if (w_end > end_all) w_end = end_all;
    unsigned long long next = w_begin;                 // warp-uniform

    bool active = false;        // the lane's pair has events left
    unsigned long long pair = 0;
    bool done = false;          // the lane holds a finished pair not yet queued for summing
    typename PhysState<Real, PHYS>::type st;
    st.fresh = true;
    // queues of started and finished pairs (see StartedPairs)
    constexpr bool kQueues = COUPLED && PHYS == 0 && !WARP;
    // Sums in shared memory with queues (they change once per 32 pairs) and in
    // FP64, so that the event loop has the registers (FP32 coupled: 64, 8
    // blocks per SM).
    constexpr bool kSharedSums = kQueues || std::is_same<Real, double>::value;
    __shared__ LaneSums<MODE> s_sums[kSharedSums ? kThreads : 1];
    LaneSums<MODE> r_sums;
    LaneSums<MODE> &sums = kSharedSums ? s_sums[kSharedSums ? threadIdx.x : 0] : r_sums;
    PairSums<MODE> &mom = sums.mom;
    unsigned long long &ev_f_sum = sums.ev_f, &ev_c_sum = sums.ev_c;
    mom.zero();
    ev_f_sum = 0;
    ev_c_sum = 0;
    const unsigned lower = (1u << lane) - 1u;

    auto record = [&](unsigned long long pair, Real xf, Real xc, uint32_t kf, uint32_t kc) {
        if (P.dbg_xf && MLKD_DCHECK(pair - P.first_pair < P.n_pairs)) {
            const unsigned long long j = pair - P.first_pair;
            P.dbg_xf[j] = (double)xf;
            if (P.dbg_xc) P.dbg_xc[j] = COUPLED ? (double)xc : 0.0;
            if (P.dbg_kf) P.dbg_kf[j] = (int32_t)kf;
            if (P.dbg_kc) P.dbg_kc[j] = (int32_t)kc;
        }
    };
    // QoI, sums and histogram of one finished pair.
    auto account = [&](Real xf, Real xc, uint32_t kf, uint32_t kc) {
        add_pair_fk(mom, xf, xc, COUPLED, P.fkind);
        ev_f_sum += kf;
        ev_c_sum += kc;
        if (nbins > 0) {
            int bf = bins(xf);
            if (!MLKD_DCHECK(bf < nbins)) bf = -1;
            if (bf >= 0) atomicAdd(&s_hist[bf], 1u);
            if (COUPLED) {
                int bc = bins(xc);
                if (!MLKD_DCHECK(bc < nbins)) bc = -1;
                if (bc >= 0) atomicAdd(&s_hist[nbins + bc], 1u);
                if (bc >= 0 && bc == bf) atomicAdd(&s_hist[2 * nbins + bf], 1u);
            }
        }
    };

    if constexpr (WARP) {
        // One pair per warp, 32 of its events per step (choose_grid has the
        // rule); lane (pair mod 32) sums it.
        for (pair = w_begin; pair < w_end; ++pair) {
            bool none = pair_start<Real, CPL, RECIPE>(st, pair, L, P.keys, COUPLED);
            if (P.init == 2) set_start(st, (Real)P.x0);
            while (!none) none = warp_pair_step<Real, RECIPE>(st, L, P.keys, COUPLED, lane);
            if (lane == (int)(pair & 31ull)) {
                pair_drift<Real, CPL>(st, L, COUPLED);
                account(st.xf, st.xc, st.k, st.evc);
                record(pair, st.xf, st.xc, st.k, st.evc);
            }
        }
    } else if constexpr (kQueues) {
    // warp-uniform: started pairs taken and held, the number of the first of
    // them, and the ring of finished pairs
    __shared__ StartedPairs<Real> s_started[kWarpsPerBlock];
    __shared__ FinishedPairs<Real> s_finished[kWarpsPerBlock];
    StartedPairs<Real> &SP = s_started[threadIdx.x >> 5];
    FinishedPairs<Real> &FP = s_finished[threadIdx.x >> 5];
    unsigned long long sp_base = w_begin;
    int sp_i = 0, sp_n = 0, fp_head = 0, fp_n = 0;
    // Moves the lane's finished pair to T.
    auto drift = [&]() {
        pair_drift<Real, CPL>(st, L, COUPLED);
        if (P.dbg_xf) record(((unsigned long long)(st.word2 ^ L.word2) << 32) | st.pair_lo, st.xf, st.xc, st.k, st.evc);
    };
    // Sums the first cnt queued pairs, one per lane.
    auto sum_finished = [&](int cnt) {
        __syncwarp();
        if (lane < cnt) {
            const int i = (fp_head + lane) & 63;
            account(FP.xf[i], FP.xc[i], FP.kf[i], FP.kc[i]);
        }
        fp_head = (fp_head + cnt) & 63;
        fp_n -= cnt;
        __syncwarp();
    };
    // Queues the pairs of the lanes with f set, in lane order; fewer than 32
    // are queued before and after.
    auto queue_finished = [&](bool f, Real xf, Real xc, uint32_t kf, uint32_t kc) {
        const unsigned m = __ballot_sync(kFullMask, f);
        if (f) {
            const int i = (fp_head + fp_n + __popc(m & lower)) & 63;
            FP.xf[i] = xf;
            FP.xc[i] = xc;
            FP.kf[i] = kf;
            FP.kc[i] = kc;
        }
        fp_n += __popc(m);
        if (fp_n >= 32) sum_finished(32);
    };
    // Starts the next pairs of the warp's range, one per lane (with no started
    // pair left).  A pair without a collision before T is finished at once.
    auto start_pairs = [&]() {
        const unsigned long long rest = w_end - next;
        const int nav = rest < 32ull ? (int)rest : 32;
        const unsigned long long p = next + (unsigned long long)lane;
        const bool have = lane < nav;
        Real x0 = Real(0), v0 = Real(0), q0 = Real(0);
        bool dead = false;
        if (have) {
            pair_start_values<Real, RECIPE>(x0, v0, q0, p, L, P.keys);
            if (P.init == 2) x0 = (Real)P.x0;
            dead = !collides_before_T(L, q0);
        }
        const Real xT = dead ? straight_to_T<Real, PHYS>(x0, v0, L) : Real(0);
        if (dead) record(p, xT, xT, 0u, 0u);
        queue_finished(dead, xT, xT, 0u, 0u);
        const bool live = have && !dead;
        const unsigned lm = __ballot_sync(kFullMask, live);
        __syncwarp();
        if (live) {
            const int i = __popc(lm & lower);
            SP.x0[i] = x0;
            SP.v0[i] = v0;
            SP.q0[i] = q0;
            SP.off[i] = lane;
        }
        sp_base = next;
        sp_n = __popc(lm);
        sp_i = 0;
        next += (unsigned long long)nav;
        __syncwarp();
    };
    unsigned idle = kFullMask;
    int need = kRefillMin<PHYS, COUPLED>;          // idle lanes that end the event loop
    for (;;) {
        if (__any_sync(kFullMask, done)) {
            if (done) drift();
            queue_finished(done, st.xf, st.xc, st.k, st.evc);
            done = false;
        }
        while (idle != 0u) {
            if (sp_i == sp_n) {
                if (next >= w_end) break;
                start_pairs();
                continue;
            }
            const int avail = sp_n - sp_i, rank = __popc(idle & lower);
            if (!active && rank < avail) {
                const int e = sp_i + rank;
                pair_init<Real, CPL>(st, sp_base + (unsigned long long)SP.off[e], SP.x0[e], SP.v0[e], SP.q0[e], L,
                                     COUPLED);
                active = true;
            }
            sp_i += min(__popc(idle), avail);
            idle = __ballot_sync(kFullMask, !active);
        }
        if (idle == kFullMask) break;
        // with nothing left to hand out, the rest runs to its end
        if (next >= w_end && sp_i == sp_n) need = 32;
        do {
            if (active && pair_event<Real, CPL, RECIPE>(st, L, P.keys, COUPLED)) {
                active = false;
                done = true;
            }
            idle = __ballot_sync(kFullMask, !active);
        } while (__popc(idle) < need);
    }
    if (fp_n > 0) sum_finished(fp_n);
    } else
    for (;;) {
        // Lanes whose pair reached T stay idle until kRefillMin of them (or
        // the whole warp) can be summed and restarted from the warp's chunk
        // in one pass.
        const unsigned idle = __ballot_sync(kFullMask, !active);
        if (idle != 0u && (__popc(idle) >= kRefillMin<PHYS, COUPLED> || idle == kFullMask)) {
            if (done) {
                if constexpr (PHYS == 1)
                    het_pair_drift<Real>(st, H, COUPLED);
                else
                    pair_drift<Real, CPL>(st, L, COUPLED);
                account(st.xf, COUPLED ? st.xc : Real(0), st.k, st.evc);
                record(pair, st.xf, st.xc, st.k, st.evc);
                done = false;
            }
            if (next < w_end) {
                const unsigned rank = __popc(idle & ((1u << lane) - 1u));
                const unsigned long long cand = next + rank;
                if (!active && cand < w_end) {
                    pair = cand;
                    bool none;
                    if constexpr (PHYS == 1) {
                        none = het_pair_start<Real, RECIPE>(st, cand, H, P.keys, COUPLED);
                    } else {
                        none = pair_start<Real, CPL, RECIPE>(st, cand, L, P.keys, COUPLED);
                        if (P.init == 2) set_start(st, (Real)P.x0);
                    }
                    if (none)
                        done = true;
                    else
                        active = true;
                }
                next += __popc(idle);
                if (next > w_end) next = w_end;
            }
        }
        if (!__any_sync(kFullMask, active)) {
            if (next >= w_end && !__any_sync(kFullMask, done)) break;
            continue;
        }
        if (active) {
            bool fin;
            if constexpr (PHYS == 1)
                fin = het_pair_event<Real, RECIPE>(st, H, P.keys, COUPLED);
            else
                fin = pair_event<Real, CPL, RECIPE>(st, L, P.keys, COUPLED);
            if (fin) {
                active = false;
                done = true;
            }
        }
    }

    // ---- block reduction of the sums (fixed order) ----
    mom.warp_reduce();
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ev_f_sum += __shfl_down_sync(kFullMask, ev_f_sum, off);
        ev_c_sum += __shfl_down_sync(kFullMask, ev_c_sum, off);
    }
    const int warp = threadIdx.x >> 5;
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < 6; ++j) s_red[warp][j] = mom.value(j);
        s_red[warp][6] = (double)ev_f_sum;
        s_red[warp][7] = (double)ev_c_sum;
    }
    __syncthreads();
    if (threadIdx.x < kPartialWords && MLKD_DCHECK(blockIdx.x < (unsigned)P.partial_rows)) {
        double acc = 0.0;
#pragma unroll
        for (int w = 0; w < kWarpsPerBlock; ++w) acc += s_red[w][threadIdx.x];
        P.partials[(size_t)blockIdx.x * kPartialWords + threadIdx.x] = acc;
    }
    if (nbins > 0 && P.hist) {
        for (int i = threadIdx.x; i < 3 * nbins; i += blockDim.x) {
            const unsigned int c = s_hist[i];
            if (c) atomicAdd(&P.hist[i], (unsigned long long)c);
        }
    }

    close_launch(P, s_red);
}

// ---------------------------------------------------------------------------
// Coarse random numbers of each pair (validation of Sec. 5.1): one thread
// per pair runs the same pair_start/pair_event as the pair kernel and
// records the first per_pair coarse steps' (nu~, E~, chi~).
// ---------------------------------------------------------------------------
struct CoarseTrace {
    double *nu, *E, *chi;
    int cap, n;
    template <typename Real> __device__ void coarse(Real a, Real b, Real c)
    {
        if (n < cap) {
            nu[n] = (double)a;
            E[n] = (double)b;
            chi[n] = (double)c;
        }
        ++n;
    }
};

template <typename Real, int MODE>
__global__ void __launch_bounds__(kThreads)
coarse_draws_kernel(const __grid_constant__ PairLaunch P, int per_pair, double *nu, double *E,
                    double *chi, int32_t *count)
{
    init_draw_tables<Real>();
    const unsigned long long j = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= P.n_pairs) return;
    const BgParams<Real> &bp = level_params<Real>(P);
    LevelCtx<Real> L;
    L.bg.R = bp.R;
    L.bg.invR = bp.invR;
    L.bg.mu = bp.mu;
    L.bg.sigma = bp.sigma;
    L.bg.two_c2 = bp.two_c2;
    L.bg.dt = bp.dt;
    L.bg.Rdt = bp.Rdt;
    L.bg.inv_Rdt = bp.inv_Rdt;
    L.bg.c = bp.c;
    L.bg.c_lo = bp.c_lo;
    L.n = P.n;
    L.M = P.M;
    L.divM.init(P.M);
    L.init = P.init;
    L.word2 = P.word2;
    L.request = P.request;
    const size_t base = (size_t)j * (size_t)per_pair;
    CoarseTrace tr{nu + base, E + base, chi + base, per_pair, 0};
    PairState<Real> st;
    st.fresh = true;
    bool done = pair_start<Real, 1, ModeRecipe<MODE>::value>(st, P.first_pair + j, L, P.keys, true);
    // a pair has at most n fine events
    for (int it = 0; !done && it <= P.n; ++it)
        done = pair_event<Real, 1, ModeRecipe<MODE>::value, CoarseTrace>(st, L, P.keys, true, &tr);
    count[j] = tr.n;
}

cudaError_t launch_coarse_draws(int mode, const PairLaunch &p, int per_pair, double *nu, double *E,
                                double *chi, int32_t *count, cudaStream_t stream)
{
    if (p.n_pairs == 0) return cudaSuccess;
    const unsigned long long blocks = (p.n_pairs + kThreads - 1) / kThreads;
    switch (mode) {
    case kModeFP64:
        coarse_draws_kernel<double, kModeFP64><<<(unsigned)blocks, kThreads, 0, stream>>>(p, per_pair, nu, E, chi, count);
        break;
    case kModeFP64U24:
        coarse_draws_kernel<double, kModeFP64U24><<<(unsigned)blocks, kThreads, 0, stream>>>(p, per_pair, nu, E, chi, count);
        break;
    default:
        coarse_draws_kernel<float, kModeFP32Comp><<<(unsigned)blocks, kThreads, 0, stream>>>(p, per_pair, nu, E, chi, count);
        break;
    }
    return cudaGetLastError();
}

// KD coefficients of eqs. advection/diffusion and the aggregation quantities
// exactly as the pair kernels compute them in precision Real, for given
// (theta, v' - mu); the level constants are prepared as for a launch (FP64 on
// the host, rounded once to Real).  In FP64 that is kd_unit, whose results in
// units of sigma/R are scaled here.  What a pair of a homogeneous background
// never has (theta < 0, sigma = 0, |v' - mu| beyond 2^400 sigma) takes
// kd_coeffs, which the heterogeneous FP64 pairs use.
template <typename Real>
__global__ void debug_kd_kernel(double R, double mu, double sigma, const double *theta,
                                const double *dv, unsigned long long n, double *a, double *d,
                                double *hs, double *om, double *bh2)
{
    Background<Real> bg;
    bg.R = (Real)R;
    bg.invR = (Real)(1.0 / R);
    bg.mu = (Real)mu;
    bg.sigma = (Real)sigma;
    bg.two_c2 = (Real)(2.0 * sigma * sigma / (R * R));
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        Real ai, di, hsi, omi;
        if constexpr (std::is_same<Real, double>::value) {
            const double s = R * theta[i], nu = fabs(dv[i]) / sigma;
            if (Arith<double>::normal_(s) && nu < 0x1p400) {
                const fx::Pos p = fx::pos_of(nu);
                const Background<double>::Unit u = Background<double>::kd_unit<true>(fx::pos_of(s), p * p);
                const double c = sigma / R, c_lo = fma(-c, R, sigma) / R;
                a[i] = fma(dv[i] * u.om, bg.invR, mu * theta[i]);
                d[i] = fma(c, u.D, c_lo * u.D);
                hs[i] = u.hs;
                om[i] = u.om;
                bh2[i] = u.beta * u.beta;
                continue;
            }
        }
        bg.kd_coeffs((Real)theta[i], (Real)dv[i], ai, di, hsi, omi);
        a[i] = (double)ai;
        d[i] = (double)di;
        hs[i] = (double)hsi;
        om[i] = (double)omi;
        bh2[i] = (double)bg.beta_hat_sq(hsi);
    }
}

cudaError_t launch_debug_kd(int fp64, double R, double mu, double sigma, const double *theta,
                            const double *dv, unsigned long long n, double *a, double *d, double *hs,
                            double *om, double *bh2, cudaStream_t stream)
{
    if (n == 0) return cudaSuccess;
    const unsigned long long blocks = (n + 255) / 256;
    const unsigned g = (unsigned)(blocks < 65536 ? blocks : 65536);
    if (fp64)
        debug_kd_kernel<double><<<g, 256, 0, stream>>>(R, mu, sigma, theta, dv, n, a, d, hs, om, bh2);
    else
        debug_kd_kernel<float><<<g, 256, 0, stream>>>(R, mu, sigma, theta, dv, n, a, d, hs, om, bh2);
    return cudaGetLastError();
}

__global__ void debug_transforms_kernel(const uint32_t *words, unsigned long long n, float *log_u,
                                        float *sn, float *cs)
{
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t w = words[i];
        if (log_u) log_u[i] = log_unit24(w);
        float a, b;
        sincos_2pi_unit24(w, &a, &b);
        if (sn) sn[i] = a;
        if (cs) cs[i] = b;
    }
}

// ---------------------------------------------------------------------------
// Sample-count controller in FP64 (eqs. mse, Nopt1, Noptj): one block.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
controller_kernel(const DevLevelStats *acc, const unsigned long long *hist_acc, int n_levels,
                  int nbins, double h, int density_qoi, double tol, DevControl *out)
{
    __shared__ double s_var[16];
    __shared__ double s_max[256];
    const int t = threadIdx.x;
    for (int l = 0; l < n_levels; ++l) {
        const double n = (double)acc[l].n;
        double v = 0.0;
        if (density_qoi && nbins > 0) {
            double m = 0.0;
            for (int b = t; b < nbins; b += 256) {
                const unsigned long long *H = hist_acc + (size_t)l * 3 * nbins;
                const double sy = (double)H[b] - (double)H[nbins + b];
                const double sy2 = (double)H[b] + (double)H[nbins + b] - 2.0 * (double)H[2 * nbins + b];
                const double vb = n >= 2.0 ? (sy2 - sy * sy / n) / (n - 1.0) : 0.0;
                m = fmax(m, vb);
            }
            s_max[t] = m;
            __syncthreads();
            for (int stride = 128; stride > 0; stride >>= 1) {
                if (t < stride) s_max[t] = fmax(s_max[t], s_max[t + stride]);
                __syncthreads();
            }
            v = s_max[0] / (h * h);
            __syncthreads();
        } else if (n >= 2.0) {
            v = (acc[l].sy2 - acc[l].sy * acc[l].sy / n) / (n - 1.0);
        }
        if (t == 0) s_var[l] = v > 0.0 ? v : 0.0;
    }
    __syncthreads();
    if (t == 0) {
        double est = 0.0, var = 0.0, total = 0.0;
        for (int l = 0; l < n_levels; ++l) {
            const double n = (double)acc[l].n;
            const double c = n > 0.0 ? (double)(acc[l].events_f + acc[l].events_c) / n : 0.0;
            out->var_level[l] = s_var[l];
            out->cost_level[l] = c;
            if (n > 0.0) {
                est += acc[l].sy / n;
                var += s_var[l] / n;
            }
            total += sqrt(s_var[l] * c);
        }
        for (int l = 0; l < n_levels; ++l) {
            const double v = s_var[l], c = out->cost_level[l];
            long long target = 0;
            if (v > 0.0 && c > 0.0 && tol > 0.0) {
                const double tg = ceil(2.0 / (tol * tol) * sqrt(v / c) * total);
                target = tg < 1e15 ? (long long)tg : 1000000000000000LL;
            }
            out->target[l] = target;
        }
        out->estimate = est;
        out->variance = var;
    }
}

// ---------------------------------------------------------------------------
// Host-side launch helpers.
// ---------------------------------------------------------------------------
namespace {

typedef void (*PairKernelFn)(const PairLaunch);

template <int PHYS>
PairKernelFn pick_lane(int mode, bool coupled)
{
    switch (mode) {
    case kModeFP64:
        return coupled ? pair_kernel<double, kModeFP64, true, PHYS> : pair_kernel<double, kModeFP64, false, PHYS>;
    case kModeFP32DY64:
        return coupled ? pair_kernel<float, kModeFP32DY64, true, PHYS>
                       : pair_kernel<float, kModeFP32DY64, false, PHYS>;
    case kModeFP64U24:
        return coupled ? pair_kernel<double, kModeFP64U24, true, PHYS>
                       : pair_kernel<double, kModeFP64U24, false, PHYS>;
    default:
        return coupled ? pair_kernel<float, kModeFP32Comp, true, PHYS>
                       : pair_kernel<float, kModeFP32Comp, false, PHYS>;
    }
}

PairKernelFn pick(int mode, bool coupled, int background, bool warp_pair)
{
    if (warp_pair)
        return mode == kModeFP64 ? pair_kernel<double, kModeFP64, true, 0, true>
                                 : pair_kernel<double, kModeFP64U24, true, 0, true>;
    return background ? pick_lane<1>(mode, coupled) : pick_lane<0>(mode, coupled);
}

}  // namespace

cudaError_t pair_kernel_info(int mode, bool coupled, int nbins, KernelInfo *out, int background, bool warp_pair)
{
    int blocks = 0;
    const size_t smem = (size_t)3 * nbins * sizeof(unsigned int);
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &blocks, (const void *)pick(mode, coupled, background, warp_pair), kThreads, smem);
    out->blocks_per_sm = blocks;
    return e;
}

cudaError_t launch_pair_kernel(int mode, bool coupled, const PairLaunch &p, int grid, cudaStream_t stream,
                               bool max_shared)
{
    cudaLaunchAttribute split;
    split.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    split.val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = (size_t)3 * p.nbins * sizeof(unsigned int);
    cfg.stream = stream;
    cfg.attrs = &split;
    cfg.numAttrs = max_shared ? 1u : 0u;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, pick(mode, coupled, p.background, p.warp_pair != 0), p);
    if (e != cudaSuccess) cudaGetLastError();     // returned here, not left for the caller's next check
    return e;
}

cudaError_t launch_controller(const DevLevelStats *acc, const unsigned long long *hist_acc,
                              int n_levels, int nbins, double h, int density_qoi, double tol,
                              DevControl *out, cudaStream_t stream)
{
    controller_kernel<<<1, 256, 0, stream>>>(acc, hist_acc, n_levels, nbins, h, density_qoi, tol,
                                             out);
    return cudaGetLastError();
}

cudaError_t launch_debug_transforms(const uint32_t *words, unsigned long long n, float *log_u,
                                    float *sn, float *cs, cudaStream_t stream)
{
    if (n == 0) return cudaSuccess;
    const unsigned long long blocks = (n + 255) / 256;
    debug_transforms_kernel<<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, stream>>>(words, n, log_u, sn, cs);
    return cudaGetLastError();
}

#ifdef MLKD_CHECKS
__global__ void check_selftest_kernel(int n)
{
    // a check that fails on purpose: the index stays clamped, nothing is written
    int i = n;
    if (!MLKD_DCHECK(i < 0)) i = 0;
    (void)i;
}
#endif

cudaError_t launch_check_selftest(cudaStream_t stream)
{
#ifdef MLKD_CHECKS
    check_selftest_kernel<<<1, 32, 0, stream>>>(1);
    return cudaGetLastError();
#else
    (void)stream;
    return cudaErrorNotSupported;
#endif
}

cudaError_t check_word_kernels(unsigned *line)
{
    *line = 0u;
#ifdef MLKD_CHECKS
    cudaError_t e = cudaMemcpyFromSymbol(line, g_mlkd_check_line, sizeof(unsigned));
    if (e != cudaSuccess) return e;
    if (*line) {
        const unsigned zero = 0u;
        e = cudaMemcpyToSymbol(g_mlkd_check_line, &zero, sizeof(unsigned));
    }
    return e;
#else
    return cudaSuccess;
#endif
}

}  // namespace mlkd
