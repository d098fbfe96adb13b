// ALNS on the device (Section 4.2, Algorithm 1): the six destroy operators
// of Section 4.2.2 (random, worst, Shaw, cluster, route, critical path), the
// four repair operators of Section 4.2.3 (greedy, regret-2, regret-3,
// regret-m) over the full insertion-delta matrix, simulated-annealing
// acceptance with gated reheat (Section 4.2.4) and adaptive roulette weights
// (Section 4.2.1).
//
// One persistent cooperative launch; a team of CTAs runs one ALNS instance
// and meets at bounded team barriers.  Per iteration:
//   gains   (worst removal only) one skip-walk per customer across the team:
//           the makespan without that customer;
//   begin   rank 0 marks the removed customers (Fisher-Yates, or a block
//           bitonic sort of (key, customer) for the structured operators) and
//           builds W = current solution without them.
// Then one insertion step per removed customer:
//   prep    each CTA stages W in shared memory (op codes packed with their
//           travel-in times), or carries the last insertion out on the copy it
//           has.  After a full step, warps walk W from the depot (node times H,
//           makespan) and from every op u (row u of the all-pairs longest-path
//           table LP, and the tail T(u)); after a plain insertion the table is
//           updated from the inserted pair instead.  Threads flag "shortcut"
//           gaps, where d(x,c) + d(c,y) < d(x,y) because of the nint rounding;
//   gaps    per-gap vectors (H of the stop before, T of the stop after, the
//           removed leg, stock prefix/suffix extremes), per-(customer, gap)
//           row and column vectors and their minima per 32 gaps, and sparse
//           tables of the stock prefix; the team then starts the shortcut
//           simulations (schedules with the single shortcut stop added) without
//           waiting for them;
//   matrix  32 x 64 tiles of (dropoff gap, pickup gap) entries for every
//           customer still to insert.  Without shortcut gaps the new makespan
//           is exactly max(z, beta, gamma, delta, epsilon): the old makespan,
//           the longest path through the new drop only, through the new pickup
//           only, through drop -> pickup by the processing edge, and through
//           drop -> route -> pickup (the LP table).  Capacity and pool are O(1)
//           from the prefix/suffix extremes.  All tiles are tested against the
//           best entries known so far first; those that may matter are scored
//           from registers and their row minima folded by route into 64-bit
//           atomics.  Entries on shortcut gaps come from the simulations;
//   select  per-customer argmin of (delta z, delta travel, flat index), then
//           the repair operator's choice across customers, by the CTA that
//           arrives last; the others carry the choice out in the next step.
// Rank 0 ends the iteration: the repaired solution, whose makespan the last
// insertion gave, is accepted or not, the temperature and weights are updated
// and the next operators are drawn.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>

#include "device_common.cuh"
#include "internal.h"

namespace vrp {

constexpr int NEG = -(1 << 30);               // "unreachable" in the longest-path table
constexpr int UNRES = INT32_MIN;               // ready value not yet published
constexpr int SKIPV = 1 << 28;                 // excluded matrix entry; schedule times stay below 2^27
// Shortcut gaps per greedy step whose simulations run ahead, in the gap phase
// (more than this, rare, are simulated inside the matrix phase instead).
// Per shortcut gap: departures and tails with the drop alone (H1, T1) and with
// the pickup alone (H2, T2), N words each, then z1, h_v1, t_v1, z2, h_v2, t_v2.
constexpr int SC_CAP = 64;
// Each shortcut item is handed out as FB_SPLIT pieces, each taking every
// FB_SPLIT-th block of the row or column: an item's entries are long chains of
// dependent loads, and whole items outlasted the rest of the matrix phase.
constexpr int FB_SPLIT = 8;
constexpr int TR = 32, TC = 64;                // matrix tile rows, cols
constexpr int ALNS_THREADS = 256;
constexpr int ALNS_WARPS = ALNS_THREADS / 32;
constexpr unsigned long long KEY_NONE = ~0ull;
constexpr long long REGRET_INF = 1ll << 40;

struct AlnsCtl {
    int iter, q, nrem, di, rj;
    int z_cur, z_best, z_work, z_next;   // z_next: z_work after the insertion just selected
    unsigned st_work;
    int stagnation, repair_fail, wsel, err;
    unsigned long long wait_ns;       // limit of each spin-wait; one that runs out sets err
    double T, T_init;
    double wd[8], wr[4];
    int sd[8], sr[4], ad[8], ar[4];
    int accepted, improved, new_best, reheats, rejected;
    int z_init;
    // set by the selection when the insertion it applied used no shortcut gap:
    // the next step updates the longest-path table in place of re-walking W.
    // upd from 1 on: c, x_a, y_a, x_b, y_b (old positions, -1 = depot), adjacent, new
    // positions of D_c and P_c, old length, d(x_a,c), d(c,y_a), d(x_b,c),
    // d(c,y_b), d(c,c), p_c, routes of D_c and P_c
    int incr;
    int upd[18];
    unsigned long long steps_incr, steps_full;
    unsigned long long phase_ns[7];   // begin, prep, gaps, matrix, select, end, local search (rank 0 wall time)
    // periodic local search: the pass's candidates, the bottleneck vehicle,
    // whether the last pass moved, moves applied and new bests so far
    int ls_ncand, ls_bott, ls_moved, ls_moves, ls_new_best;
    unsigned long long ls_bound;      // least (makespan, travel) a move of the pass has reached so far
    int imports;                      // best-of-all solutions this replica took at checkpoints
    // Words that the whole team hits with atomics or polls, each group on a
    // cache line of its own: the CTA that selects an insertion while the
    // others wait reads and writes the state above without meeting their
    // traffic.
    alignas(128) unsigned bar_count;
    alignas(128) unsigned bar_gen;
    alignas(128) int work_counter;
    alignas(128) int walks_done;      // CTAs that have finished their shortcut simulations in this greedy step
    alignas(128) int tests_done;      // CTAs that have tested their share of the matrix tiles in this step
    alignas(128) int n_short;
    int sum_load;
    alignas(128) unsigned long long entries, fallback_entries;
    unsigned long long pruned;        // tile entries skipped by the bound (counted in entries too)
    unsigned long long tiles, tiles_pruned;  // matrix tiles run, and those with no customer left to score
};

// 32-bit words of one bit per matrix tile
__host__ __device__ inline int tile_words(int G) {
    return (((G + TR - 1) / TR) * ((G + TC - 1) / TC) + 31) / 32;
}

struct AlnsTeam {
    // instance
    int n, m, R, Q, load_full;
    const int* d32;
    const int* p;          // p[0..n]
    // parameters
    double T0, alpha, reheat, r, w_min;
    int stagnation_limit, tau, sigma1, sigma2, sigma3, q_min, q_max, iterations, repair_mask;
    int destroy_mask;        // bit 0 random, 1 worst, 2 Shaw, 3 cluster, 4 route, 5 critical path
    int ls_pickup, ls_relocate;  // local-search periods in iterations (0 = off)
    int replica, nreplicas, sync_every;   // multi-instance: this team's index, team count, checkpoint period
    unsigned* gbar;          // [2] grid barrier over all teams: count, generation
    const AlnsTeam* sib;     // device array of all teams (siblings' best solutions at checkpoints)
    unsigned long long key;  // RNG stream key
    int mode;                // 0 = search, 1 = one-customer matrix dump, 2 = refine the start solution,
                             // 3 = dump_steps repair steps, then mode 1 on the first customer left
    int refine_rounds;       // mode 2: local-search rounds at most
    int dump_c;
    int dump_steps;          // mode 3
    const int* coords;       // device (n+1) x 2 when distances can be recomputed exactly, else null
    // state and scratch (device)
    AlnsCtl* ctl;
    int *cur_ops, *cur_off, *best_ops, *best_off;
    int *W_ops[2], *W_off[2];
    int *rem;
    int *H, *T, *Ms;
    int *H2, *T2, *Ms2;      // the other copy of each: written by the incremental update, then swapped
    int *S_, *PMINp, *PMAXp, *SMINs, *SMAXs;
    int *spmin, *spmax;      // [LOG][2n]
    int log_levels;
    int *gx, *gy, *gw, *gsb, *gpmin, *gpmax, *gsmin, *gsmax, *groute, *gpos;
    int *rload;              // start load per route
    int *growc, *gcolc;      // [G][RV], [G][CV]: per-gap constants of the matrix tiles
    int4 *vrow, *vcol;       // [q_max][G]: per (customer, gap) row / column vectors of the matrix
    int2 *vadj;              // [q_max][G]: per (customer, gap) adjacent-pair vector (null but for dumps)
    unsigned long long* keys;  // [q_max][G]: per drop gap, best (dz, dt, col)
    unsigned long long* rkeys; // [q_max][32]: per drop vehicle, best (dz, dt, row)
    unsigned long long* gmin;  // [q_max][4]: per vehicle group (v mod 4), best (dz, dt) seen so far
    int4* bands;               // [bands][band_stride]: per 32 gaps and customer, least row x, row w, col x, col w
    int band_stride;
    unsigned* tmask;           // [tile_words(G)]: tiles that passed the phase's first test, in the order they go out
    unsigned char* sc;         // [q_max][G]
    int* slist;                // [q_max * G] entries t * G + g
    int* scix;                 // [q_max][G]: index in slist of a shortcut (customer, gap)
    int* scw;                  // [SC_CAP][scw_stride]: walks of the first SC_CAP shortcut gaps (below)
    int scw_stride;
    int graph_warps;           // warps of a CTA that simulate a shortcut gap at once
    int* scpair;               // [SC_CAP][SC_CAP]: makespan with both stops in two shortcut gaps of one customer
    int* trace;
    int* gains;                // [n+1]: removal gain z(cur) - z(cur - c), worst removal; local search: places of the ops
    double* pw;                // [n+1]: prefix sums of the worst removal's weights r^-6
    int* lscand;               // [n+1]: local-search candidates of the current pass
    int* dump_delta;
    int* dump_travel;
};

// ---------------------------------------------------------------------------
// shared-memory layout of one CTA
// ---------------------------------------------------------------------------
struct Smem {
    int* sW;        // packed W ops [2n + 4]
    int* sWoff;     // [m + 1]
    int* sp;        // p[0..n]
    int* rdy;       // [warps][n + 1] walk buffers; also the matrix batch vectors and select / begin scratch
    int* rowv;      // [TR][RV]
    int* colv;      // [TC][CV]
    int* misc;      // 64 ints
    unsigned long long* counts;  // entries, pruned entries, tiles, pruned tiles of this CTA
    unsigned char* flags;  // [n + 1] removed flags / route-start bits
    int* xy;        // coordinates [n + 1][2] (when staged)
};
constexpr int RV = 16, CV = 12;   // row / col vector widths (ints)
constexpr int CB = 8;             // customers per matrix batch
// A tile's two batches of vectors, (in a dump) the adjacent pairs' and two batches
// of row minima (words), then the list of the customers the tile still has to
// score with their best entries so far (up to ACT_CAP of them; with more
// customers waiting, every tile scores every customer).
constexpr int TILE_WORDS = 2 * CB * 4 * (TC + TR) + 2 * TR + 2 * CB * TR * 2;
constexpr int ACT_CAP = 256;

// Walk buffers (one ready array per warp).  The same words hold a matrix
// tile's batch vectors, row minima and pair list, a shortcut item's
// two walk buffers with its departure and tail arrays, the selection's
// per-customer results (5 words per removed customer) and the removal
// permutation (n words) or a structured destroy's sort keys and per-customer
// facts; no phase needs two of these at once.
__host__ __device__ inline size_t rdy_words(int n) {
    const size_t rw = static_cast<size_t>(((n + 1) + 3) & ~3);
    const size_t walks = static_cast<size_t>(ALNS_WARPS) * rw;
    const size_t fb = 2 * rw + 2 * ((static_cast<size_t>(2 * n) + 3) & ~static_cast<size_t>(3));
    // tile: column and row vectors per customer of a batch, adjacent-pair vectors;
    // the range tables' two buffers (512 + 4n words at most) fit in the larger of this and the walks
    const size_t batch = static_cast<size_t>(TILE_WORDS) + 3 * ACT_CAP;
    const size_t sel = 5 * static_cast<size_t>(n) + 8;
    size_t w = walks > batch ? walks : batch;
    w = w > fb ? w : fb;
    w = w > sel ? w : sel;
    w = w > static_cast<size_t>(n) + 4 ? w : static_cast<size_t>(n) + 4;
    // structured destroy: u64 sort keys (a power of two >= n) and five
    // per-customer arrays
    size_t P = 1;
    while (P < static_cast<size_t>(n)) P <<= 1;
    w = w > 2 * P + 5 * rw ? w : 2 * P + 5 * rw;
    return (w + 3) & ~static_cast<size_t>(3);
}

__host__ __device__ inline size_t alns_smem_words(int n, int m, bool with_coords) {
    size_t w = 0;
    w += ((2 * n + 4) + 3) & ~3;
    w += ((m + 1) + 3) & ~3;
    w += ((n + 1) + 3) & ~3;
    w += rdy_words(n);
    w += TR * RV + TC * CV + 64 + 8;
    w += ((n + 1 + 3) / 4 + 3) & ~3;
    if (with_coords) w += ((2 * (n + 1)) + 3) & ~3;   // coordinates
    return w;
}

__device__ inline Smem carve(int* base, int n, int m) {
    Smem s;
    int* q = base;
    s.sW = q; q += ((2 * n + 4) + 3) & ~3;
    s.sWoff = q; q += ((m + 1) + 3) & ~3;
    s.sp = q; q += ((n + 1) + 3) & ~3;
    s.rdy = q; q += rdy_words(n);
    s.rowv = q; q += TR * RV;
    s.colv = q; q += TC * CV;
    s.misc = q; q += 64;
    s.counts = reinterpret_cast<unsigned long long*>(q); q += 8;
    s.flags = reinterpret_cast<unsigned char*>(q);
    q += ((n + 1 + 3) / 4 + 3) & ~3;
    s.xy = q;
    return s;
}

__device__ __forceinline__ int D(const AlnsTeam& t, int a, int b) { return __ldg(t.d32 + a * (t.n + 1) + b); }

// Same value as D: recomputed exactly (EUC_2D) from shared-memory coordinates
// when the instance has small ones, so no L2 round trip sits on the path.
__device__ __forceinline__ int Dx(const AlnsTeam& t, const Smem& s, int a, int b) {
    if (t.coords) return euc2d_small(s.xy[2 * a], s.xy[2 * a + 1], s.xy[2 * b], s.xy[2 * b + 1]);
    return __ldg(t.d32 + a * (t.n + 1) + b);
}

// ---------------------------------------------------------------------------
// team barrier: all CTAs of the team; bounded (about 2 s).  Arrivals are one
// counter's acquire-release additions and the release is an addition to the
// generation word that the others poll, whose top bit says that the run has failed
// (ctl->err says why): a step meets three barriers, and full fences, pauses between
// polls and a read of err behind each made a step 2.4 us longer at n = 1000 (63.0
// instead of 60.6 us, 456 CTAs) and 0.8 us at n = 120 (32 CTAs).
// ---------------------------------------------------------------------------
constexpr unsigned GEN_FAILED = 0x80000000u;

__device__ __forceinline__ unsigned add_acq_rel(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
// Whatever fails in a run goes through here: the barriers read the flag, not err.
__device__ __forceinline__ void fail_run(AlnsCtl* ctl, int why) {
    atomicExch(&ctl->err, why);
    atomicOr(&ctl->bar_gen, GEN_FAILED);
}

// thread 0: this CTA has arrived (its threads' writes before the block barrier are visible); true for the last
__device__ __forceinline__ bool arrive_last(AlnsCtl* ctl, int team_blocks) {
    return add_acq_rel(&ctl->bar_count, 1u) + 1u == static_cast<unsigned>(team_blocks);
}
// thread 0 of the last CTA: the others go on; false if the run has failed
__device__ __forceinline__ bool release_team(AlnsCtl* ctl, unsigned gen) {
    ctl->bar_count = 0u;
    return add_acq_rel(&ctl->bar_gen, 1u) == gen;
}
// one thread: until a counter of the step has come to want (false: the wait ran out).
// The two waits are out of line: inlined, their registers cost the tiles more spills
// (32 replicas at n = 1000: 632 ms instead of 623).
[[nodiscard]] __device__ __noinline__ bool await_count(AlnsCtl* ctl, const int* count, int want) {
    const uint64_t t0 = global_ns();
    const unsigned long long limit = ctl->wait_ns;
    int v;
    for (;;) {
        asm volatile("ld.relaxed.gpu.s32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
        if (v >= want) break;
        if (global_ns() - t0 > limit) {
            fail_run(ctl, DEV_TIMEOUT_BARRIER);
            return false;
        }
    }
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    return true;
}
// thread 0 of the others: until the last has come
__device__ __noinline__ bool await_release(AlnsCtl* ctl, unsigned gen) {
    const uint64_t t0 = global_ns();
    const unsigned long long limit = ctl->wait_ns;
    unsigned v;
    for (;;) {
        asm volatile("ld.relaxed.gpu.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->bar_gen) : "memory");
        if (v != gen) break;
        if (global_ns() - t0 > limit) {
            fail_run(ctl, DEV_TIMEOUT_BARRIER);
            return false;
        }
    }
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    return v == gen + 1u;
}

__device__ bool team_barrier(AlnsCtl* ctl, int team_blocks, unsigned& gen) {
    __syncthreads();
    if (team_blocks == 1) return *reinterpret_cast<volatile int*>(&ctl->err) == 0;
    bool failed = false;
    if (threadIdx.x == 0) failed = !(arrive_last(ctl, team_blocks) ? release_team(ctl, gen) : await_release(ctl, gen));
    gen += 1u;
    return !__syncthreads_or(failed);
}

// The same barrier in two halves, so a CTA can do work that no one waits on
// at the barrier (the shortcut simulations) between arriving and waiting.
__device__ void team_arrive(AlnsCtl* ctl, int team_blocks, unsigned gen) {
    __syncthreads();
    if (team_blocks > 1 && threadIdx.x == 0 && arrive_last(ctl, team_blocks)) release_team(ctl, gen);
}

__device__ bool team_wait(AlnsCtl* ctl, int team_blocks, unsigned& gen) {
    __syncthreads();
    if (team_blocks == 1) return *reinterpret_cast<volatile int*>(&ctl->err) == 0;
    const bool failed = threadIdx.x == 0 && !await_release(ctl, gen);
    gen += 1u;
    return !__syncthreads_or(failed);
}

// ---------------------------------------------------------------------------
// stage W into shared memory: packed (travel-in << 12 | op)
// ---------------------------------------------------------------------------
__device__ void stage_ops(const AlnsTeam& t, const Smem& s, const int* W, const int* Wo) {
    const int m = t.m;
    for (int i = threadIdx.x; i <= m; i += blockDim.x) s.sWoff[i] = Wo[i];
    __syncthreads();
    const int N = s.sWoff[m];
    // every load of a thread in flight together: its ops and the ops before them
    constexpr int SU = 8;
    for (int k0 = 0; k0 < N; k0 += SU * ALNS_THREADS) {
        int o[SU], pr[SU];
#pragma unroll
        for (int u = 0; u < SU; ++u) {
            const int k = k0 + u * ALNS_THREADS + static_cast<int>(threadIdx.x);
            o[u] = k < N ? W[k] : 0;
            pr[u] = (k < N && k > 0) ? W[k - 1] : 0;
        }
#pragma unroll
        for (int u = 0; u < SU; ++u) {
            const int k = k0 + u * ALNS_THREADS + static_cast<int>(threadIdx.x);
            if (k >= N) break;
            // the op before k on its route: none if k starts a route
            int lo = 0, hi = m;                // find route r with off[r] <= k < off[r+1]
            while (hi - lo > 1) {
                int mid = (lo + hi) >> 1;
                if (s.sWoff[mid] <= k) lo = mid; else hi = mid;
            }
            const int prev = (k == s.sWoff[lo]) ? 0 : (pr[u] >> 1);
            s.sW[k] = (Dx(t, s, prev, o[u] >> 1) << PACK_SHIFT) | o[u];
        }
    }
    __syncthreads();
}

__device__ void stage_W(const AlnsTeam& t, const Smem& s) {
    stage_ops(t, s, t.W_ops[t.ctl->wsel], t.W_off[t.ctl->wsel]);
}

// ---------------------------------------------------------------------------
// walks (one warp; lane r walks route r; m <= 32)
// ---------------------------------------------------------------------------
// From the depot: makespan and status.
__device__ void walk_depot(const AlnsTeam& t, const Smem& s, int* rdy_, int* z_out, unsigned* st_out) {
    const int* __restrict__ sW = s.sW;
    const int* __restrict__ spp = s.sp;

    const int lane = threadIdx.x & 31, m = t.m, n = t.n;
    volatile int* rdy = rdy_;
    for (int c = lane; c <= n; c += 32) rdy[c] = UNRES;
    __syncwarp();
    const bool mine = lane < m;
    int pos = mine ? s.sWoff[lane] : 0, end = mine ? s.sWoff[lane + 1] : 0;
    const int start = pos;
    int dep = 0, last = 0, sv = 0, smin = 0, smax = 0;
    bool walking = mine && pos < end, cyc = false;
    // up to two ops per lane per step, both reads up front (see walk_source)
    bool alive = __any_sync(FULL_MASK, walking);
    while (alive) {
        const bool can1 = walking, can2 = walking && pos + 1 < end;
        const int w1 = can1 ? sW[pos] : 0, w2 = can2 ? sW[pos + 1] : 0;
        const int c1 = (w1 & PACK_MASK) >> 1, c2 = (w2 & PACK_MASK) >> 1;
        const bool k1 = (w1 & 1) != 0, k2 = (w2 & 1) != 0;
        const int r1 = (can1 && k1) ? rdy[c1] : 0;
        const int r2 = (can2 && k2) ? rdy[c2] : 0;
        const bool go1 = can1 && (!k1 || r1 != UNRES);
        const bool go2 = go1 && can2 && (!k2 || r2 != UNRES);
        const int a1 = dep + (w1 >> PACK_SHIFT);
        const int d1 = k1 ? max(a1, r1) : a1;
        const int a2 = d1 + (w2 >> PACK_SHIFT);
        const int d2 = k2 ? max(a2, r2) : a2;
        if (go1) {
            if (!k1) rdy[c1] = a1 + spp[c1];
            sv += k1 ? 1 : -1;
            smin = min(smin, sv);
            smax = max(smax, sv);
            dep = d1;
            last = c1;
        }
        if (go2) {
            if (!k2) rdy[c2] = a2 + spp[c2];
            sv += k2 ? 1 : -1;
            smin = min(smin, sv);
            smax = max(smax, sv);
            dep = d2;
            last = c2;
        }
        pos += (go1 ? 1 : 0) + (go2 ? 1 : 0);
        const bool more = pos < end;
        const unsigned prog = __ballot_sync(FULL_MASK, go1);
        if (walking && more && prog == 0u) cyc = true;
        walking = walking && more && prog != 0u;
        __syncwarp();
        alive = prog != 0u && __any_sync(FULL_MASK, walking);
    }
    if (cyc)
        for (; pos < end; ++pos) {
            const int o = sW[pos] & PACK_MASK;
            if (o & 1) { ++sv; smax = max(smax, sv); } else { --sv; smin = min(smin, sv); }
        }
    int ret = (mine && !cyc && end > start) ? dep + Dx(t, s, last, 0) : 0;
    int load = 0;
    bool bad = false;
    if (mine) {
        if (t.load_full) { bad = smin < -t.Q || smax > 0; load = t.Q; }
        else { bad = -smin + smax > t.Q; load = -smin; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        ret = max(ret, __shfl_xor_sync(FULL_MASK, ret, o));
        load += __shfl_xor_sync(FULL_MASK, load, o);
    }
    const unsigned anycyc = __ballot_sync(FULL_MASK, cyc), anybad = __ballot_sync(FULL_MASK, bad);
    unsigned st = (anycyc ? VRPRPD_CYCLE : 0u) | (anybad ? VRPRPD_VEH_CAP : 0u) | (load > t.R ? VRPRPD_POOL : 0u);
    if (anycyc) ret = 0x7fffffff;
    *z_out = ret;
    *st_out = st;
}

// What one stop of a walk needs from shared memory, by shared-window addresses.
// A round is a chain of dependent instructions, and through the generic pointers
// of Smem the compiler reads those pointers again after every store of a ready
// time: 0.19 us a round, and 0.08 us so (one warp, n = 1000, m = 20).
struct WalkMem {
    unsigned w, p, r;                          // packed ops, processing times, ready times (or tails)
    __device__ __forceinline__ WalkMem(const Smem& s, const int* rdy) : w(smem_u32(s.sW)), p(smem_u32(s.sp)), r(smem_u32(rdy)) {}
    static __device__ __forceinline__ int ld(unsigned a) {
        int v;
        asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a));
        return v;
    }
    static __device__ __forceinline__ void st(unsigned a, int v) { asm volatile("st.shared.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
    __device__ __forceinline__ int op(int pos) const { return ld(w + 4u * static_cast<unsigned>(pos)); }
    // byte offset of the customer of packed op x in a per-customer array
    static __device__ __forceinline__ unsigned at(int x) { return static_cast<unsigned>(x & (PACK_MASK & ~1)) << 1; }
};
constexpr int FREE = INT32_MIN + 1;            // "ready time" of a stop that waits for nothing
// Rounds between two looks at whether any lane still moves: the vote is as long
// as a shared-memory load, and rounds in which no lane moves change nothing.
constexpr int WALK_ROUNDS = 4;

// One warp: departures of the staged (acyclic) solution into H; its makespan.
__device__ int walk_heads(const AlnsTeam& t, const Smem& s, int* rdy_, int* H) {
    const int lane = threadIdx.x & 31, n = t.n;
    for (int c = lane; c <= n; c += 32) rdy_[c] = UNRES;
    __syncwarp();
    const WalkMem M(s, rdy_);
    int pos = lane < t.m ? s.sWoff[lane] : 0;
    const int start = pos, end = lane < t.m ? s.sWoff[lane + 1] : 0;
    int dep = 0, last = 0, x = pos < end ? M.op(pos) : 0;
    bool moved;
    do {
        moved = false;
#pragma unroll
        for (int k = 0; k < WALK_ROUNDS; ++k) {
            const unsigned ca = M.at(x);
            const bool pick = (x & 1) != 0;
            const int rv = M.ld(M.r + ca), p = M.ld(M.p + ca), nx = M.op(pos + 1);
            const int r = pick ? rv : FREE;
            const bool go = pos < end && r != UNRES;
            const int d = max(dep + (x >> PACK_SHIFT), r);
            if (go && !pick) M.st(M.r + ca, d + p);
            if (go) H[pos] = d;
            dep = go ? d : dep;
            last = go ? x : last;
            pos += go ? 1 : 0;
            x = go ? (pos < end ? nx : 0) : x;
            moved |= go;
            __syncwarp();
        }
    } while (__any_sync(FULL_MASK, moved));
    int ret = end > start ? dep + Dx(t, s, (last & PACK_MASK) >> 1, 0) : 0;
    for (int o = 16; o > 0; o >>= 1) ret = max(ret, __shfl_xor_sync(FULL_MASK, ret, o));
    return ret;
}

// From op u: row u of LP (NEG where unreachable) and T(u).  One op per lane and
// round; ready times have one writer (the dropping lane) and are read volatile,
// so a pickup sees "unresolved" (and retries) or the final value, and the
// __syncwarp closing each round makes every write of a round visible in the
// next: rounds in which no lane moves end the walk, and a route not ended then
// means a precedence cycle.  (Two ops a round, with every choice written out,
// took more instructions: the preparation of a step 27.8 us at n=1000, 7 of 36
// steps full; one op a round takes 24 us, bound by the row's scattered stores;
// 9.8 and 8.3 us at n=120.)
__device__ void walk_source(const AlnsTeam& t, const Smem& s, int* rdy_, int u, int N) {
    const int lane = threadIdx.x & 31, m = t.m, n = t.n;
    for (int c = lane; c <= n; c += 32) rdy_[c] = UNRES;
    __syncwarp();
    const WalkMem M(s, rdy_);
    int pos = lane < m ? s.sWoff[lane] : 0;
    const int end = lane < m ? s.sWoff[lane + 1] : 0;
    int val = NEG, last = 0, x = pos < end ? M.op(pos) : 0;
    int* row = t.Ms + static_cast<long long>(u) * N;
    bool moved;
    do {
        moved = false;
#pragma unroll
        for (int k = 0; k < WALK_ROUNDS; ++k) {
            const unsigned ca = M.at(x);
            const bool pick = (x & 1) != 0, at = pos == u;
            const int rv = M.ld(M.r + ca), p = M.ld(M.p + ca), nx = M.op(pos + 1);
            const int r = pick && !at ? rv : NEG;  // (the source's own time is 0 whatever it waits for)
            const bool go = pos < end && r != UNRES;
            const int via = max(val == NEG ? NEG : val + (x >> PACK_SHIFT), r);
            const int v = at ? 0 : via;
            if (go && !pick) M.st(M.r + ca, v == NEG ? NEG : v + p);
            if (go) row[pos] = v;
            val = go ? v : val;
            last = go ? x : last;
            pos += go ? 1 : 0;
            x = go ? (pos < end ? nx : 0) : x;
            moved |= go;
            __syncwarp();
        }
    } while (__any_sync(FULL_MASK, moved));
    if (pos < end) fail_run(t.ctl, DEV_BAD_STATE);
    int tail = (lane < m && val != NEG) ? val + Dx(t, s, (last & PACK_MASK) >> 1, 0) : NEG;
    for (int o = 16; o > 0; o >>= 1) tail = max(tail, __shfl_xor_sync(FULL_MASK, tail, o));
    if (lane == 0) t.T[u] = tail;
}

// A route of the staged W with up to two new stops in it, as one sequence of
// packed (travel-in << PACK_SHIFT | op) words: the new stops sit at places q0 < q1
// (SEQ_NONE: not there), and a stop behind one has its leg from there.  A lane's
// walk asks for the word of each place in turn, so the walks themselves are those
// of W, one stop a round.
constexpr int SEQ_NONE = 1 << 29;
struct Seq {
    int base, len, q0 = SEQ_NONE, q1 = SEQ_NONE;
    int x0 = 0, y0 = 0, x1 = 0, y1 = 0;        // words of the new stops, and of the stops behind them
    __device__ __forceinline__ int pos(int q) const { return base + q - (q > q0 ? 1 : 0) - (q > q1 ? 1 : 0); }
    __device__ __forceinline__ int at(const WalkMem& M, int q) const {
        int x = M.op(pos(max(q, 0)));
        x = q >= 0 && q < len ? x : 0;
        if (q == q0 + 1) x = y0;
        if (q == q0) x = x0;
        if (q == q1) x = x1;
        if (q == q1 + 1) x = y1;
        return x;
    }
};

// lane's route with stop o1 at gap (a, i) and o2 at gap (b, j) (a < 0 or b < 0
// leaves one out; o1 goes first when both share a gap)
__device__ __forceinline__ Seq make_seq(const AlnsTeam& t, const Smem& s, int a, int i, int o1, int b, int j, int o2) {
    const int lane = threadIdx.x & 31;
    Seq u;
    u.base = lane < t.m ? s.sWoff[lane] : 0;
    const int L = lane < t.m ? s.sWoff[lane + 1] - u.base : 0;
    u.len = L;
    const bool va = lane == a, vb = lane == b;
    if (va || vb) {
        const int g0 = va ? i : j, v0 = va ? o1 : o2;
        auto word = [&](int k) { return k < L ? s.sW[u.base + k] & PACK_MASK : 0; };
        auto leg_in = [&](int op, int k) {     // op with its leg from W position k (the depot below 0)
            return Dx(t, s, k >= 0 ? word(k) >> 1 : 0, op >> 1) << PACK_SHIFT | op;
        };
        auto behind = [&](int op, int k) { return Dx(t, s, op >> 1, word(k) >> 1) << PACK_SHIFT | word(k); };
        u.q0 = g0;
        u.x0 = leg_in(v0, g0 - 1);
        u.y0 = behind(v0, g0);
        u.len = L + 1;
        if (va && vb) {
            u.q1 = j + 1;
            u.x1 = j == i ? Dx(t, s, o1 >> 1, o2 >> 1) << PACK_SHIFT | o2 : leg_in(o2, j - 1);
            u.y1 = behind(o2, j);
            u.len = L + 2;
        }
    }
    return u;
}

// Forward simulation of W plus up to two stops, V1 (op code o1) at gap (a, i)
// and V2 (op code o2) at gap (b, j); a < 0 or b < 0 leaves one out, and V1
// goes first when both share a gap.  Returns the makespan (INT32_MAX on a
// precedence cycle); with Hb non-null the departure of every W position goes
// to Hb[pos] and V1's to *hv.  One stop per lane and round, the next one's word
// read ahead: the 200 rounds of a solution with n = 1000, m = 20 take 15 us, and
// 43 us with two stops a round and every choice between them written out.
__device__ int walk_fwd(const AlnsTeam& t, const Smem& s, int* rdy_, int a, int i, int o1, int b, int j, int o2,
                        int* Hb, int* hv) {
    const WalkMem M(s, rdy_);
    const Seq u = make_seq(t, s, a, i, o1, b, j, o2);
    int q = 0, dep = 0, last = 0, h = 0, x = u.at(M, 0);
    bool moved;
    do {
        moved = false;
#pragma unroll
        for (int k = 0; k < WALK_ROUNDS; ++k) {
            const unsigned ca = M.at(x);
            const bool pick = (x & 1) != 0;
            const int rv = M.ld(M.r + ca), p = M.ld(M.p + ca), nx = u.at(M, q + 1);
            const int r = pick ? rv : FREE;
            const bool go = q < u.len && r != UNRES;
            const int d = max(dep + (x >> PACK_SHIFT), r);
            if (go && !pick) M.st(M.r + ca, d + p);
            if (Hb != nullptr && go && q != u.q0 && q != u.q1) Hb[u.pos(q)] = d;
            h = go && q == u.q0 ? d : h;
            dep = go ? d : dep;
            last = go ? x : last;
            q += go ? 1 : 0;
            x = go ? nx : x;
            moved |= go;
            __syncwarp();
        }
    } while (__any_sync(FULL_MASK, moved));
    if (Hb != nullptr && static_cast<int>(threadIdx.x & 31) == a) *hv = h;
    int ret = u.len > 0 ? dep + Dx(t, s, (last & PACK_MASK) >> 1, 0) : 0;
    for (int o = 16; o > 0; o >>= 1) ret = max(ret, __shfl_xor_sync(FULL_MASK, ret, o));
    return __any_sync(FULL_MASK, q < u.len) ? 0x7fffffff : ret;
}

// Full simulation of W + D_c at gap (a,i) + P_c at gap (b,j): makespan or
// INT32_MAX on a precedence cycle.
__device__ int walk_insert(const AlnsTeam& t, const Smem& s, int* rdy, int c, int a, int i, int b, int j) {
    const int lane = threadIdx.x & 31, n = t.n;
    for (int q = lane; q <= n; q += 32) rdy[q] = UNRES;
    __syncwarp();
    return walk_fwd(t, s, rdy, a, i, 2 * c, b, j, 2 * c + 1, nullptr, nullptr);
}

// W plus one stop V (op code ov) at gap (a, i), forward: the departure time of
// every W position into Hb[pos] and of V into *hv; returns the makespan
// (INT32_MAX on a precedence cycle).  A pickup V without its drop leaves at
// arrival (its ready time is set to 0): the drop's edge comes with the second
// stop, not here.
__device__ int walk_fwd1(const AlnsTeam& t, const Smem& s, int* rdy, int ov, int a, int i, int* Hb, int* hv) {
    const int lane = threadIdx.x & 31, n = t.n;
    for (int q = lane; q <= n; q += 32) rdy[q] = UNRES;
    __syncwarp();
    if (lane == 0 && (ov & 1)) rdy[ov >> 1] = 0;
    __syncwarp();
    return walk_fwd(t, s, rdy, a, i, ov, -1, 0, 0, Hb, hv);
}

// The same graph backward: the tail of every W position (longest path from its
// departure to the end of the schedule, return leg included) into Tb[pos] and
// V's into *tv.  A drop's tail also takes p plus its pickup's tail; V has no
// partner in this graph.  tp: per-customer pickup tails (n + 1 words).
__device__ void walk_bwd1(const AlnsTeam& t, const Smem& s, int* tp_, int ov, int a, int i, int* Tb, int* tv) {
    const int lane = threadIdx.x & 31, n = t.n;
    for (int c = lane; c <= n; c += 32) tp_[c] = UNRES;
    __syncwarp();
    const WalkMem M(s, tp_);
    const Seq u = make_seq(t, s, a, i, ov, -1, 0, 0);
    int q = u.len - 1, x = u.at(M, q), acc = 0, tl = 0;
    int leg = q >= 0 ? Dx(t, s, (x & PACK_MASK) >> 1, 0) : 0;
    bool moved;
    do {
        moved = false;
#pragma unroll
        for (int k = 0; k < WALK_ROUNDS; ++k) {
            const unsigned ca = M.at(x);
            const bool virt = q == u.q0, pick = (x & 1) != 0, waits = !pick && !virt;
            const int rv = M.ld(M.r + ca), p = M.ld(M.p + ca), nx = u.at(M, q - 1);
            const int r = waits ? rv : FREE;
            const bool go = q >= 0 && r != UNRES;
            const int after = acc + leg, d = waits ? max(after, p + r) : after;
            if (go && pick && !virt) M.st(M.r + ca, d);
            if (go && !virt) Tb[u.pos(q)] = d;
            tl = go && virt ? d : tl;
            acc = go ? d : acc;
            leg = go ? x >> PACK_SHIFT : leg;
            q -= go ? 1 : 0;
            x = go ? nx : x;
            moved |= go;
            __syncwarp();
        }
    } while (__any_sync(FULL_MASK, moved));
    if (lane == a) *tv = tl;
    if (q >= 0) fail_run(t.ctl, DEV_BAD_STATE);
}

// ---------------------------------------------------------------------------
// capacity helpers (Eqs. 13-18 with the minimal or the full start load)
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool cap_ok(const AlnsTeam& t, int mn, int mx, int& load) {
    if (t.load_full) { load = t.Q; return mn >= -t.Q && mx <= 0; }
    mn = min(mn, 0);
    mx = max(mx, 0);
    load = -mn;
    return load + mx <= t.Q;
}

__device__ __forceinline__ int range_min(const AlnsTeam& t, int lo, int hi, int N) {
    const int len = hi - lo + 1;
    const int l = 31 - __clz(len);
    return min(t.spmin[l * N + lo], t.spmin[l * N + hi - (1 << l) + 1]);
}
__device__ __forceinline__ int range_max(const AlnsTeam& t, int lo, int hi, int N) {
    const int len = hi - lo + 1;
    const int l = 31 - __clz(len);
    return max(t.spmax[l * N + lo], t.spmax[l * N + hi - (1 << l) + 1]);
}

__device__ __forceinline__ unsigned long long pack_key(int dz, int dt, int col) {
    return (static_cast<unsigned long long>(static_cast<unsigned>(dz) ^ 0x80000000u) << 32) |
           (static_cast<unsigned long long>(static_cast<unsigned>(dt + (1 << 19)) & 0xFFFFFu) << 12) |
           static_cast<unsigned long long>(col & 0xFFF);
}

// Capacity + pool of one entry from the per-gap arrays (global memory).
// Returns false when infeasible.
__device__ bool entry_capacity(const AlnsTeam& t, int row, int col, int N) {
    const int a = t.groute[row], i = t.gpos[row], b = t.groute[col], j = t.gpos[col];
    int la = 0, lb = 0;
    const int sumL = t.ctl->sum_load;
    if (a != b) {
        const int mnA = min(min(t.gpmin[row], t.gsb[row] - 1), t.gsmin[row] - 1);
        const int mxA = max(t.gpmax[row], t.gsmax[row] - 1);
        const int mnB = min(t.gpmin[col], t.gsmin[col] + 1);
        const int mxB = max(max(t.gpmax[col], t.gsb[col] + 1), t.gsmax[col] + 1);
        if (!cap_ok(t, mnA, mxA, la) || !cap_ok(t, mnB, mxB, lb)) return false;
        return sumL - t.rload[a] - t.rload[b] + la + lb <= t.R;
    }
    if (j == i) {
        const int mn = min(min(t.gpmin[row], t.gsb[row] - 1), t.gsmin[row]);
        const int mx = max(t.gpmax[row], t.gsmax[row]);
        if (!cap_ok(t, mn, mx, la)) return false;
        return sumL - t.rload[a] + la <= t.R;
    }
    const int lo = t.gy[row], hi = t.gx[col];   // stock prefixes between the two gaps
    const int mn = min(min(min(t.gpmin[row], t.gsb[row] - 1), range_min(t, lo, hi, N) - 1), t.gsmin[col]);
    const int mx = max(max(max(t.gpmax[row], range_max(t, lo, hi, N) - 1), t.S_[hi]), t.gsmax[col]);
    if (!cap_ok(t, mn, mx, la)) return false;
    return sumL - t.rload[a] + la <= t.R;
}

__device__ __forceinline__ int travel_delta(const AlnsTeam& t, const Smem& s, int c, int row, int col) {
    auto locx = [&](int g) { return t.gx[g] >= 0 ? (s.sW[t.gx[g]] & PACK_MASK) >> 1 : 0; };
    auto locy = [&](int g) { return t.gy[g] >= 0 ? (s.sW[t.gy[g]] & PACK_MASK) >> 1 : 0; };
    const int xr = locx(row), yr = locy(row);
    if (t.groute[row] == t.groute[col] && t.gpos[row] == t.gpos[col])
        return Dx(t, s, xr, c) + Dx(t, s, c, c) + Dx(t, s, c, yr) - t.gw[row];
    const int xc = locx(col), yc = locy(col);
    return (Dx(t, s, xr, c) + Dx(t, s, c, yr) - t.gw[row]) + (Dx(t, s, xc, c) + Dx(t, s, c, yc) - t.gw[col]);
}

// ---------------------------------------------------------------------------
// phases
// ---------------------------------------------------------------------------
// Stock prefix arrays of route r from the staged W (one warp): what the walk
// from the depot writes, S_ (stock after each op), its running min / max with
// the start at 0, and the suffix min / max of S_ within the route; the route's
// start load goes to rload[r] and is added to sum_load.
__device__ void scan_route_stock(const AlnsTeam& t, const Smem& s, int r) {
    const int lane = threadIdx.x & 31;
    const int st = s.sWoff[r], en = s.sWoff[r + 1];
    int carry = 0, cmin = 0, cmax = 0;
    for (int base = st; base < en; base += 32) {
        const int k = base + lane;
        const bool in = k < en;
        int v = in ? (((s.sW[k] & PACK_MASK) & 1) ? 1 : -1) : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL_MASK, v, o);
            if (lane >= o) v += y;
        }
        const int sv = carry + v;
        int mn = in ? sv : INT32_MAX, mx = in ? sv : INT32_MIN;
        for (int o = 1; o < 32; o <<= 1) {
            const int y1 = __shfl_up_sync(FULL_MASK, mn, o), y2 = __shfl_up_sync(FULL_MASK, mx, o);
            if (lane >= o) { mn = min(mn, y1); mx = max(mx, y2); }
        }
        mn = min(mn, cmin);
        mx = max(mx, cmax);
        if (in) { t.S_[k] = sv; t.PMINp[k] = mn; t.PMAXp[k] = mx; }
        carry = __shfl_sync(FULL_MASK, sv, 31);
        cmin = __shfl_sync(FULL_MASK, mn, 31);
        cmax = __shfl_sync(FULL_MASK, mx, 31);
    }
    __syncwarp();
    int smn = INT32_MAX, smx = INT32_MIN;
    for (int top = en - 1; top >= st; top -= 32) {
        const int k = top - lane;
        const bool in = k >= st;
        const int sv = in ? t.S_[k] : 0;
        int mn = in ? sv : INT32_MAX, mx = in ? sv : INT32_MIN;
        for (int o = 1; o < 32; o <<= 1) {
            const int y1 = __shfl_up_sync(FULL_MASK, mn, o), y2 = __shfl_up_sync(FULL_MASK, mx, o);
            if (lane >= o) { mn = min(mn, y1); mx = max(mx, y2); }
        }
        mn = min(mn, smn);
        mx = max(mx, smx);
        if (in) { t.SMINs[k] = mn; t.SMAXs[k] = mx; }
        smn = __shfl_sync(FULL_MASK, mn, 31);
        smx = __shfl_sync(FULL_MASK, mx, 31);
    }
    if (lane == 0) {
        const int load = t.load_full ? t.Q : -cmin;
        t.rload[r] = load;
        atomicAdd(&t.ctl->sum_load, load);
    }
}

// After inserting D_c into gap (x_a, y_a) and P_c into gap (x_b, y_b), neither
// a shortcut for c, every path of the old graph survives with at least its old
// length, and a new path meets D_c, or P_c, or both.  With LP the old table,
//     A(u) = LP(u,x_a) + d(x_a,c)                    (reaching D_c)
//     E(u) = max(LP(u,x_b), A(u) + d(c,y_a) + LP(y_a,x_b)) + d(x_b,c)
//     B(v) = d(c,y_b) + LP(y_b,v)                    (leaving P_c)
//     D(v) = max(d(c,y_a) + max(LP(y_a,v), LP(y_a,x_b) + d(x_b,c) + B(v)), p_c + B(v))
//     LP'(u,v) = max(LP(u,v), A(u) + D(v), E(u) + B(v)),
// and the same with the depot's start as u (heads H) and its end as v (tails
// T).  When both stops share one gap, D_c is P_c's only predecessor:
// D(v) = max(d(c,c), p_c) + B(v) and the E term drops.  Unreachable is NEG;
// sums stay clear of overflow by clamping NEG to -2^28 first and mapping every
// negative result back to NEG.  Old positions move right by the new stops
// before them; the new table has stride N + 2 and goes to the second buffers.
constexpr int NEGC = -(1 << 28);

__device__ void phase_update(const AlnsTeam& t, const Smem& s, int rank, int team_blocks) {
    AlnsCtl* ctl = t.ctl;
    const int* up = ctl->upd;
    const int xa = up[2], ya = up[3], xb = up[4], yb = up[5], adj = up[6], Pd = up[7], Pp = up[8];
    const int No = up[9], Nn = No + 2;
    const int dxa = up[10], dya = up[11], dxb = up[12], dyb = up[13], dcc = up[14], pc = up[15];
    const int* Mo = t.Ms;
    int* Mn = t.Ms2;
    auto cl = [](int x) { return x == NEG ? NEGC : x; };
    auto fix = [](int x) { return x < 0 ? NEG : x; };
    const int mcp = max(dcc, pc);
    const int Lyx = (!adj && ya >= 0 && xb >= 0) ? cl(Mo[static_cast<long long>(ya) * No + xb]) : NEGC;
    const int hA = (xa >= 0 ? t.H[xa] : 0) + dxa;
    const int hE = adj ? NEGC : max(xb >= 0 ? t.H[xb] : 0, hA + dya + Lyx) + dxb;
    const int tB = dyb + (yb >= 0 ? t.T[yb] : 0);
    const int tD = adj ? mcp + tB : max(dya + (ya >= 0 ? max(t.T[ya], Lyx + dxb + tB) : 0), pc + tB);
    const int LPdp = adj ? mcp : max(pc, Lyx + dya + dxb);
    if (rank == 0 && threadIdx.x == 0) {
        const int z = ctl->z_work;
        ctl->z_work = max(max(z, hA + tD), hE + tB);
    }
    // new position -> 0 (old op, index in *old), 1 (D_c), 2 (P_c)
    auto kind_of = [&](int k, int* old) {
        if (k == Pd) return 1;
        if (k == Pp) return 2;
        *old = k - (k > Pd ? 1 : 0) - (k > Pp ? 1 : 0);
        return 0;
    };
    constexpr int UR = 16;                     // rows per tile; columns = threads
    int* rowA = s.rowv;                        // [UR] A, E, kind, old index
    int* rowE = rowA + UR;
    int* rowK = rowE + UR;
    int* rowO = rowK + UR;
    const int ntr = (Nn + UR - 1) / UR, ntc = (Nn + ALNS_THREADS - 1) / ALNS_THREADS;
    for (int tile = rank; tile < ntr * ntc; tile += team_blocks) {
        const int r0 = (tile / ntc) * UR, c0 = (tile % ntc) * ALNS_THREADS;
        __syncthreads();                       // the previous tile is done with the row values
        if (threadIdx.x < UR) {
            const int k = r0 + threadIdx.x;
            int kind = 3, u = 0, A = NEGC, E = NEGC;
            if (k < Nn) {
                kind = kind_of(k, &u);
                if (kind == 0) {
                    const long long ro = static_cast<long long>(u) * No;
                    A = xa >= 0 ? cl(Mo[ro + xa]) + dxa : NEGC;
                    E = (adj || xb < 0) ? NEGC : max(cl(Mo[ro + xb]), A + dya + Lyx) + dxb;
                }
                if (c0 == 0)
                    t.T2[k] = kind == 0 ? max(t.T[u], max(A + tD, E + tB)) : (kind == 1 ? tD : tB);
            }
            rowA[threadIdx.x] = A;
            rowE[threadIdx.x] = E;
            rowK[threadIdx.x] = kind;
            rowO[threadIdx.x] = u;
        }
        __syncthreads();
        const int k = c0 + threadIdx.x;
        if (k >= Nn) continue;
        int v = 0;
        const int ck = kind_of(k, &v);
        int B = NEGC, D = NEGC;
        if (ck == 0) {
            B = yb >= 0 ? dyb + cl(Mo[static_cast<long long>(yb) * No + v]) : NEGC;
            D = adj ? mcp + B
                    : max(ya >= 0 ? dya + max(cl(Mo[static_cast<long long>(ya) * No + v]), Lyx + dxb + B) : NEGC,
                          pc + B);
        }
        if (r0 == 0)
            t.H2[k] = ck == 0 ? max(t.H[v], max(hA + D, hE + B)) : (ck == 1 ? hA : (adj ? hA + mcp : max(hE, hA + pc)));
        // all old values of this column first: the stores below may not be
        // ordered ahead of these loads
        int old[UR];
#pragma unroll
        for (int rr = 0; rr < UR; ++rr)
            old[rr] = (ck == 0 && rowK[rr] == 0) ? Mo[static_cast<long long>(rowO[rr]) * No + v] : NEG;
#pragma unroll
        for (int rr = 0; rr < UR; ++rr) {
            const int rk = rowK[rr];
            if (rk == 3) break;
            const int A = rowA[rr], E = rowE[rr];
            int val;
            if (rk == 0) {
                if (ck == 0) val = fix(max(old[rr], max(A + D, E + B)));
                else if (ck == 1) val = fix(A);
                else val = fix(adj ? A + mcp : max(E, A + pc));
            } else if (rk == 1) {
                val = ck == 0 ? fix(D) : (ck == 1 ? 0 : LPdp);
            } else {
                val = ck == 0 ? fix(B) : (ck == 1 ? NEG : 0);
            }
            Mn[static_cast<long long>(r0 + rr) * Nn + k] = val;
        }
    }
}

// The staged solution without customer cx: makespan (INT32_MAX on a cycle).
// The stop after a skipped one is reached from the last kept stop (or the
// depot); a route left empty returns at 0.  One stop per lane per step.
__device__ int walk_skip(const AlnsTeam& t, const Smem& s, int* rdy_, int cx) {
    const int lane = threadIdx.x & 31, n = t.n;
    for (int c = lane; c <= n; c += 32) rdy_[c] = c == cx ? FREE : UNRES;
    __syncwarp();
    const WalkMem M(s, rdy_);
    int pos = lane < t.m ? s.sWoff[lane] : 0;
    const int end = lane < t.m ? s.sWoff[lane + 1] : 0;
    int dep = 0, last = 0, x = pos < end ? M.op(pos) : 0;
    bool skipped = false;                      // the stop before is left out: the leg starts at last
    bool moved;
    do {
        moved = false;
#pragma unroll
        for (int k = 0; k < WALK_ROUNDS; ++k) {
            const unsigned ca = M.at(x);
            const int c = static_cast<int>(ca >> 2);
            const bool pick = (x & 1) != 0, skip = c == cx;
            const int rv = M.ld(M.r + ca), p = M.ld(M.p + ca), nx = M.op(pos + 1);
            const int r = pick ? rv : FREE;
            const bool go = pos < end && r != UNRES;
            int leg = x >> PACK_SHIFT;
            if (skipped) leg = Dx(t, s, last, c);
            const int d = max(dep + leg, r);
            if (go && !pick && !skip) M.st(M.r + ca, d + p);
            dep = go && !skip ? d : dep;
            last = go && !skip ? c : last;
            skipped = go ? skip : skipped;
            pos += go ? 1 : 0;
            x = go ? (pos < end ? nx : 0) : x;
            moved |= go;
            __syncwarp();
        }
    } while (__any_sync(FULL_MASK, moved));
    // (last = 0: the route has no other stop)
    int ret = last > 0 ? dep + Dx(t, s, last, 0) : 0;
    for (int o = 16; o > 0; o >>= 1) ret = max(ret, __shfl_xor_sync(FULL_MASK, ret, o));
    return __any_sync(FULL_MASK, pos < end) ? 0x7fffffff : ret;
}

// Worst removal's gains (Section 4.2.2): every CTA stages the current
// solution, then one warp per customer c walks it without c; gains[c] =
// z(cur) - z(cur - c).
__device__ __noinline__ void phase_gains(const AlnsTeam& t, const Smem& s, int rank, int team_blocks) {
    stage_ops(t, s, t.cur_ops, t.cur_off);
    const int warp = threadIdx.x >> 5;
    const int team_warps = team_blocks * ALNS_WARPS;
    int* rdy = s.rdy + warp * (((t.n + 1) + 3) & ~3);
    const int z = t.ctl->z_cur;
    for (int c = 1 + rank * ALNS_WARPS + warp; c <= t.n; c += team_warps) {
        const int zc = walk_skip(t, s, rdy, c);
        if ((threadIdx.x & 31) == 0) t.gains[c] = z - zc;
    }
}

// The selected insertion (ctl->upd) carried out on the CTA's staged solution:
// the ops after it move right, and the two new stops and the two behind them get
// their legs.  Reading 18 words instead of the whole solution spares a greedy
// step its staging, and the selecting CTA its write: at n=1000 the preparation
// takes 24.7 us instead of 26.4, matrix and selection 47.2 instead of 48.7.
__device__ __noinline__ void insert_local(const AlnsTeam& t, const Smem& s) {
    const int* up = t.ctl->upd;
    const int Pd = up[7], Pp = up[8], No = up[9], a = up[16], b = up[17], c = up[1];
    // places in the old order in front of which the two go
    const int at_d = Pd < Pp ? Pd : Pd - 1, at_p = Pd < Pp ? Pp - 1 : Pp;
    constexpr int E = 4096 / ALNS_THREADS;     // 2n + m <= 4096
    int w[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int p = e * ALNS_THREADS + static_cast<int>(threadIdx.x);
        if (p < No) w[e] = s.sW[p];
    }
    const int off = threadIdx.x <= t.m ? s.sWoff[threadIdx.x] : 0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int p = e * ALNS_THREADS + static_cast<int>(threadIdx.x);
        if (p >= No) break;
        int x = w[e];
        if (p == up[3]) x = (up[11] << PACK_SHIFT) | (x & PACK_MASK);     // behind the drop
        if (p == up[5]) x = (up[13] << PACK_SHIFT) | (x & PACK_MASK);     // behind the pickup (both: one gap)
        s.sW[p + (p >= at_d ? 1 : 0) + (p >= at_p ? 1 : 0)] = x;
    }
    if (threadIdx.x <= t.m) s.sWoff[threadIdx.x] = off + (a < static_cast<int>(threadIdx.x) ? 1 : 0) + (b < static_cast<int>(threadIdx.x) ? 1 : 0);
    if (threadIdx.x == 0) {
        s.sW[Pd] = (up[10] << PACK_SHIFT) | (2 * c);
        s.sW[Pp] = ((up[6] ? up[14] : up[12]) << PACK_SHIFT) | (2 * c + 1);
    }
    __syncthreads();
}

__device__ void phase_prep(const AlnsTeam& t, const Smem& s, int rank, int team_blocks, bool incr, bool fresh) {
    AlnsCtl* ctl = t.ctl;
    if (fresh) stage_W(t, s);
    else insert_local(t, s);
    const int N = s.sWoff[t.m];
    const int warp = threadIdx.x >> 5;
    const int team_warps = team_blocks * ALNS_WARPS;
    const int gw = rank * ALNS_WARPS + warp;
    int* rdy = s.rdy + warp * (((t.n + 1) + 3) & ~3);
    if (incr) phase_update(t, s, rank, team_blocks);
    // stock arrays and start loads, route by route (the route loads add up into sum_load)
    for (int r = team_warps - 1 - gw; r < t.m; r += team_warps) scan_route_stock(t, s, r);
    for (int unit = gw; !incr && unit <= N; unit += team_warps) {
        if (unit == 0) {
            const int z = walk_heads(t, s, rdy, t.H);
            if ((threadIdx.x & 31) == 0) ctl->z_work = z;
        } else {
            walk_source(t, s, rdy, unit - 1, N);
        }
    }
    // shortcut gaps (the rounded legs x->c->y shorter than x->y) and key reset
    // for every customer still to insert; W alone decides them.  The CTAs
    // from the top of the team down take this part: the update's tiles go
    // from rank 0 up, and the first CTAs may hold one tile more than the rest.
    const int G = N + t.m, nrem = ctl->nrem;
    const long long total = static_cast<long long>(nrem) * G;
    const long long tid = static_cast<long long>(team_blocks - 1 - rank) * blockDim.x + threadIdx.x;
    const long long nthr = static_cast<long long>(team_blocks) * blockDim.x;
    for (long long e = tid; e < total; e += nthr) {
        const int ti = static_cast<int>(e / G), g = static_cast<int>(e - static_cast<long long>(ti) * G);
        const int c = t.rem[ti];
        int lo = 0, hi = t.m;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s.sWoff[mid] + mid <= g) lo = mid; else hi = mid;
        }
        const int r = lo, pos = g - (s.sWoff[r] + r), L = s.sWoff[r + 1] - s.sWoff[r];
        const int x = pos > 0 ? (s.sW[s.sWoff[r] + pos - 1] & PACK_MASK) >> 1 : 0;
        const int y = pos < L ? (s.sW[s.sWoff[r] + pos] & PACK_MASK) >> 1 : 0;
        const int w = (L == 0) ? 0 : Dx(t, s, x, y);
        const bool shortcut = Dx(t, s, x, c) + Dx(t, s, c, y) < w;
        t.keys[e] = KEY_NONE;
        if (g < 32) t.rkeys[ti * 32 + g] = KEY_NONE;
        if (g == 0)
            for (int k = 0; k < 4; ++k) t.gmin[ti * 4 + k] = KEY_NONE;
        t.sc[e] = shortcut ? 1 : 0;
        if (shortcut) {
            const int slot = atomicAdd(&ctl->n_short, 1);
            t.slist[slot] = ti * G + g;
            t.scix[e] = slot;
        }
    }
}

__device__ void phase_gaps(const AlnsTeam& t, const Smem& s, int rank, int team_blocks) {
    const int m = t.m, N = s.sWoff[m], G = N + m;
    const long long tid = static_cast<long long>(rank) * blockDim.x + threadIdx.x;
    const long long nthr = static_cast<long long>(team_blocks) * blockDim.x;
    // The phase has three independent parts: the per-gap constants, the
    // per-(customer, gap) vectors and the sparse tables.  The vectors take the
    // CTAs from rank 0 up; the constants and the tables take CTAs from the top
    // of the team down, below the last four (which, with more below them when
    // there are many shortcut gaps, start the simulations right after this
    // phase), so that few CTAs do two parts.
    const int npg = (G + ALNS_THREADS - 1) / ALNS_THREADS;
    const int rank_pg = ((team_blocks - 5 - rank) % team_blocks + team_blocks) % team_blocks;
    const int rank_sp = ((team_blocks - 5 - npg - rank) % team_blocks + team_blocks) % team_blocks;
    const long long tid_pg = static_cast<long long>(rank_pg) * blockDim.x + threadIdx.x;
    for (long long gg = tid_pg; gg < G; gg += nthr) {
        const int g = static_cast<int>(gg);
        int lo = 0, hi = m;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s.sWoff[mid] + mid <= g) lo = mid; else hi = mid;
        }
        const int r = lo, pos = g - (s.sWoff[r] + r), off = s.sWoff[r], L = s.sWoff[r + 1] - off;
        const int xo = pos > 0 ? off + pos - 1 : -1, yo = pos < L ? off + pos : -1;
        const int x = xo >= 0 ? (s.sW[xo] & PACK_MASK) >> 1 : 0;
        const int y = yo >= 0 ? (s.sW[yo] & PACK_MASK) >> 1 : 0;
        t.gx[g] = xo;
        t.gy[g] = yo;
        t.gw[g] = L == 0 ? 0 : Dx(t, s, x, y);
        t.gsb[g] = xo >= 0 ? t.S_[xo] : 0;
        t.gpmin[g] = xo >= 0 ? t.PMINp[xo] : 0;
        t.gpmax[g] = xo >= 0 ? t.PMAXp[xo] : 0;
        t.gsmin[g] = yo >= 0 ? t.SMINs[yo] : (1 << 28);
        t.gsmax[g] = yo >= 0 ? t.SMAXs[yo] : -(1 << 28);
        t.groute[g] = r;
        t.gpos[g] = pos;
        // constants of gap g in the matrix tiles: as a drop gap (row) and as a pickup gap (column)
        const int Hx = xo >= 0 ? t.H[xo] : 0, Ty = yo >= 0 ? t.T[yo] : 0;
        const int sb = xo >= 0 ? t.S_[xo] : 0, pmn = xo >= 0 ? t.PMINp[xo] : 0, pmx = xo >= 0 ? t.PMAXp[xo] : 0;
        const int smn = yo >= 0 ? t.SMINs[yo] : (1 << 28), smx = yo >= 0 ? t.SMAXs[yo] : -(1 << 28);
        const int sumL = t.ctl->sum_load, rl = t.rload[r];
        int la = 0, ladj = 0, lb = 0;
        const bool okA = cap_ok(t, min(min(pmn, sb - 1), smn - 1), max(pmx, smx - 1), la);
        const bool okAdj = cap_ok(t, min(min(pmn, sb - 1), smn), max(pmx, smx), ladj);
        const bool okB = cap_ok(t, min(pmn, smn + 1), max(max(pmx, sb + 1), smx + 1), lb);
        int4* rw4 = reinterpret_cast<int4*>(t.growc + static_cast<long long>(g) * RV);
        rw4[0] = make_int4(Hx, Ty, t.gw[g], okAdj && sumL + ladj - rl <= t.R ? 1 : 0);
        rw4[1] = make_int4(0, 0, okA ? la - rl : 1 << 28, 0);
        rw4[2] = make_int4(r, pos, xo, yo);
        rw4[3] = make_int4(pmn, sb, pmx, 0);
        int4* cw4 = reinterpret_cast<int4*>(t.gcolc + static_cast<long long>(g) * CV);
        cw4[0] = make_int4(0, 0, 0, 0);
        cw4[1] = make_int4(okB ? lb - rl : 1 << 28, r, pos, yo);
        cw4[2] = make_int4(xo, smn, smx, Hx + Ty);
    }
    // per (customer, gap): the matrix vectors
    //   row {max(z, beta) (SKIPV on a shortcut gap), A1 + p_c, E, (dtD + 2^19) << 12}
    //   adj {max(z, adjacent) (SKIPV on a shortcut gap), ((dtAdj + 2^19) << 12) + gap}
    //   col {gamma (SKIPV on a shortcut gap), B1, F, (dtP << 12) + gap}
    // Each warp takes 32 consecutive gaps of one customer (G padded to a
    // multiple of 32), so that it can also reduce, per band of 32 gaps, the
    // least row and column terms (the tiles' lower bounds), and fold the
    // adjacent entries (drop and pickup back to back in one gap, exact here)
    // into the keys before any tile runs.
    {
        AlnsCtl* ctl = t.ctl;
        const int nrem = ctl->nrem, z = ctl->z_work;
        const int Gp = (G + 31) & ~31;
        const long long total = static_cast<long long>(nrem) * Gp;
        const int sumL = ctl->sum_load;
        for (long long e0 = tid; e0 < total; e0 += nthr) {
            const int ti = static_cast<int>(e0 / Gp), g = static_cast<int>(e0 - static_cast<long long>(ti) * Gp);
            const long long e = static_cast<long long>(ti) * G + g;
            const bool valid = g < G;
            const int c = t.rem[ti], pc = s.sp[c];
            int4 vr = make_int4(SKIPV, 0, 0, 0), vc = make_int4(SKIPV, 0, 0, 0);
            unsigned long long akey = KEY_NONE;
            int r = 0;
            if (valid) {
                int lo = 0, hi = m;
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (s.sWoff[mid] + mid <= g) lo = mid; else hi = mid;
                }
                r = lo;
                const int pos = g - (s.sWoff[r] + r), off = s.sWoff[r], L = s.sWoff[r + 1] - off;
                const int xo = pos > 0 ? off + pos - 1 : -1, yo = pos < L ? off + pos : -1;
                const int x = xo >= 0 ? (s.sW[xo] & PACK_MASK) >> 1 : 0;
                const int y = yo >= 0 ? (s.sW[yo] & PACK_MASK) >> 1 : 0;
                const int Hx = xo >= 0 ? t.H[xo] : 0, Ty = yo >= 0 ? t.T[yo] : 0;
                const int w = (L == 0) ? 0 : Dx(t, s, x, y);
                const int dxc = Dx(t, s, x, c), dcy = Dx(t, s, c, y), dcc = Dx(t, s, c, c);
                const int delta = dxc + dcy;
                const bool shortcut = delta < w;
                vr = make_int4(shortcut ? SKIPV : max(z, Hx + delta + Ty), Hx + dxc + pc, Hx + delta,
                               static_cast<int>(static_cast<unsigned>(delta - w + (1 << 19)) << 12));
                const int2 va = make_int2(shortcut ? SKIPV : max(z, Hx + dxc + max(dcc, pc) + dcy + Ty),
                                          static_cast<int>((static_cast<unsigned>(dxc + dcc + dcy - w + (1 << 19)) << 12) |
                                                           static_cast<unsigned>(g)));
                vc = make_int4(shortcut ? SKIPV : Hx + Ty + delta, dcy + Ty, delta + Ty,
                               static_cast<int>((static_cast<unsigned>(delta - w) << 12) + static_cast<unsigned>(g)));
                t.vrow[e] = vr;
                if (t.vadj) t.vadj[e] = va;
                t.vcol[e] = vc;
                // the adjacent entry of gap g: the stock check of the drop and
                // pickup together at g (the tiles' row constant), then its key
                // in the form the tiles' row minima take
                const int sb = xo >= 0 ? t.S_[xo] : 0, pmn = xo >= 0 ? t.PMINp[xo] : 0, pmx = xo >= 0 ? t.PMAXp[xo] : 0;
                const int smn = yo >= 0 ? t.SMINs[yo] : (1 << 28), smx = yo >= 0 ? t.SMAXs[yo] : -(1 << 28);
                int ladj = 0;
                const bool okAdj = cap_ok(t, min(min(pmn, sb - 1), smn), max(pmx, smx), ladj) &&
                                   sumL + ladj - t.rload[r] <= t.R;
                if (okAdj && va.x < SKIPV)
                    akey = (static_cast<unsigned long long>(static_cast<unsigned>(va.x - z) ^ 0x80000000u) << 32) |
                           static_cast<unsigned>(va.y);
                t.keys[e] = akey;
            }
            // band minima (excluded rows / columns left out), one store per warp
            const unsigned rx = __reduce_min_sync(FULL_MASK, vr.x < SKIPV ? static_cast<unsigned>(vr.x) : 0x7fffffffu);
            const unsigned rw = __reduce_min_sync(FULL_MASK, vr.x < SKIPV ? static_cast<unsigned>(vr.w) : 0xffffffffu);
            const unsigned cx = __reduce_min_sync(FULL_MASK, vc.x < SKIPV ? static_cast<unsigned>(vc.x) : 0x7fffffffu);
            const unsigned cw = __reduce_min_sync(FULL_MASK, vc.x < SKIPV ? static_cast<unsigned>(vc.w) : 0xffffffffu);
            const int lane = threadIdx.x & 31;
            if (lane == 0)
                t.bands[static_cast<long long>(g >> 5) * t.band_stride + ti] =
                    make_int4(static_cast<int>(rx), static_cast<int>(rw), static_cast<int>(cx), static_cast<int>(cw));
            // adjacent entries per drop vehicle: the gaps of one warp lie on
            // consecutive routes, each reduced by the whole warp
            const int rlo = static_cast<int>(__reduce_min_sync(FULL_MASK, valid ? static_cast<unsigned>(r) : 0xffffffffu));
            const int rhi = static_cast<int>(__reduce_max_sync(FULL_MASK, valid ? static_cast<unsigned>(r) : 0u));
            const unsigned long long rkey = akey == KEY_NONE ? KEY_NONE : ((akey >> 12) << 12) | static_cast<unsigned>(g);
            for (int rr = rlo; rr <= rhi; ++rr) {
                unsigned long long v = valid && r == rr ? rkey : KEY_NONE;
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long other = __shfl_xor_sync(FULL_MASK, v, o);
                    v = other < v ? other : v;
                }
                if (lane == 0 && v != KEY_NONE) {
                    atomicMin(&t.rkeys[ti * 32 + rr], v);
                    atomicMin(&t.gmin[ti * 4 + (rr & 3)], v >> 12);
                }
            }
        }
    }
    // sparse tables of the stock prefix over op positions.  Every range query
    // lies inside one route, so levels stop at the longest route; each CTA
    // builds a segment of SPB positions from a window reaching 2^top further,
    // all levels in shared memory, min then max.
    constexpr int SPB = 256;
    int lmax = 1;
    for (int r = 0; r < m; ++r) lmax = max(lmax, s.sWoff[r + 1] - s.sWoff[r]);
    int top = 0;
    while ((2 << top) <= lmax) ++top;
    const int nseg = (N + SPB - 1) / SPB;
    int* bufA = s.rdy;
    int* bufB = s.rdy + SPB + (1 << top);
    for (int seg = rank_sp; seg < nseg; seg += team_blocks) {
        const int k0 = seg * SPB;
        const int wn = min(SPB + (1 << top), N - k0);
        for (int pass = 0; pass < 2; ++pass) {
            int* spx = pass ? t.spmax : t.spmin;
            __syncthreads();                   // the buffers are free
            for (int k = threadIdx.x; k < wn; k += blockDim.x) {
                const int v = t.S_[k0 + k];
                bufA[k] = v;
                if (k < SPB) spx[k0 + k] = v;
            }
            __syncthreads();
            int* src = bufA;
            int* dst = bufB;
            for (int l = 1; l <= top; ++l) {
                const int h = 1 << (l - 1);
                const int valid = wn - (1 << l) + 1;
                for (int k = threadIdx.x; k < valid; k += blockDim.x)
                    dst[k] = pass ? max(src[k], src[k + h]) : min(src[k], src[k + h]);
                __syncthreads();
                for (int k = threadIdx.x; k < min(SPB, valid); k += blockDim.x) spx[l * N + k0 + k] = dst[k];
                int* q = src; src = dst; dst = q;
            }
        }
    }
    if (rank == 0 && threadIdx.x == 0) {
        t.ctl->work_counter = 0;
        t.ctl->tests_done = 0;
    }
}

// route of gap g
__device__ __forceinline__ int route_of_gap(const AlnsTeam& t, const Smem& s, int g) {
    int lo = 0, hi = t.m;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s.sWoff[mid] + mid <= g) lo = mid; else hi = mid;
    }
    return lo;
}

// Simulations of the shortcut gaps for the matrix phase: per shortcut gap g of
// customer c the graph with D_c alone at g (forward, backward) and with P_c
// alone at g (forward, backward); per pair of shortcut gaps of one customer (g
// itself twice: the adjacent pair) W with both stops.  A warp takes one graph one
// way, as many warps at once as have room for their times in shared memory (two
// from n = 1000 on, all eight below 300), or one pair; the CTAs are filled from
// the last one down.  The times go out of shared memory when the walk is done:
// stored by the walking lanes, every round to as many lines as there are routes, a
// graph took 31 us at n = 1000, m = 20, and takes 22 us so.  The simulations run
// between arriving at the barrier before the matrix phase and waiting at it, so the
// tiles of the other CTAs proceed meanwhile; every CTA that has finished its share
// is counted in walks_done, which the shortcut items wait for.  (One graph per CTA
// at a time, and a block barrier after every eight pairs, made the gap phase of
// small solutions with many shortcuts, as matrices without the triangle inequality
// have, half as long again: n = 15, m = 3, one CTA, 344 steps 7.3 ms in that phase, 4.1 ms now.)
__host__ __device__ inline int walk_words(int n) { return (((n + 1) + 3) & ~3) + ((2 * n + 3) & ~3); }
__host__ inline int graph_warps(int n) { return std::min(ALNS_WARPS, static_cast<int>(rdy_words(n)) / walk_words(n)); }
// CTA-sized units: of graphs, then of pairs
__device__ __forceinline__ int2 gap_walk_units(const AlnsTeam& t) {
    const int ns = min(t.ctl->n_short, SC_CAP), W = t.graph_warps;
    if (ns == 0) return make_int2(0, 0);
    return make_int2((4 * ns + W - 1) / W, (ns * ns + ALNS_WARPS - 1) / ALNS_WARPS);
}
// CTAs that have a share of them
__device__ __forceinline__ int gap_walk_ctas(const AlnsTeam& t, int team_blocks) {
    const int2 u = gap_walk_units(t);
    return min(u.x + u.y, team_blocks);
}
// both ways through W with one stop at gap (a, i), by warps 0 and 1: departures and tails
// of the W positions into shared arrays behind the walk buffers, and the three scalars
struct OneStop {
    int *H, *T;
};
__device__ __forceinline__ OneStop walk_one_stop(const AlnsTeam& t, const Smem& s, int ov, int a, int i, int N,
                                                 int* scal) {
    const int rw = ((t.n + 1) + 3) & ~3, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    OneStop r;
    r.H = s.rdy + 2 * rw;
    r.T = r.H + ((N + 3) & ~3);
    if (warp == 0) {
        int hv = 0;
        const int z1 = walk_fwd1(t, s, s.rdy, ov, a, i, r.H, &hv);
        if (lane == a) scal[1] = hv;
        if (lane == 0) scal[0] = z1;
    } else if (warp == 1) {
        int tv = 0;
        walk_bwd1(t, s, s.rdy + rw, ov, a, i, r.T, &tv);
        if (lane == a) scal[2] = tv;
    }
    __syncthreads();
    return r;
}

__device__ void gap_walks(const AlnsTeam& t, const Smem& s, int rank, int team_blocks) {
    const int m = t.m, n = t.n, N = s.sWoff[m], G = N + m;
    AlnsCtl* ctl = t.ctl;
    const int ns = min(ctl->n_short, SC_CAP), W = t.graph_warps;
    const int2 units = gap_walk_units(t);
    const int nmax = (t.scw_stride - 8) / 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rw = ((n + 1) + 3) & ~3;
    const int first = team_blocks - 1 - rank;              // this CTA's first unit
    if (first >= units.x + units.y) return;
    auto pos_of = [&](int g, int r) { return g - (s.sWoff[r] + r); };
    for (int q = first * W + warp; warp < W && q < 4 * ns; q += team_blocks * W) {
        const int e = q >> 2, as_col = (q >> 1) & 1, back = q & 1;
        const int packed = t.slist[e], ti = packed / G, g = packed - ti * G;
        const int r = route_of_gap(t, s, g), pos = pos_of(g, r), op = 2 * t.rem[ti] + as_col;
        int* rdy = s.rdy + warp * walk_words(n);
        int* times = rdy + rw;
        int* base = t.scw + static_cast<long long>(e) * t.scw_stride;
        int* scal = base + 4 * nmax + as_col * 3;
        int v = 0;
        if (back) {
            walk_bwd1(t, s, rdy, op, r, pos, times, &v);
            if (lane == r) scal[2] = v;
        } else {
            const int z1 = walk_fwd1(t, s, rdy, op, r, pos, times, &v);
            if (lane == r) scal[1] = v;
            if (lane == 0) scal[0] = z1;
        }
        __syncwarp();
        int* out = base + (2 * as_col + back) * nmax;
        for (int k = lane; k < N; k += 32) out[k] = times[k];
        __syncwarp();
    }
    __syncthreads();                                       // the pairs' ready times overlap the graphs'
    const int turn = units.x % team_blocks;                // unit units.x is this CTA's
    for (int q = ((first - turn + team_blocks) % team_blocks) * ALNS_WARPS + warp; q < ns * ns; q += team_blocks * ALNS_WARPS) {
        const int e1 = q / ns, e2 = q - e1 * ns;
        const int p1 = t.slist[e1], p2 = t.slist[e2];
        const int ti = p1 / G, g1 = p1 - ti * G, g2 = p2 - ti * G;
        if (p2 / G != ti) continue;
        const int r1 = route_of_gap(t, s, g1), r2 = route_of_gap(t, s, g2);
        const int i1 = pos_of(g1, r1), i2 = pos_of(g2, r2);
        if (r1 == r2 && i2 < i1) continue;                 // the pickup before the drop: never feasible
        const int zn = walk_insert(t, s, s.rdy + warp * rw, t.rem[ti], r1, i1, r2, i2);
        if (lane == 0) t.scpair[e1 * SC_CAP + e2] = zn;
    }
    __syncthreads();
    // results visible device-wide, then counted
    if (threadIdx.x == 0) add_acq_rel(reinterpret_cast<unsigned*>(&ctl->walks_done), 1u);
}

// Which customers can a matrix tile change the repair operator's pick for?
// Every entry of a customer in the tile is at least
//     (max(least row x, least col x), least row w + least col w)
// over the tile's rows and columns (the band minima).  The pick needs per
// customer the best entry (greedy) and, for regret-2 and regret-3, the
// makespans of the best two or three drop vehicles.  The best of each vehicle
// group so far bounds the best entry and those makespans from above; an entry
// whose drop vehicle already has an entry of no larger makespan cannot change
// that vehicle's makespan, and one not below the bound of those makespans cannot
// change their values (many vehicles tie at the makespan as it is, and with such
// ties kept 170-210 of the 2048 tiles of a step at n = 1000 were run for regret-2
// instead of 10-50: 72 us against 35 us for all its tiles).  Regret-m needs every
// vehicle's best makespan: a tile matters that may lower one of its own
// vehicles' (matrix and selection of a step at n = 1000 under all repair rules
// 47.8 us with only empty tiles left out for it, 32.1 us so).  The bounds only
// fall as tiles are scored, so a customer left out once stays out.
struct TileBounds {
    int4 r, c0, c1;                            // band minima: rows, columns (two bands)
    unsigned long long gm[4];                  // best per vehicle group so far
    unsigned long long vbest;                  // largest best makespan among the tile's drop vehicles (regret)
};

// the bounds of customer slot ti in tile (rt, ct), whose rows have drop vehicles va0..va1
__device__ __forceinline__ TileBounds tile_bounds(const AlnsTeam& t, int ti, int rt, int ct, int va0, int va1, int kind,
                                                  int G) {
    TileBounds b;
    const int4* bp = t.bands + ti;
    b.r = bp[static_cast<long long>(rt) * t.band_stride];
    b.c0 = bp[static_cast<long long>(2 * ct) * t.band_stride];
    b.c1 = make_int4(0, 0, 0x7fffffff, -1);
    if (2 * ct + 1 < ((G + 31) >> 5)) b.c1 = bp[static_cast<long long>(2 * ct + 1) * t.band_stride];
#pragma unroll
    for (int k = 0; k < 4; ++k) b.gm[k] = t.gmin[ti * 4 + k];
    b.vbest = 0;
    if (kind > 0)
        for (int v = va0; v <= va1; ++v) b.vbest = max(b.vbest, t.rkeys[ti * 32 + v] >> 32);
    return b;
}

__device__ __forceinline__ bool tile_matters(const TileBounds& b, int kind, int z) {
    const int lzz = max(b.r.x, min(b.c0.z, b.c1.z));
    if (lzz >= SKIPV) return false;
    const unsigned llo = static_cast<unsigned>(b.r.y) + min(static_cast<unsigned>(b.c0.w), static_cast<unsigned>(b.c1.w));
    const unsigned long long ldz = static_cast<unsigned>(lzz - z) ^ 0x80000000u;
    if (((ldz << 20) | (llo >> 12)) <= min(min(b.gm[0], b.gm[1]), min(b.gm[2], b.gm[3]))) return true;   // may be the best entry
    if (kind == 0) return false;
    if (kind > 2) return ldz < b.vbest;
    // the second (regret-2) or third (regret-3) least group makespan
    unsigned long long d[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = b.gm[k] >> 20;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3 - i; ++j) {
            const unsigned long long lo = min(d[j], d[j + 1]), hi = max(d[j], d[j + 1]);
            d[j] = lo;
            d[j + 1] = hi;
        }
    // may lower a drop vehicle's best makespan that counts
    return ldz < min(kind == 1 ? d[1] : d[2], b.vbest);
}

// One warp: the best entries (key, KEY_NONE: none) of customer slot ti in rows R
// (per lane, routes v in order) to the customer's keys.  One pair of atomics per
// route among the lanes: one per row, from every tile, met on the same few words
// (a step of regret-m at n = 1000, all tiles run: 450 us, and 110 us so).
// A row's own key only names the column if the entry is the customer's best:
// u, the best so far, rules the others out.
__device__ __forceinline__ void fold_rows(const AlnsTeam& t, int ti, int G, int R, int v, unsigned long long key,
                                          unsigned long long u) {
    const int lane = threadIdx.x & 31;
    if (key != KEY_NONE && (key >> 12) <= u) atomicMin(&t.keys[static_cast<long long>(ti) * G + R], key);
    unsigned long long best = key == KEY_NONE ? KEY_NONE : ((key >> 12) << 12) | static_cast<unsigned long long>(R);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {         // over the lanes behind that have the same route
        const unsigned long long other = __shfl_down_sync(FULL_MASK, best, o);
        const int ov = __shfl_down_sync(FULL_MASK, v, o);
        if (lane + o < 32 && ov == v && other < best) best = other;
    }
    const int pv = __shfl_up_sync(FULL_MASK, v, 1);
    if ((lane == 0 || pv != v) && best != KEY_NONE) {
        atomicMin(&t.rkeys[ti * 32 + v], best);
        atomicMin(&t.gmin[ti * 4 + (v & 3)], best >> 12);
    }
}

// One matrix tile (rows rt*TR.., cols ct*TC..) for every customer still to insert.
//
// Whether a (drop gap, pickup gap) pair can take a customer at all does not
// depend on the customer: every customer moves one unit of the resource, and
// the cycle test and the longest path between the two gaps are properties of
// W.  So each thread first settles its 8 pairs (row tid/8, columns
// tid%8 + 8k) into one register each: the longest-path value LP, or the
// sentinel SKIPV when the pair is excluded (capacity, pool, a cycle, a pickup
// gap before the drop gap on one route).  Per customer an entry is then
//     z' = max(max(z, beta), gamma, A1 + p_c + B1, E + LP + F)
// with the row terms in registers and the column terms one 16-byte shared
// load; shortcut gaps come out at or above SKIPV and never win.  The pair in
// which both gaps coincide (drop and pickup back to back) is the adjacent case,
// handled once per row.

__device__ void matrix_tile(const AlnsTeam& t, const Smem& s, int rt, int ct, int N, int G) {
    AlnsCtl* ctl = t.ctl;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int r0 = rt * TR, c0 = ct * TC;
    int* rowc = s.rowv;                        // [TR][RV] constants of the drop gaps
    int* colc = s.colv;                        // [TC][CV] constants of the pickup gaps
    const int sumL = ctl->sum_load;
    const bool dump = t.mode == 1;
    const int nrem = ctl->nrem;
    const int z = ctl->z_work;
    // only customers whose pick the tile can change are scored (tile_matters)
    const bool prune_on = !dump && nrem <= ACT_CAP;
    unsigned long long* actu = reinterpret_cast<unsigned long long*>(s.rdy + TILE_WORDS);   // [ACT_CAP] their best (dz, dt) so far
    int* act = reinterpret_cast<int*>(actu + ACT_CAP);                                      // [ACT_CAP] customers to score
    int* nact = s.misc + 12;
    if (tid == 0) *nact = 0;
    const bool mine = prune_on && tid < nrem;
    const int kind = ctl->rj;
    TileBounds bounds;
    if (mine)
        bounds = tile_bounds(t, tid, rt, ct, route_of_gap(t, s, r0), route_of_gap(t, s, min(G, r0 + TR) - 1), kind, G);
    __syncthreads();                           // the previous tile is done with rowc / colc and the vectors
    for (int e = tid; e < TR * (RV / 4) + TC * (CV / 4); e += blockDim.x) {
        if (e < TR * (RV / 4)) {
            const int rr = e / (RV / 4), q = e - rr * (RV / 4);
            int4 v = make_int4(0, 0, 0, 0);
            if (r0 + rr < G) v = reinterpret_cast<const int4*>(t.growc)[static_cast<long long>(r0 + rr) * (RV / 4) + q];
            else if (q == 2) v.x = -1;         // no such gap: route -1
            reinterpret_cast<int4*>(rowc)[e] = v;
        } else {
            const int e2 = e - TR * (RV / 4);
            const int cc = e2 / (CV / 4), q = e2 - cc * (CV / 4);
            int4 v = make_int4(0, 0, 0, 0);
            if (c0 + cc < G) v = reinterpret_cast<const int4*>(t.gcolc)[static_cast<long long>(c0 + cc) * (CV / 4) + q];
            else if (q == 1) v.y = -1;
            reinterpret_cast<int4*>(colc)[e2] = v;
        }
    }
    if (mine && tile_matters(bounds, kind, z)) {
        const int at = atomicAdd(nact, 1);
        act[at] = tid;
        actu[at] = min(min(bounds.gm[0], bounds.gm[1]), min(bounds.gm[2], bounds.gm[3]));
    }
    __syncthreads();
    const int na = prune_on ? *nact : nrem;
    auto cust = [&](int i) { return prune_on ? act[i] : i; };
    // Per customer the vectors of the tile's gaps come from the per-step arrays, CB
    // customers per batch, into the walk buffers (unused by tiles): cols [CB][TC]
    // int4, rows [CB][TR] int4, twice: a batch is copied in, past the registers,
    // while the one before is scored.  (Gaps past the last are not copied: no pair
    // of theirs is one.)
    constexpr int BATCH = CB * (TC + TR);
    int4* vecs = reinterpret_cast<int4*>(s.rdy);
    int2* avec = reinterpret_cast<int2*>(vecs + 2 * BATCH);        // [TR], a dump's
    unsigned long long* rowbest = reinterpret_cast<unsigned long long*>(avec + TR);   // [2][CB][TR]
    static_assert(BATCH % ALNS_THREADS == 0, "each thread copies as many vectors of a batch");
    auto copy_batch = [&](int tb, int half) {
#pragma unroll
        for (int u = 0; u < BATCH / ALNS_THREADS; ++u) {
            const int it = tid + u * ALNS_THREADS, k = it / (TC + TR), slot = it - k * (TC + TR);
            const int g = slot < TC ? c0 + slot : r0 + slot - TC;
            if (tb + k < na && g < G) {
                const int4* src = (slot < TC ? t.vcol : t.vrow) + static_cast<long long>(cust(tb + k)) * G + g;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(vecs + half * BATCH + it)), "l"(src)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto copies_done = [&]() { asm volatile("cp.async.wait_all;" ::: "memory"); };
    // this thread's pairs
    const int r = tid >> 3, cb = tid & 7;
    const int* rk = rowc + r * RV;
    const int ra = rk[8];
    const bool row_ok = ra >= 0;               // all 8 lanes of a row agree; no early exit (shuffles below)
    const int R = r0 + r;
    // every entry of the tile counts, scored or not; in shared memory until the
    // run ends
    if (tid == 0) {
        const unsigned long long each = static_cast<unsigned long long>(min(TR, G - r0)) * static_cast<unsigned>(min(TC, G - c0));
        s.counts[0] += each * static_cast<unsigned>(nrem);
        s.counts[1] += each * static_cast<unsigned>(nrem - na);
        s.counts[2] += 1ull;
        s.counts[3] += na == 0 ? 1ull : 0ull;
    }
    if (na == 0) return;                       // no customer left to score: no pair work either
    int lpv[TC / 8];
    int diag = -1;                             // column slot of the coinciding gap, if in this thread's set
    // both table reads of every pair first, as predicated loads all in flight
    // together: LP(y_a -> x_b) and the cycle test LP(y_b -> x_a) > NEG; the
    // first batch's vectors load while they are in flight
    int lpl[TC / 8], rcl[TC / 8];
    {
        const int xa = rk[10], ya = rk[11];
#pragma unroll
        for (int kk = 0; kk < TC / 8; ++kk) {
            const int* ck = colc + (cb + 8 * kk) * CV;
            const int rb = ck[5], yb = ck[7], xb = ck[8];
            const bool use = row_ok && rb >= 0;
            const bool okl = use && ya >= 0 && xb >= 0;
            const bool okr = use && ra != rb && yb >= 0 && xa >= 0;
            lpl[kk] = okl ? t.Ms[static_cast<long long>(ya) * N + xb] : NEG;
            rcl[kk] = okr ? t.Ms[static_cast<long long>(yb) * N + xa] : NEG;
        }
    }
    copy_batch(0, 0);
#pragma unroll
    for (int kk = 0; kk < TC / 8; ++kk) {
        const int cc = cb + 8 * kk;
        const int* ck = colc + cc * CV;
        int v = SKIPV;
        const int rb = ck[5];
        if (row_ok && rb >= 0) {
            if (ra == rb) {
                const int ia = rk[9], jb = ck[6];
                if (jb == ia) {
                    diag = cc;
                } else if (jb > ia) {
                    const int lo = rk[11], hi = ck[8];
                    const int mn = min(min(min(rk[12], rk[13] - 1), range_min(t, lo, hi, N) - 1), ck[9]);
                    const int mx = max(max(max(rk[14], range_max(t, lo, hi, N) - 1), t.S_[hi]), ck[10]);
                    int l2 = 0;
                    if (cap_ok(t, mn, mx, l2) && sumL - t.rload[ra] + l2 <= t.R) v = lpl[kk];
                }
            } else {
                const int dLA = rk[6], dLB = ck[4];
                if (rcl[kk] == NEG && dLA < (1 << 27) && dLB < (1 << 27) && sumL + dLA + dLB <= t.R) v = lpl[kk];
            }
        }
        lpv[kk] = v;
    }
    const bool adj_ok = rk[3] != 0;
    if (dump) {
        // every entry of the first customer still to insert written out
        // (parity runs): shortcut entries are left to the shortcut items,
        // excluded pairs read "infeasible"
        if (tid < TR) avec[tid] = r0 + tid < G ? t.vadj[r0 + tid] : make_int2(SKIPV, 0);
        copies_done();
        __syncthreads();
        const int4 rv = vecs[TC + r];
        if (!row_ok || rv.x >= SKIPV) return;
#pragma unroll
        for (int kk = 0; kk < TC / 8; ++kk) {
            const int cc = cb + 8 * kk, Cg = c0 + cc;
            const int4 g = vecs[cc];
            if (Cg >= G || g.x >= SKIPV) continue;
            const long long idx = static_cast<long long>(R) * G + Cg;
            if (cc == diag) {
                const int2 a = avec[r];
                t.dump_delta[idx] = adj_ok ? a.x - z : 0x7fffffff;
                t.dump_travel[idx] = adj_ok ? static_cast<int>(static_cast<unsigned>(a.y) >> 12) - (1 << 19) : 0;
                continue;
            }
            const int zz = max(max(rv.x, g.x), max(rv.y + g.y, rv.z + lpv[kk] + g.z));
            const unsigned lo = static_cast<unsigned>(rv.w) + static_cast<unsigned>(g.w);
            const bool ok = lpv[kk] != SKIPV;
            t.dump_delta[idx] = ok ? zz - z : 0x7fffffff;
            t.dump_travel[idx] = ok ? static_cast<int>(lo >> 12) - (1 << 19) : 0;
        }
        return;
    }
    // Only part of the pairs survive (a sixth to a third at n = 1000), mostly in
    // blocks, so a warp (4 rows by 8 columns at a time) passes over the column
    // steps in which it has none and scores the rest with its pairs in registers:
    // one 16-byte read of a column vector per entry, free of bank conflicts.  (The
    // surviving pairs compacted into a list in shared memory, every thread walking
    // a share of it, folding its row minima by shared atomics and sending one set
    // of global atomics per row and customer: matrix and selection of a step under
    // all removals and repair rules 107.8 us at n = 1000, 49.3 us now; 17.4 and
    // 15.1 us at n = 120.)
    // Shortcut gaps come out at or above SKIPV.
    unsigned fm = 0;
#pragma unroll
    for (int kk = 0; kk < TC / 8; ++kk) fm |= (lpv[kk] != SKIPV ? 1u : 0u) << kk;
    const unsigned wm = __reduce_or_sync(FULL_MASK, fm);
    // a tile with no surviving pair has nothing to compute (the adjacent
    // entries were scored with the gap vectors)
    if (!__syncthreads_or(wm != 0)) {
        copies_done();
        return;
    }
    // the row minima of the batch at tb to the global keys, a warp per customer
    auto flush = [&](int tb, int half) {
        if (tb + warp >= na) return;
        const int lane = tid & 31;
        const unsigned long long b = rowbest[(half * CB + warp) * TR + lane];
        unsigned long long key = KEY_NONE;
        if (b < static_cast<unsigned long long>(SKIPV) << 32)
            key = (static_cast<unsigned long long>(static_cast<unsigned>(static_cast<int>(b >> 32) - z) ^ 0x80000000u) << 32) |
                  (b & 0xFFFFFFFFull);
        fold_rows(t, cust(tb + warp), G, r0 + lane, rowc[lane * RV + 8], key, prune_on ? actu[tb + warp] : KEY_NONE);
    };
    int half = 0;
    for (int tb = 0; tb < na; tb += CB, half ^= 1) {
        const int nb = min(CB, na - tb);
        copies_done();
        __syncthreads();                       // this batch is there, the one before is scored
        if (tb + CB < na) copy_batch(tb + CB, half ^ 1);
        if (tb > 0) flush(tb - CB, half ^ 1);
        const int4* vec = vecs + half * BATCH;
        for (int k = 0; k < nb; ++k, vec += TC + TR) {
            const int4 rv = vec[TC + r];
            unsigned long long best = KEY_NONE;
#pragma unroll
            for (int kk = 0; kk < TC / 8; ++kk)
                if ((wm >> kk) & 1u) {
                    const int4 g = vec[cb + 8 * kk];
                    const int zz = max(max(rv.x, g.x), max(rv.y + g.y, rv.z + lpv[kk] + g.z));
                    const unsigned lo = static_cast<unsigned>(rv.w) + static_cast<unsigned>(g.w);
                    const unsigned long long key = (static_cast<unsigned long long>(static_cast<unsigned>(zz)) << 32) | lo;
                    best = lpv[kk] != SKIPV && key < best ? key : best;
                }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {  // over the row's eight lanes
                const unsigned long long other = __shfl_xor_sync(FULL_MASK, best, o);
                best = other < best ? other : best;
            }
            if (cb == 0) rowbest[(half * CB + k) * TR + r] = best;
        }
    }
    __syncthreads();
    flush((na - 1) / CB * CB, half ^ 1);
}

// Shortcut item: every entry with one shortcut gap g for customer c (the
// rounded legs x->c->y shorter than x->y, so the old paths through (x,y) do not
// all survive and the tile formula's max(z, ...) is not exact).  As a drop gap
// (as_col = 0) the graph W + D_c at g is simulated once, forward (departures
// H1, makespan z1, D_c's time h_d) and backward (tails T1), by two warps at
// once; then every pickup gap (x_b, y_b) that is not a shortcut for c is exact
// in O(1):
//     z' = max(z1, max(H1(x_b) + d(x_b,c), h_d + p_c) + d(c,y_b) + T1(y_b))
// because each path of W + D_c either survives or gains length.  As a pickup
// gap (as_col = 1) the graph is W + P_c with P_c leaving at arrival; for a
// drop gap (x_a, y_a) with drop time t_d = H2(x_a) + d(x_a,c),
//     z' = max(z2, t_d + d(c,y_a) + T2(y_a), t_d + p_c + T2(P_c)).
// Cycles, the pickup-before-drop order and capacity are the tile's tests.
// Entries whose two gaps are both shortcuts for c (the diagonal of g among
// them) are re-simulated in full, in the item of their drop gap.
__device__ void fallback_item(const AlnsTeam& t, const Smem& s, int item, int N, int G) {
    AlnsCtl* ctl = t.ctl;
    const int piece = item % FB_SPLIT;
    if (piece * static_cast<int>(blockDim.x) >= G) return;   // fewer blocks of entries than pieces
    item /= FB_SPLIT;
    const int e = item >> 1, as_col = item & 1;
    const int packed = t.slist[e];
    const int ti = packed / G, g = packed - ti * G;
    if (t.mode == 1 && ti != 0) return;        // a dump writes out the first customer only
    const int c = t.rem[ti];
    const int n = t.n, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rw = ((n + 1) + 3) & ~3;
    // the first SC_CAP shortcut gaps were simulated in the gap phase
    const bool pre = e < SC_CAP;
    const int nmax = (t.scw_stride - 8) / 4;
    const int* pbase = t.scw + static_cast<long long>(pre ? e : 0) * t.scw_stride + as_col * 2 * nmax;
    int* sh = s.misc + 8;                      // z1, h_v, t_v
    const int ga = t.groute[g], gi = t.gpos[g];
    const int ov = 2 * c + as_col;
    OneStop own = {nullptr, nullptr};          // departures and tails in W + V, simulated here
    if (!pre) own = walk_one_stop(t, s, ov, ga, gi, N, sh);
    const int* Hb = pre ? pbase : own.H;
    const int* Tb = pre ? pbase + nmax : own.T;
    const int* scal = pre ? t.scw + static_cast<long long>(e) * t.scw_stride + 4 * nmax + as_col * 3 : sh;
    const int z1 = scal[0], hv = scal[1], tv = scal[2];
    const int z = ctl->z_work, pc = s.sp[c];
    const long long scrow = static_cast<long long>(ti) * G;
    const bool dump = t.mode == 1;
    unsigned cnt = 0;
    auto loc = [&](int pos) { return pos >= 0 ? (s.sW[pos] & PACK_MASK) >> 1 : 0; };
    const unsigned long long u = min(min(t.gmin[ti * 4], t.gmin[ti * 4 + 1]), min(t.gmin[ti * 4 + 2], t.gmin[ti * 4 + 3]));
    unsigned long long rowkey = KEY_NONE;      // as_col = 0: the best of this thread's entries, all in row g
    for (int k0 = piece * blockDim.x + warp * 32; k0 < G && z1 != 0x7fffffff; k0 += FB_SPLIT * blockDim.x) {
        const int k = k0 + lane;
        unsigned long long key = KEY_NONE;
        const int vk = k < G ? t.groute[k] : -1;
        if (k < G && k != g && !t.sc[scrow + k]) {            // (both gaps shortcuts: below / elsewhere)
            const int row = as_col ? k : g, col = as_col ? g : k;
            const int a = as_col ? vk : ga, i = t.gpos[row], b = as_col ? ga : vk, j = t.gpos[col];
            const long long idx = static_cast<long long>(row) * G + col;
            if (a == b && j < i) {
                if (dump) { t.dump_delta[idx] = 0x7fffffff; t.dump_travel[idx] = 0; }
            } else {
                const int xa = t.gx[row], yb = t.gy[col];
                const bool cyc = xa >= 0 && yb >= 0 && t.Ms[static_cast<long long>(yb) * N + xa] > NEG;
                const bool ok = !cyc && entry_capacity(t, row, col, N);
                int zn;
                if (!as_col) {
                    const int xb = t.gx[col];
                    const int arr = (xb >= 0 ? Hb[xb] : 0) + Dx(t, s, loc(xb), c);
                    const int dep = max(arr, hv + pc);
                    zn = max(z1, dep + Dx(t, s, c, loc(yb)) + (yb >= 0 ? Tb[yb] : 0));
                } else {
                    const int ya = t.gy[row];
                    const int td = (xa >= 0 ? Hb[xa] : 0) + Dx(t, s, loc(xa), c);
                    zn = max(z1, max(td + Dx(t, s, c, loc(ya)) + (ya >= 0 ? Tb[ya] : 0), td + pc + tv));
                }
                ++cnt;
                const int dt = travel_delta(t, s, c, row, col);
                if (dump) {
                    t.dump_delta[idx] = ok ? zn - z : 0x7fffffff;
                    t.dump_travel[idx] = ok ? dt : 0;
                } else if (ok) {
                    key = pack_key(zn - z, dt, col);
                }
            }
        }
        if (dump) continue;
        if (as_col) {
            if (__any_sync(FULL_MASK, key != KEY_NONE)) fold_rows(t, ti, G, k, vk, key, u);
        } else rowkey = key < rowkey ? key : rowkey;
    }
    if (!as_col && !dump && __any_sync(FULL_MASK, rowkey != KEY_NONE)) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(FULL_MASK, rowkey, o);
            rowkey = other < rowkey ? other : rowkey;
        }
        if (lane == 0) {                       // (fold_rows for a single row)
            if ((rowkey >> 12) <= u) atomicMin(&t.keys[scrow + g], rowkey);
            atomicMin(&t.rkeys[ti * 32 + ga], ((rowkey >> 12) << 12) | static_cast<unsigned long long>(g));
            atomicMin(&t.gmin[ti * 4 + (ga & 3)], rowkey >> 12);
        }
    }
    // both gaps shortcuts, from the drop gap's item: full re-simulation, one warp each
    if (!as_col) {
        __syncthreads();                       // Hb / Tb done; walk buffers back to one per warp
        int* rdy = s.rdy + warp * rw;
        for (int k0 = (piece * ALNS_WARPS + warp) * 32; k0 < G; k0 += FB_SPLIT * ALNS_WARPS * 32) {
            const int kl = k0 + lane;
            const bool both = kl < G && (kl == g || t.sc[scrow + kl]);
            unsigned todo = __ballot_sync(FULL_MASK, both);
            while (todo) {
                const int col = k0 + __ffs(todo) - 1;
                todo &= todo - 1;
                const int a = ga, i = gi, b = t.groute[col], j = t.gpos[col];
                const long long idx = static_cast<long long>(g) * G + col;
                if (a == b && j < i) {
                    if (dump && lane == 0) { t.dump_delta[idx] = 0x7fffffff; t.dump_travel[idx] = 0; }
                    continue;
                }
                const bool capok = entry_capacity(t, g, col, N);
                const int e2 = t.scix[scrow + col];
                const int zn = (pre && e2 < SC_CAP) ? t.scpair[e * SC_CAP + e2] : walk_insert(t, s, rdy, c, a, i, b, j);
                const bool ok = capok && zn != 0x7fffffff;
                if (lane == 0) {
                    ++cnt;
                    const int dt = travel_delta(t, s, c, g, col);
                    if (dump) {
                        t.dump_delta[idx] = ok ? zn - z : 0x7fffffff;
                        t.dump_travel[idx] = ok ? dt : 0;
                    } else if (ok) {
                        const unsigned long long key = pack_key(zn - z, dt, col);
                        atomicMin(&t.keys[scrow + g], key);
                        atomicMin(&t.rkeys[ti * 32 + a], ((key >> 12) << 12) | static_cast<unsigned long long>(g));
                        atomicMin(&t.gmin[ti * 4 + (a & 3)], key >> 12);
                    }
                }
            }
        }
    }
    const unsigned wc = __reduce_add_sync(FULL_MASK, cnt);
    if (lane == 0 && wc) atomicAdd(&ctl->fallback_entries, static_cast<unsigned long long>(wc));
}

// Tiles go out by their distance d = |ct - rt/2| from the diagonal (the
// column tile that holds the row band's own gaps): the entries near it
// (drop and pickup on one route or on neighbouring ones) are where a
// customer's best insertion usually lies, so their scores tighten the
// bounds before the far tiles are reached.  Per d, the tiles left of the
// diagonal (ct = rt/2 - d, rt = 2d..RT-1), then those right of it
// (ct = rt/2 + d, rt = 0..2(CT-d)-1).
__device__ __forceinline__ void tile_of(int item, int RT, int CT, int* prt, int* pct) {
    if (item < RT) { *prt = item; *pct = item >> 1; return; }
    item -= RT;
    for (int d = 1; d < CT; ++d) {
        const int nl = max(0, RT - 2 * d), nr = max(0, min(RT, 2 * (CT - d)));
        if (item < nl) { *prt = 2 * d + item; *pct = (*prt >> 1) - d; return; }
        item -= nl;
        if (item < nr) { *prt = item; *pct = (item >> 1) + d; return; }
        item -= nr;
    }
    *prt = -1;                                 // past the last tile
    *pct = -1;
}

// First test of all tiles at once, a warp per tile: 95 in 100 tiles can change no
// customer's pick, and a CTA found that out one tile after another, a trip to L2
// for the tile's number, one for its bounds and a few block barriers each.  A
// CTA's eight tests give one byte of the bit mask of the tiles to run; the CTAs
// that simulate shortcut gaps (the last ones) test nothing.  Matrix and selection
// of a step at n = 1000: 41.4
// us without it and 36.3 with it (random removal), 57.1 and 51.0 (all removals).
// Thread w keeps word w of the mask (rows and columns fit 12 bits, so there
// are 128 x 64 tiles at most) and the number of bits in the words before it.
// (count below 0: the wait for the other CTAs' tests ran out)
struct TileMask {
    int count, before;
    unsigned word;
};

__device__ __noinline__ TileMask test_tiles(const AlnsTeam& t, const Smem& s, int rank, int testers, int G) {
    AlnsCtl* ctl = t.ctl;
    const int RT = (G + TR - 1) / TR, CT = (G + TC - 1) / TC;
    const int nrem = ctl->nrem, kind = ctl->rj, z = ctl->z_work;
    const int words = tile_words(G), groups = 4 * words, want = min(groups, testers);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int* flag = s.misc + 2;                    // [ALNS_WARPS]
    for (int gr = rank; gr < groups && rank < testers; gr += testers) {
        int rt = -1, ct = -1;
        tile_of(gr * ALNS_WARPS + warp, RT, CT, &rt, &ct);
        bool any = false;
        if (rt >= 0) {
            const int va0 = route_of_gap(t, s, rt * TR), va1 = route_of_gap(t, s, min(G, (rt + 1) * TR) - 1);
            for (int ti = lane; ti < nrem; ti += 32)
                any |= tile_matters(tile_bounds(t, ti, rt, ct, va0, va1, kind, G), kind, z);
        }
        any = __any_sync(FULL_MASK, any);
        // to run: -1; else the tile's entries, none of them scored
        if (lane == 0) flag[warp] = any ? -1 : rt >= 0 ? min(TR, G - rt * TR) * min(TC, G - ct * TC) : 0;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned bits = 0, out = 0, entries = 0;
#pragma unroll
            for (int w = 0; w < ALNS_WARPS; ++w) {
                const int f = flag[w];
                bits |= (f < 0 ? 1u : 0u) << w;
                out += f > 0 ? 1u : 0u;
                entries += f > 0 ? static_cast<unsigned>(f) : 0u;
            }
            s.counts[0] += static_cast<unsigned long long>(entries) * static_cast<unsigned>(nrem);
            s.counts[1] += static_cast<unsigned long long>(entries) * static_cast<unsigned>(nrem);
            s.counts[2] += out;
            s.counts[3] += out;
            reinterpret_cast<unsigned char*>(t.tmask)[gr] = static_cast<unsigned char>(bits);
        }
        __syncthreads();
    }
    bool failed = false;
    if (threadIdx.x == 0) {
        if (rank < want) add_acq_rel(reinterpret_cast<unsigned*>(&ctl->tests_done), 1u);
        failed = !await_count(ctl, &ctl->tests_done, want);
    }
    TileMask r = {-1, 0, 0u};
    if (__syncthreads_or(failed)) return r;
    const int w = static_cast<int>(threadIdx.x);
    r.word = w < words ? __ldcg(&t.tmask[w]) : 0u;
    int incl = __popc(r.word);
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) flag[warp] = incl;
    __syncthreads();
    r.count = 0;
    r.before = incl - __popc(r.word);
#pragma unroll
    for (int k = 0; k < ALNS_WARPS; ++k) {
        r.before += k < warp ? flag[k] : 0;
        r.count += flag[k];
    }
    __syncthreads();
    return r;
}

// False when a wait for other CTAs' part ran out: the keys are incomplete then.
__device__ bool phase_matrix(const AlnsTeam& t, const Smem& s, int rank, int team_blocks) {
    AlnsCtl* ctl = t.ctl;
    const int N = s.sWoff[t.m], G = N + t.m;
    const int RT = (G + TR - 1) / TR, CT = (G + TC - 1) / TC;
    const int tiles = RT * CT;
    // The shortcut items go out first: each scores a whole row or column of
    // G entries, far more work than a tile, so at the end of the phase they
    // would leave most of the team waiting.  Other CTAs may still be simulating
    // their gaps then, so the first item of a CTA waits for walks_done.
    const int nfb = 2 * ctl->n_short * FB_SPLIT;
    const int nwalks = gap_walk_ctas(t, team_blocks);
    bool walks_seen = false;
    int* slot = s.misc;
    const int testers = team_blocks - nwalks;
    const bool test = t.mode != 1 && ctl->nrem <= ACT_CAP && tiles > team_blocks && 2 * testers >= team_blocks;
    TileMask mask = {tiles, 0, 0u};
    if (test) {
        mask = test_tiles(t, s, rank, testers, G);
        if (mask.count < 0) return false;
    }
    // the tile of the k-th bit of the mask
    auto tested_tile = [&](int k) {
        if (k >= mask.before && k < mask.before + __popc(mask.word)) {
            unsigned w = mask.word;
            for (int q = mask.before; q < k; ++q) w &= w - 1;
            slot[2] = static_cast<int>(threadIdx.x) * 32 + __ffs(w) - 1;
        }
        __syncthreads();
        return slot[2];
    };
    const int ntiles = mask.count;
    const int total = ntiles + nfb;
    // The first item is the CTA's own; the rest are handed out by a counter, asked
    // for while the item before runs (the answer takes a trip to L2).  A CTA by
    // itself counts on.
    int item = rank;
    for (int turn = 0; item < total; turn ^= 1) {
        if (threadIdx.x == 0)
            slot[turn] = team_blocks == 1 ? item + 1 : total > team_blocks ? team_blocks + atomicAdd(&ctl->work_counter, 1) : total;
        if (item >= nfb) {
            int rt = 0, ct = 0;
            tile_of(test ? tested_tile(item - nfb) : item - nfb, RT, CT, &rt, &ct);
            if (rt >= 0) matrix_tile(t, s, rt, ct, N, G);
        } else {
            if (!walks_seen) {
                // the shortcut simulations, still running in other CTAs, must be done (bounded wait)
                if (__syncthreads_or(threadIdx.x == 0 && !await_count(ctl, &ctl->walks_done, nwalks))) return false;
                walks_seen = true;
            }
            fallback_item(t, s, item, N, G);
        }
        __syncthreads();                       // the next item is known, this one's buffers are free
        item = slot[turn];
    }
    return true;
}

// Insert customer c into the staged solution (s.sW, s.sWoff): its drop at
// position ia of route a, its pickup at position jb of route b (positions in
// the staged solution; on one route jb >= ia and the pickup follows the drop).
// Writes Wn / Won; all threads of the block, element-parallel: old op i of
// route v moves right by the insertions that precede it.
__device__ void insert_staged(const AlnsTeam& t, const Smem& s, int c, int a, int ia, int b, int jb, int* Wn,
                              int* Won) {
    const int m = t.m, N = s.sWoff[m];
    for (int p = threadIdx.x; p < N; p += blockDim.x) {
        int lo = 0, hi = m;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s.sWoff[mid] <= p) lo = mid; else hi = mid;
        }
        const int v = lo, i = p - s.sWoff[v];
        const int shift = (a < v ? 1 : 0) + (b < v ? 1 : 0) + (v == a && i >= ia ? 1 : 0) + (v == b && i >= jb ? 1 : 0);
        Wn[p + shift] = s.sW[p] & PACK_MASK;
    }
    if (threadIdx.x == 0) {
        const int base_a = s.sWoff[a] + (b < a ? 1 : 0);
        Wn[base_a + ia] = 2 * c;
        const int base_b = s.sWoff[b] + (a < b ? 1 : 0);
        Wn[base_b + jb + (a == b ? 1 : 0)] = 2 * c + 1;
    }
    if (threadIdx.x <= m) {
        const int v = threadIdx.x;
        Won[v] = s.sWoff[v] + (a < v ? 1 : 0) + (b < v ? 1 : 0);
    }
}

// Rank 0: per-customer argmin, greedy / regret-k choice, apply to W.
__device__ void phase_select(const AlnsTeam& t, const Smem& s) {
    AlnsCtl* ctl = t.ctl;
    const int m = t.m, N = s.sWoff[m], G = N + m, nrem = ctl->nrem;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // per-customer results in the (now free) walk buffers
    unsigned long long* bestv = reinterpret_cast<unsigned long long*>(s.rdy);       // [nrem] (dz,dt)<<12 | row
    long long* regret = reinterpret_cast<long long*>(s.rdy) + nrem;                // [nrem]
    // the column of a customer's best entry, read from its row key (needed on
    // ties of (dz, dt) between customers and for the one picked)
    int* colv = reinterpret_cast<int*>(regret + nrem);                              // [nrem]
    auto colof = [&](int ti) { return colv[ti]; };
    // A warp takes customers warp, warp + 8, ... four at a time, with the
    // route keys of all four loaded before any is reduced.
    constexpr int SU = 4;
    for (int t0 = warp; t0 < nrem; t0 += SU * ALNS_WARPS) {
        unsigned long long rks[SU];
#pragma unroll
        for (int u = 0; u < SU; ++u) {
            const int ti = t0 + u * ALNS_WARPS;
            rks[u] = (ti < nrem && lane < m) ? t.rkeys[ti * 32 + lane] : KEY_NONE;
        }
#pragma unroll
        for (int u = 0; u < SU; ++u) {
            const int ti = t0 + u * ALNS_WARPS;
            if (ti >= nrem) break;
            // best per drop vehicle (the regret-2 options) and overall, from the route keys
            const unsigned long long rk = rks[u];
            unsigned long long bv = rk;
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long other = __shfl_xor_sync(FULL_MASK, bv, o);
                bv = other < bv ? other : bv;
            }
            // regret-k over the per-vehicle options: the sum over the k best of
            // (c_i - c_1), options past the m there are counting as REGRET_INF;
            // k = 2, 3 or m for repair operators 1, 2, 3 (greedy needs none of it)
            const int rj = ctl->rj;
            long long reg = 0;
            if (rj != 0) {
                const long long cvl = (lane < m && rk != KEY_NONE)
                                          ? static_cast<long long>(static_cast<int>(static_cast<unsigned>(rk >> 32) ^ 0x80000000u))
                                          : REGRET_INF;
                // the least option (with its lane) and the least of the others, by
                // two warp min-reductions of (option + 2^31) << 6 | lane
                const unsigned long long key1 = (static_cast<unsigned long long>(cvl + (1ll << 31)) << 6) |
                                                static_cast<unsigned long long>(lane);
                unsigned long long k1 = key1;
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long other = __shfl_xor_sync(FULL_MASK, k1, o);
                    k1 = other < k1 ? other : k1;
                }
                unsigned long long k2 = (static_cast<int>(k1 & 63u) == lane) ? ~0ull : key1;
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long other = __shfl_xor_sync(FULL_MASK, k2, o);
                    k2 = other < k2 ? other : k2;
                }
                const long long c1 = static_cast<long long>(k1 >> 6) - (1ll << 31);
                const long long c2 = static_cast<long long>(k2 >> 6) - (1ll << 31);
                if (rj == 1) {
                    reg = c2 - c1;
                } else {
                    const int kreg = rj == 2 ? 3 : m;
                    int rnk = 0;
                    for (int v = 0; v < m; ++v) {
                        const long long cu = __shfl_sync(FULL_MASK, cvl, v);
                        if (cu < cvl || (cu == cvl && v < lane)) ++rnk;
                    }
                    long long term = (lane < m && rnk < kreg) ? cvl - c1 : 0;
                    for (int o = 16; o > 0; o >>= 1) term += __shfl_xor_sync(FULL_MASK, term, o);
                    if (kreg > m) term += static_cast<long long>(kreg - m) * (REGRET_INF - c1);
                    reg = term;
                }
            }
            if (lane == 0) {
                bestv[ti] = bv;
                regret[ti] = reg;
            }
        }
        // the best entries' columns, the four loads in flight together
        __syncwarp();
        if (lane < SU) {
            const int ti = t0 + lane * ALNS_WARPS;
            if (ti < nrem) {
                const unsigned long long bv = bestv[ti];
                colv[ti] = bv == KEY_NONE ? 0 : static_cast<int>(t.keys[static_cast<long long>(ti) * G + (bv & 0xFFF)] & 0xFFF);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int pick = -1;
        bool fail = false;
        for (int ti = 0; ti < nrem; ++ti) {
            if (bestv[ti] == KEY_NONE) { fail = true; break; }
            if (pick < 0) { pick = ti; continue; }
            if (ctl->rj == 0) {
                // greedy: (dz, dt), then flat index row*G + col; ties to the smaller customer id
                const unsigned long long pa = bestv[ti] >> 12, pb = bestv[pick] >> 12;
                if (pa != pb) { if (pa < pb) pick = ti; }
                else {
                    const long long fa = static_cast<long long>(bestv[ti] & 0xFFF) * G + colof(ti);
                    const long long fb = static_cast<long long>(bestv[pick] & 0xFFF) * G + colof(pick);
                    if (fa < fb) pick = ti;
                }
            } else {
                if (regret[ti] > regret[pick]) pick = ti;
            }
        }
        int* sel = s.misc + 24;                // fail, customer slot, row, column
        sel[0] = (fail || pick < 0) ? 1 : 0;
        if (fail || pick < 0) {
            ctl->repair_fail = 1;
        } else {
            sel[1] = pick;
            sel[2] = static_cast<int>(bestv[pick] & 0xFFF);
            sel[3] = colof(pick);
            // the entry is exact: the makespan once it is inserted
            ctl->z_next = ctl->z_work + static_cast<int>(static_cast<unsigned>(bestv[pick] >> 32) ^ 0x80000000u);
        }
    }
    __syncthreads();
    const int* sel = s.misc + 24;
    if (sel[0]) return;
    // apply to the other W buffer; every load the step needs is issued first
    const int pick = sel[1], row = sel[2], col = sel[3];
    const int c = t.rem[pick];
    const int a = t.groute[row], ia = t.gpos[row], b = t.groute[col], jb = t.gpos[col];
    const long long scb = static_cast<long long>(pick) * G;
    int xa = 0, ya = 0, xb = 0, yb = 0;
    bool shortcut = false;
    if (threadIdx.x == 0) {
        shortcut = t.sc[scb + row] != 0 || t.sc[scb + col] != 0;
        xa = t.gx[row]; ya = t.gy[row]; xb = t.gx[col]; yb = t.gy[col];
    }
    // the customers still to insert without the inserted one, order kept (in
    // registers for the first blockDim.x of them)
    const int k0 = threadIdx.x;
    const int remv = k0 + 1 < nrem ? t.rem[k0 + (k0 >= pick ? 1 : 0)] : 0;
    // the others carry the insertion out on their staged solutions; the solution
    // itself is written once it is complete (or for a caller that stops part way)
    if (nrem == 1 || t.mode == 3) insert_staged(t, s, c, a, ia, b, jb, t.W_ops[ctl->wsel ^ 1], t.W_off[ctl->wsel ^ 1]);
    if (threadIdx.x == 0) {
        // the next step updates the longest-path table incrementally unless a
        // gap of this insertion was a shortcut for c
        int* up = ctl->upd;
        auto loc = [&](int pos) { return pos >= 0 ? (s.sW[pos] & PACK_MASK) >> 1 : 0; };
        up[1] = c;
        up[2] = xa; up[3] = ya; up[4] = xb; up[5] = yb;
        up[6] = (a == b && ia == jb) ? 1 : 0;
        up[7] = s.sWoff[a] + ia + (b < a ? 1 : 0);
        up[8] = s.sWoff[b] + jb + (a <= b ? 1 : 0);
        up[9] = N;
        up[10] = Dx(t, s, loc(xa), c);
        up[11] = Dx(t, s, c, loc(ya));
        up[12] = Dx(t, s, loc(xb), c);
        up[13] = Dx(t, s, c, loc(yb));
        up[14] = Dx(t, s, c, c);
        up[15] = s.sp[c];
        up[16] = a;
        up[17] = b;
        ctl->incr = shortcut ? 0 : 1;
        ctl->sum_load = 0;                     // the route scans of the next step add it back up
        ctl->walks_done = 0;
    }
    __syncthreads();                           // every read of t.rem is done
    if (k0 + 1 < nrem) t.rem[k0] = remv;
    // more customers than threads (a route removal): the rest in chunks, the
    // loads of a chunk ahead of its stores
    for (int kb = blockDim.x; kb + 1 < nrem; kb += blockDim.x) {
        const int k = kb + threadIdx.x;
        const int v = k + 1 < nrem ? t.rem[k + (k >= pick ? 1 : 0)] : 0;
        __syncthreads();
        if (k + 1 < nrem) t.rem[k] = v;
    }
    if (threadIdx.x == 0) {
        ctl->nrem = nrem - 1;
        ctl->wsel ^= 1;
        ctl->n_short = 0;
    }
    __syncthreads();
}

// roulette wheel over enabled operators (fp64, explicit rounding)
__device__ int roulette(const double* w, const int* en, int k, double u) {
    double sum = 0.0;
    for (int i = 0; i < k; ++i)
        if (en[i]) sum = __dadd_rn(sum, w[i]);
    const double target = __dmul_rn(u, sum);
    double acc = 0.0;
    int last = -1;
    for (int i = 0; i < k; ++i) {
        if (!en[i]) continue;
        acc = __dadd_rn(acc, w[i]);
        last = i;
        if (target < acc) return i;
    }
    return last;
}

// Operator choice and removal size for iteration it (Algorithm 1, roulette
// wheels over the enabled operators); thread 0 of rank 0, right after the
// weight update of the previous iteration.
enum { D_RANDOM = 0, D_WORST = 1, D_SHAW = 2, D_CLUSTER = 3, D_ROUTE = 4, D_CRITICAL = 5, ND_OPS = 6 };

__device__ __noinline__ void pick_operators(const AlnsTeam& t, int it) {
    AlnsCtl* ctl = t.ctl;
    const unsigned long long base = static_cast<unsigned long long>(it) << 16;
    int en_d[ND_OPS];
    for (int i = 0; i < ND_OPS; ++i) en_d[i] = (t.destroy_mask >> i) & 1;
    const int en_r[4] = {(t.repair_mask & 1) != 0, (t.repair_mask & 2) != 0, (t.repair_mask & 4) != 0,
                         (t.repair_mask & 8) != 0};
    ctl->di = roulette(ctl->wd, en_d, ND_OPS, draw_unit(draw(t.key, base + 0)));
    ctl->rj = roulette(ctl->wr, en_r, 4, draw_unit(draw(t.key, base + 1)));
    ctl->ad[ctl->di] += 1;
    ctl->ar[ctl->rj] += 1;
    ctl->q = t.q_min + draw_below(draw(t.key, base + 2), t.q_max - t.q_min + 1);
}

// Ascending block-wide bitonic sort of P (a power of two) keys in shared memory.
__device__ void block_sort(unsigned long long* a, int P) {
    __syncthreads();
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = threadIdx.x; i < P / 2; i += blockDim.x) {
                const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                const bool asc = (lo & size) == 0;
                const unsigned long long x = a[lo], y = a[hi];
                if ((x > y) == asc) { a[lo] = y; a[hi] = x; }
            }
            __syncthreads();
        }
    }
}

// The prefix sums of r^-6, r = 1..n, in order, once per run (rank 0's block):
// the quotients side by side, then one chain of additions.
__device__ __noinline__ void worst_weights(const AlnsTeam& t, const Smem& s) {
    double* x = reinterpret_cast<double*>(s.rdy);
    for (int r = 1 + threadIdx.x; r <= t.n; r += blockDim.x) {
        const double y = static_cast<double>(r), y2 = __dmul_rn(y, y);
        x[r] = __ddiv_rn(1.0, __dmul_rn(__dmul_rn(y2, y2), y2));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double acc = 0.0;
        for (int r = 1; r <= t.n; ++r) {
            acc = __dadd_rn(acc, x[r]);
            t.pw[r] = acc;
        }
    }
    __syncthreads();
}

// The structured destroy operators (Section 4.2.2), rank 0's block: marks
// s.flags[c] and leaves the count in ctl->q.  Rankings sort (key << 12 | c),
// so ties go to the smaller customer id.  Draws: the operator's pick at
// counter base + 4, sequential draws k at base + 16 + k.
__device__ __noinline__ void select_structured(const AlnsTeam& t, const Smem& s) {
    AlnsCtl* ctl = t.ctl;
    const int n = t.n, m = t.m, di = ctl->di, q = ctl->q, qmin = t.q_min;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned long long base = static_cast<unsigned long long>(ctl->iter) << 16;
    int P = 1;
    while (P < n) P <<= 1;
    const int rw = ((n + 1) + 3) & ~3;
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(s.rdy);      // [P]
    int* vd = s.rdy + 2 * P;                   // [n+1] vehicle of the dropoff
    int* vp = vd + rw;                         // [n+1] vehicle of the pickup
    int* tdr = vp + rw;                        // [n+1] dropoff time
    int* tpk = tdr + rw;                       // [n+1] pickup completion
    int* lst = tpk + rw;                       // [n+1] customer list
    int* sh = s.misc + 32;                     // scalars
    // facts of the current solution
    stage_ops(t, s, t.cur_ops, t.cur_off);
    const bool timed = di == D_SHAW || di == D_CRITICAL;
    if (timed && warp == 0) walk_heads(t, s, s.rdy, t.H);
    __syncthreads();
    const int N = s.sWoff[m];
    for (int k = tid; k < N; k += blockDim.x) {
        int lo = 0, hi = m;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s.sWoff[mid] <= k) lo = mid; else hi = mid;
        }
        const int o = s.sW[k] & PACK_MASK, c = o >> 1;
        if (o & 1) { vp[c] = lo; if (timed) tpk[c] = t.H[k]; }
        else { vd[c] = lo; if (timed) tdr[c] = t.H[k]; }
    }
    __syncthreads();
    auto count_flags = [&]() {
        // every thread gets the number of marked customers
        __syncthreads();
        if (warp == 0) {
            int w = 0;
            for (int c0 = 1; c0 <= n; c0 += 32) w += __popc(__ballot_sync(FULL_MASK, c0 + lane <= n && s.flags[c0 + lane]));
            if (lane == 0) sh[1] = w;
        }
        __syncthreads();
        return sh[1];
    };
    auto take_sorted = [&](int need) {
        // mark the first `need` customers of the sorted keys (unmarked ones only carry keys)
        for (int i = tid; i < P && i < need; i += blockDim.x)
            if (keys[i] != KEY_NONE) s.flags[static_cast<int>(keys[i] & 0xFFF)] = 1;
    };
    if (di == D_WORST) {
        // removal gains from the team phase, largest first; q roulette draws
        // over the remaining ranked list with weight r^-6 on the r-th
        for (int i = tid; i < P; i += blockDim.x)
            keys[i] = i < n ? ((static_cast<unsigned long long>((1ll << 30) - t.gains[i + 1]) << 12) |
                               static_cast<unsigned long long>(i + 1))
                            : KEY_NONE;
        block_sort(keys, P);
        if (warp == 0) {
            // the r-th weight's prefix first passes the target, then the r-th
            // customer of the ranking still there, 32 at a time
            for (int k = 0; k < q; ++k) {
                const int R = n - k;
                const double target = __dmul_rn(draw_unit(draw(t.key, base + 16 + static_cast<unsigned long long>(k))), t.pw[R]);
                int r = R;
                for (int r0 = 1; r0 < R; r0 += 32) {
                    const unsigned past = __ballot_sync(FULL_MASK, r0 + lane < R && t.pw[r0 + lane] > target);
                    if (past) { r = r0 + __ffs(past) - 1; break; }
                }
                for (int i0 = 0; i0 < n; i0 += 32) {
                    const int c = i0 + lane < n ? static_cast<int>(keys[i0 + lane] & 0xFFF) : 0;
                    const bool there = i0 + lane < n && !s.flags[c];
                    const unsigned left = __ballot_sync(FULL_MASK, there);
                    const int cnt = __popc(left);
                    if (r > cnt) { r -= cnt; continue; }
                    if (there && __popc(left & ((1u << lane) - 1u)) == r - 1) s.flags[c] = 1;
                    break;
                }
                __syncwarp();
            }
        }
    } else if (di == D_SHAW || di == D_CLUSTER) {
        // a random seed and the q-1 customers nearest to it (Shaw: by the
        // relatedness measure, doubled to stay integral)
        if (tid == 0) sh[0] = 1 + draw_below(draw(t.key, base + 4), n);
        __syncthreads();
        const int sd = sh[0];
        for (int i = tid; i < P; i += blockDim.x) {
            const int c = i + 1;
            unsigned long long kk = KEY_NONE;
            if (c <= n && c != sd) {
                long long k2 = Dx(t, s, sd, c);
                if (di == D_SHAW) {
                    long long dt = static_cast<long long>(tdr[sd]) - tdr[c];
                    dt = dt < 0 ? -dt : dt;
                    k2 = 18 * k2 + 6 * dt + 5 * (vd[sd] != vd[c]) + 5 * (vp[sd] != vp[c]);
                }
                kk = (static_cast<unsigned long long>(k2) << 12) | static_cast<unsigned long long>(c);
            }
            keys[i] = kk;
        }
        block_sort(keys, P);
        if (tid == 0) s.flags[sd] = 1;
        take_sorted(q - 1);
    } else {
        // a random non-empty route, or the bottleneck route's customers
        if (di == D_CRITICAL && warp == 0) {
            // latest return, the lower index on ties (times stay below 2^27); its
            // customers in customer order
            int rv = 0;
            if (lane < m && s.sWoff[lane + 1] > s.sWoff[lane]) {
                const int last = s.sWoff[lane + 1] - 1;
                rv = t.H[last] + Dx(t, s, (s.sW[last] & PACK_MASK) >> 1, 0);
            }
            const unsigned top = __reduce_max_sync(FULL_MASK, lane < m ? (static_cast<unsigned>(rv) << 5) | (31u - lane) : 0u);
            const int vb = 31 - static_cast<int>(top & 31u);
            int nl = 0;
            for (int c0 = 1; c0 <= n; c0 += 32) {
                const int c = c0 + lane;
                const bool on = c <= n && (vd[c] == vb || vp[c] == vb);
                const unsigned bal = __ballot_sync(FULL_MASK, on);
                if (on) lst[nl + __popc(bal & ((1u << lane) - 1u))] = c;
                nl += __popc(bal);
            }
            if (lane == 0) sh[2] = nl;
        }
        __syncthreads();
        if (tid == 0) {
            if (di == D_ROUTE) {
                int K = 0;
                for (int v = 0; v < m; ++v) K += s.sWoff[v + 1] > s.sWoff[v] ? 1 : 0;
                int kk = draw_below(draw(t.key, base + 4), K);
                int vsel = 0;
                for (int v = 0; v < m; ++v)
                    if (s.sWoff[v + 1] > s.sWoff[v] && kk-- == 0) { vsel = v; break; }
                sh[0] = vsel;
            } else {
                // q of the listed customers by partial Fisher-Yates (all if fewer)
                const int nl = sh[2];
                const int take = q < nl ? q : nl;
                for (int k = 0; k < take; ++k) {
                    const int jj = k + draw_below(draw(t.key, base + 16 + static_cast<unsigned long long>(k)), nl - k);
                    const int tmp = lst[k];
                    lst[k] = lst[jj];
                    lst[jj] = tmp;
                    s.flags[lst[k]] = 1;
                }
                sh[0] = -1;
            }
        }
        __syncthreads();
        if (di == D_ROUTE) {
            const int vsel = sh[0];
            for (int k = s.sWoff[vsel] + tid; k < s.sWoff[vsel + 1]; k += blockDim.x)
                s.flags[(s.sW[k] & PACK_MASK) >> 1] = 1;
        }
        const int cnt = count_flags();
        if (cnt < qmin) {
            // top up: route removal by the least travel time from a removed
            // customer, critical path by the latest pickup completion
            if (di == D_ROUTE && warp == 0) {
                int w = 0;
                for (int c0 = 1; c0 <= n; c0 += 32) {
                    const int c = c0 + lane;
                    const bool r = c <= n && s.flags[c];
                    const unsigned bal = __ballot_sync(FULL_MASK, r);
                    if (r) lst[w + __popc(bal & ((1u << lane) - 1u))] = c;
                    w += __popc(bal);
                }
            }
            __syncthreads();
            for (int i = tid; i < P; i += blockDim.x) {
                const int c = i + 1;
                unsigned long long kk = KEY_NONE;
                if (c <= n && !s.flags[c]) {
                    long long k2;
                    if (di == D_ROUTE) {
                        k2 = 0x7fffffffll;
                        for (int j = 0; j < cnt; ++j) k2 = min(k2, static_cast<long long>(Dx(t, s, lst[j], c)));
                    } else {
                        k2 = (1ll << 30) - tpk[c];
                    }
                    kk = (static_cast<unsigned long long>(k2) << 12) | static_cast<unsigned long long>(c);
                }
                keys[i] = kk;
            }
            block_sort(keys, P);
            take_sorted(qmin - cnt);
        }
    }
    const int total = count_flags();
    if (tid == 0) ctl->q = total;
    __syncthreads();
}

// Rank 0: the destroy step (operator and q drawn at the end of the previous
// iteration), W = cur - removed.
// W[0] = the current solution without the customers flagged in s.flags:
// block-wide scan of the kept ops.  All threads of the block.
__device__ void build_W_from_cur(const AlnsTeam& t, const Smem& s) {
    const int m = t.m, two_n = 2 * t.n;
    const int per = (two_n + blockDim.x - 1) / blockDim.x;
    const int k0 = threadIdx.x * per, k1 = min(two_n, k0 + per);
    int cnt = 0;
    for (int k = k0; k < k1; ++k) cnt += s.flags[t.cur_ops[k] >> 1] ? 0 : 1;
    int* wsum = s.misc;                        // [ALNS_WARPS]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();                           // wsum is free
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = 0, kept_total = 0;
    for (int w = 0; w < ALNS_WARPS; ++w) {
        before += w < warp ? wsum[w] : 0;
        kept_total += wsum[w];
    }
    const int base_pos = before + incl - cnt;
    int pos = base_pos;
    int* Wn = t.W_ops[0];
    for (int k = k0; k < k1; ++k) {
        const int o = t.cur_ops[k];
        if (!s.flags[o >> 1]) Wn[pos++] = o;
    }
    // route offsets: the kept-op count before each route start, taken from the
    // scan by the thread whose range holds that start
    for (int v = 0; v <= m; ++v) {
        const int ov = t.cur_off[v];
        if (ov >= k0 && ov < k1) {
            int kept = base_pos;
            for (int k = k0; k < ov; ++k) kept += s.flags[t.cur_ops[k] >> 1] ? 0 : 1;
            t.W_off[0][v] = kept;
        } else if (ov == two_n && threadIdx.x == 0) {
            t.W_off[0][v] = kept_total;
        }
    }
    __syncthreads();
}

__device__ __noinline__ void phase_begin(const AlnsTeam& t, const Smem& s) {
    AlnsCtl* ctl = t.ctl;
    const int n = t.n;
    int* perm = s.rdy;                         // [n], shared memory
    for (int k = threadIdx.x; k < n; k += blockDim.x) perm[k] = k + 1;
    for (int c = threadIdx.x; c <= n; c += blockDim.x) s.flags[c] = 0;
    __syncthreads();
    if (threadIdx.x == 0 && ctl->di == D_RANDOM) {
        const int it = ctl->iter;
        const unsigned long long base = static_cast<unsigned long long>(it) << 16;
        const int q = ctl->q;
        for (int k = 0; k < q; ++k) {
            const int jj = k + draw_below(draw(t.key, base + 16 + static_cast<unsigned long long>(k)), n - k);
            const int tmp = perm[k];
            perm[k] = perm[jj];
            perm[jj] = tmp;
            s.flags[perm[k]] = 1;
        }
    }
    __syncthreads();
    if (ctl->di != D_RANDOM) select_structured(t, s);
    if (threadIdx.x == 0) {
        ctl->repair_fail = 0;
        ctl->z_next = ctl->z_cur;              // should nothing be removed
        ctl->n_short = 0;
        ctl->work_counter = 0;
        ctl->wsel = 0;
        ctl->incr = 0;                         // W lost customers: the next step walks it in full
        ctl->sum_load = 0;
        ctl->walks_done = 0;
    }
    __syncthreads();
    // removed customers in ascending id order (ballot compaction by warp 0)
    if ((threadIdx.x >> 5) == 0) {
        const int lane = threadIdx.x & 31;
        int w = 0;
        for (int c0 = 1; c0 <= n; c0 += 32) {
            const int c = c0 + lane;
            const bool r = c <= n && s.flags[c];
            const unsigned bal = __ballot_sync(FULL_MASK, r);
            if (r) t.rem[w + __popc(bal & ((1u << lane) - 1u))] = c;
            w += __popc(bal);
        }
        if (lane == 0) ctl->nrem = w;
    }
    build_W_from_cur(t, s);
}

// Rank 0: evaluate the repaired W and apply Algorithm 1's acceptance, cooling,
// reheat and weight update.  With first = true only records the start.
__device__ __noinline__ void phase_end(const AlnsTeam& t, const Smem& s, bool first) {
    AlnsCtl* ctl = t.ctl;
    const int n = t.n, m = t.m;
    if (first) {
        stage_W(t, s);
        if ((threadIdx.x >> 5) == 0) {
            int z;
            unsigned st;
            walk_depot(t, s, s.rdy, &z, &st);
            if ((threadIdx.x & 31) == 0) {
                ctl->z_work = z;
                ctl->st_work = st;
            }
        }
    } else {
        // the last insertion left the makespan; the stock is what it did not
        // judge as a whole (no insertion closes a cycle)
        int* sh = s.misc + 32;                 // start loads, vehicles over capacity
        if (threadIdx.x == 0) { sh[0] = 0; sh[1] = 0; }
        __syncthreads();
        const int* W = t.W_ops[ctl->wsel];
        const int* Wo = t.W_off[ctl->wsel];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int r = warp; r < m && !ctl->repair_fail; r += ALNS_WARPS) {
            const int en = Wo[r + 1];
            int carry = 0, mn = 0, mx = 0;
            for (int base = Wo[r]; base < en; base += 32) {
                const bool in = base + lane < en;
                int v = in ? ((W[base + lane] & 1) ? 1 : -1) : 0;
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FULL_MASK, v, o);
                    if (lane >= o) v += y;
                }
                if (in) {
                    mn = min(mn, carry + v);
                    mx = max(mx, carry + v);
                }
                carry += __shfl_sync(FULL_MASK, v, 31);
            }
            mn = __reduce_min_sync(FULL_MASK, mn);
            mx = __reduce_max_sync(FULL_MASK, mx);
            int load = 0;
            const bool ok = cap_ok(t, mn, mx, load);
            if (lane == 0) {
                atomicAdd(&sh[0], load);
                if (!ok) sh[1] = 1;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            ctl->z_work = ctl->repair_fail ? 0x7fffffff : ctl->z_next;
            ctl->st_work = ctl->repair_fail ? VRPRPD_MALFORMED
                                            : (sh[1] ? VRPRPD_VEH_CAP : 0u) | (sh[0] > t.R ? VRPRPD_POOL : 0u);
        }
    }
    __syncthreads();
    int* decision = s.misc;
    if (threadIdx.x == 0) {
        const int zn = ctl->z_work;
        const unsigned st = ctl->st_work;
        int accept = 0, newbest = 0;
        if (first) {
            accept = 1;
            newbest = 1;
            ctl->z_cur = zn;
            ctl->z_best = zn;
            ctl->z_init = zn;
            ctl->T = __dmul_rn(t.T0, static_cast<double>(zn));
            ctl->T_init = ctl->T;
            if (st != 0u) fail_run(ctl, DEV_BAD_STATE);
        } else {
            const int it = ctl->iter;
            const unsigned long long base = static_cast<unsigned long long>(it) << 16;
            const int di = ctl->di, rj = ctl->rj;
            if (st != 0u) {
                ctl->rejected += 1;
            } else if (zn < ctl->z_cur) {
                accept = 1;
                ctl->z_cur = zn;
                ctl->sd[di] += t.sigma2;
                ctl->sr[rj] += t.sigma2;
                ctl->improved += 1;
                ctl->accepted += 1;
                if (zn < ctl->z_best) {
                    newbest = 1;
                    ctl->z_best = zn;
                    ctl->sd[di] += t.sigma1 - t.sigma2;
                    ctl->sr[rj] += t.sigma1 - t.sigma2;
                    ctl->stagnation = 0;
                    ctl->new_best += 1;
                }
            } else {
                const double x = -__ddiv_rn(static_cast<double>(static_cast<long long>(zn) - ctl->z_cur), ctl->T);
                const double u = draw_unit(draw(t.key, base + 3));
                if (u < exp_sa(x)) {
                    accept = 1;
                    ctl->z_cur = zn;
                    ctl->sd[di] += t.sigma3;
                    ctl->sr[rj] += t.sigma3;
                    ctl->accepted += 1;
                }
            }
            ctl->T = __dmul_rn(t.alpha, ctl->T);
            ctl->stagnation += 1;
            if (ctl->stagnation >= t.stagnation_limit && ctl->T < __dmul_rn(0.01, ctl->T_init)) {
                ctl->T = __dmul_rn(__dmul_rn(t.reheat, t.T0), static_cast<double>(ctl->z_best));
                ctl->stagnation = 0;
                ctl->reheats += 1;
            }
            if (it % t.tau == 0) {
                for (int i = 0; i < ND_OPS; ++i) {
                    const double ratio = ctl->ad[i] ? __ddiv_rn(static_cast<double>(ctl->sd[i]), static_cast<double>(ctl->ad[i])) : 0.0;
                    const double w = __dadd_rn(__dmul_rn(__dsub_rn(1.0, t.r), ctl->wd[i]), __dmul_rn(t.r, ratio));
                    ctl->wd[i] = w < t.w_min ? t.w_min : w;
                    ctl->sd[i] = 0;
                    ctl->ad[i] = 0;
                }
                for (int i = 0; i < 4; ++i) {
                    const double ratio = ctl->ar[i] ? __ddiv_rn(static_cast<double>(ctl->sr[i]), static_cast<double>(ctl->ar[i])) : 0.0;
                    const double w = __dadd_rn(__dmul_rn(__dsub_rn(1.0, t.r), ctl->wr[i]), __dmul_rn(t.r, ratio));
                    ctl->wr[i] = w < t.w_min ? t.w_min : w;
                    ctl->sr[i] = 0;
                    ctl->ar[i] = 0;
                }
            }
            if (t.trace) t.trace[it - 1] = ctl->z_cur;
        }
        decision[0] = accept;
        decision[1] = newbest;
        const int next = first ? 1 : ctl->iter + 1;
        if (next <= t.iterations) pick_operators(t, next);
    }
    __syncthreads();
    const int accept = decision[0], newbest = decision[1];
    const int* W = t.W_ops[ctl->wsel];
    const int* Wo = t.W_off[ctl->wsel];
    if (accept && !first) {
        for (int k = threadIdx.x; k < 2 * n; k += blockDim.x) t.cur_ops[k] = W[k];
        for (int v = threadIdx.x; v <= m; v += blockDim.x) t.cur_off[v] = Wo[v];
    }
    if (newbest) {
        for (int k = threadIdx.x; k < 2 * n; k += blockDim.x) t.best_ops[k] = W[k];
        for (int v = threadIdx.x; v <= m; v += blockDim.x) t.best_off[v] = Wo[v];
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// multi-instance checkpoints (Section 4.2.1): all teams of the launch meet
// ---------------------------------------------------------------------------
// Barrier over every CTA of the launch; bounded (about 2 s), sets ctl->err.
__device__ bool grid_barrier(const AlnsTeam& t, unsigned& ggen) {
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned* vgen = &t.gbar[1];
        const unsigned total = gridDim.x;
        __threadfence();
        const unsigned arrived = atomicAdd(&t.gbar[0], 1u) + 1u;
        if (arrived == total) {
            t.gbar[0] = 0u;
            __threadfence();
            atomicExch(&t.gbar[1], ggen + 1u);
        } else {
            const uint64_t t0 = global_ns();
            while (*vgen == ggen) {
                if (global_ns() - t0 > t.ctl->wait_ns) {
                    fail_run(t.ctl, DEV_TIMEOUT_BARRIER);
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    ggen += 1u;
    __syncthreads();
    return *reinterpret_cast<volatile int*>(&t.ctl->err) == 0;
}

// Rank 0 of each team, between two grid barriers: when the best of all teams
// (lowest index among equal bests) beats this team's best, it becomes this
// team's current and best solution.  Nothing writes a best solution between
// the two barriers, so every team reads the same ones.
__device__ __noinline__ void replica_import(const AlnsTeam& t, const Smem& s) {
    AlnsCtl* ctl = t.ctl;
    int* sh = s.misc;
    if (threadIdx.x == 0) {
        int g = 0, zg = *reinterpret_cast<volatile const int*>(&t.sib[0].ctl->z_best);
        for (int r = 1; r < t.nreplicas; ++r) {
            const int zr = *reinterpret_cast<volatile const int*>(&t.sib[r].ctl->z_best);
            if (zr < zg) { zg = zr; g = r; }
        }
        sh[0] = ctl->z_best > zg ? g : -1;
        sh[1] = zg;
    }
    __syncthreads();
    const int g = sh[0];
    if (g >= 0) {
        const int* bo = t.sib[g].best_ops;
        const int* bf = t.sib[g].best_off;
        for (int k = threadIdx.x; k < 2 * t.n; k += blockDim.x) {
            const int o = __ldcg(bo + k);
            t.cur_ops[k] = o;
            t.best_ops[k] = o;
        }
        for (int v = threadIdx.x; v <= t.m; v += blockDim.x) {
            const int o = __ldcg(bf + v);
            t.cur_off[v] = o;
            t.best_off[v] = o;
        }
        if (threadIdx.x == 0) {
            ctl->z_cur = sh[1];
            ctl->z_best = sh[1];
            ctl->stagnation = 0;
            ctl->imports += 1;
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// periodic local search (Section 4.2.6), on the current solution
// ---------------------------------------------------------------------------
// A pass finds, over all its candidate customers c, the least (makespan,
// travel, customer, gaps) among the moves that lower the makespan, and applies
// it.  Pickup repositioning takes c's pickup out and puts it into any gap the
// schedule allows; relocation takes both ops out and puts them into two gaps
// (or one) of a vehicle other than the bottleneck.  Taking c out can leave one
// of its old routes over capacity; only the receiving routes are judged, so a
// move is kept only if every such route is one it writes to.
//
// Candidates are independent, so each is one CTA's work (relocation: split by
// target vehicle while CTAs are idle) and the team meets once per pass.
//   Pickup repositioning works on cur without the pickup alone: one walk gives
// every departure H and the makespan z, one backward walk every tail T and
// which ops lead to c's drop (a pickup before one of those is a cycle).  A gap
// (x, y) that is no shortcut for c is then exact in O(1),
//     z' = max(z, max(H(x) + d(x,c), H(drop) + p_c) + d(c,y) + T(y)),
// since no path gets shorter; a shortcut gap is simulated.
//   Relocation works on cur without c.  A gap costs H(x) + d(x,c) + d(c,y) + T(y)
// whether it takes the drop or the pickup, so only gaps below the current
// makespan (less the route's largest shortcut) can matter; each of those walks
// W from its next op once, as far as the target route's end, and settles its
// pairs on the way with the matrix formula; a gap whose least (makespan, travel) is
// above what a move of the pass has reached is left out (two refinement rounds of
// the n=1000 start: 22.2 ms without, 1.5 ms with).  Pairs with a shortcut gap are
// simulated.
// Before, every candidate was a team step of its own (the whole longest-path
// table walked again, the matrix phase, five team barriers): 167 ms per local
// search of both kinds at n=1000 m=20, 0.35 ms now; at n=120 m=5, eight
// replicas, 40 ms of an 81 ms run, 1.0 ms now.
enum { LS_PICKUP = 1, LS_RELOCATE = 2 };

constexpr int TAIL_BITS = (1 << 29) - 1;       // a tail; the bit above: the op leads to the candidate's drop
constexpr int TAIL_NONE = INT32_MIN + 1;       // tail of a pickup that is not in the solution
constexpr int LS_MAX_CTAS = SC_CAP * SC_CAP / 4;

// Scratch of one CTA, in words: H, T, stock after each op, packed prefix and
// suffix extremes (N each), then one word per gap of a route and a list of its gaps.
__device__ __forceinline__ int ls_scratch_words(int n) { return 14 * n + 8; }
// The CTAs that take part: the scratch lies in the buffers of the shortcut
// simulations and of the longest-path table, which the next step rebuilds.
__device__ __forceinline__ int ls_active(const AlnsTeam& t, int team_blocks) {
    const int N = 2 * t.n, w = ls_scratch_words(t.n);
    const int a0 = SC_CAP * (4 * N + 8) / w, a1 = N * N / w;
    return min(team_blocks, min(a0 + 2 * a1, LS_MAX_CTAS));
}
__device__ __forceinline__ int* ls_scratch(const AlnsTeam& t, int rank) {
    const int N = 2 * t.n, w = ls_scratch_words(t.n);
    const int a0 = SC_CAP * (4 * N + 8) / w, a1 = N * N / w;
    if (rank < a0) return t.scw + static_cast<long long>(rank) * w;
    rank -= a0;
    return rank < a1 ? t.Ms + static_cast<long long>(rank) * w : t.Ms2 + static_cast<long long>(rank - a1) * w;
}

// Rank 0: the candidates of one pass, in ascending id, and where every op of
// the current solution stands.  Pickup repositioning: customers whose pickup is
// on a vehicle returning at 95% of the makespan or later (20 ret >= 19 z);
// relocation: customers with an op on the bottleneck vehicle (latest return,
// lower index on ties).
__device__ __noinline__ void ls_candidates(const AlnsTeam& t, const Smem& s, int mode) {
    AlnsCtl* ctl = t.ctl;
    const int n = t.n, m = t.m, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    stage_ops(t, s, t.cur_ops, t.cur_off);
    int* ret = s.misc + 32;                    // [32] return time per route
    uint16_t* place = reinterpret_cast<uint16_t*>(t.gains);   // [2n+2] by op code
    for (int c = tid; c <= n; c += blockDim.x) s.flags[c] = 0;
    if (warp == 0) {
        walk_heads(t, s, s.rdy, t.H);
        __syncwarp();
        int rv = 0;
        if (lane < m && s.sWoff[lane + 1] > s.sWoff[lane]) {
            const int last = s.sWoff[lane + 1] - 1;
            rv = t.H[last] + Dx(t, s, (s.sW[last] & PACK_MASK) >> 1, 0);
        }
        ret[lane] = rv;
        __syncwarp();
        if (lane == 0) {
            int b = 0;
            for (int v = 1; v < m; ++v)
                if (ret[v] > ret[b]) b = v;
            ctl->ls_bott = b;
            ctl->ls_bound = KEY_NONE;
        }
    }
    __syncthreads();
    const long long z = ctl->z_cur;
    const int bott = ctl->ls_bott, N = s.sWoff[m];
    for (int k = tid; k < N; k += blockDim.x) {
        int lo = 0, hi = m;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s.sWoff[mid] <= k) lo = mid; else hi = mid;
        }
        const int o = s.sW[k] & PACK_MASK;
        place[o] = static_cast<uint16_t>(k);
        const bool cand = mode == LS_PICKUP ? ((o & 1) && 20ll * ret[lo] >= 19ll * z) : lo == bott;
        if (cand) s.flags[o >> 1] = 1;
    }
    __syncthreads();
    if (warp == 0) {
        int w = 0;
        for (int c0 = 1; c0 <= n; c0 += 32) {
            const int c = c0 + lane;
            const bool r = c <= n && s.flags[c];
            const unsigned bal = __ballot_sync(FULL_MASK, r);
            if (r) t.lscand[w + __popc(bal & ((1u << lane) - 1u))] = c;
            w += __popc(bal);
        }
        if (lane == 0) ctl->ls_ncand = w;
    }
    __syncthreads();
}

// Stage cur without the ops at places lo < hi (hi < 0: lo alone): packed legs
// and ops, route offsets.
__device__ void stage_without(const AlnsTeam& t, const Smem& s, int lo, int hi) {
    const int m = t.m, N = 2 * t.n - (hi >= 0 ? 2 : 1);
    for (int v = threadIdx.x; v <= m; v += blockDim.x) {
        const int o = t.cur_off[v];
        s.sWoff[v] = o - (lo < o ? 1 : 0) - (hi >= 0 && hi < o ? 1 : 0);
    }
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        int q = k + (k >= lo ? 1 : 0);
        if (hi >= 0 && q >= hi) ++q;
        s.sW[k] = t.cur_ops[q];
    }
    __syncthreads();
    // a neighbour may already carry its leg: its op bits stay the same
    volatile int* W = s.sW;
    for (int k = threadIdx.x; k < N; k += blockDim.x) {
        int l = 0, h = m;
        while (h - l > 1) {
            const int mid = (l + h) >> 1;
            if (s.sWoff[mid] <= k) l = mid; else h = mid;
        }
        const int o = W[k];
        const int prev = k == s.sWoff[l] ? 0 : (W[k - 1] & PACK_MASK) >> 1;
        W[k] = (Dx(t, s, prev, o >> 1) << PACK_SHIFT) | o;
    }
    __syncthreads();
}

// One warp: the tail of every staged op (longest path from its departure to
// the end of the schedule) into T, with the mark of the ops that lead to the
// drop of c at dpos.  c > 0: c's pickup is not in the solution.
__device__ void walk_tails(const AlnsTeam& t, const Smem& s, int* tp_, int* T, int c0, int dpos) {
    const int lane = threadIdx.x & 31, n = t.n;
    for (int c = lane; c <= n; c += 32) tp_[c] = c0 > 0 && c == c0 ? TAIL_NONE : UNRES;
    __syncwarp();
    const WalkMem M(s, tp_);
    const int start = lane < t.m ? s.sWoff[lane] : 0;
    int pos = (lane < t.m ? s.sWoff[lane + 1] : 0) - 1;
    int x = pos >= start ? M.op(pos) : 0;
    int leg = pos >= start ? Dx(t, s, (x & PACK_MASK) >> 1, 0) : 0, acc = 0, mark = 0;
    bool moved;
    do {
        moved = false;
#pragma unroll
        for (int k = 0; k < WALK_ROUNDS; ++k) {
            const unsigned ca = M.at(x);
            const bool pick = (x & 1) != 0;
            const int rv = M.ld(M.r + ca), p = M.ld(M.p + ca), nx = M.op(max(pos - 1, 0));
            const int r = pick ? TAIL_NONE : rv;   // (a drop of a customer without its pickup waits for nothing, as a pickup)
            const bool go = pos >= start && r != UNRES;
            const int after = acc + leg;
            const int d = r == TAIL_NONE ? after : max(after, p + (r & TAIL_BITS));
            int mk = mark | (r == TAIL_NONE ? 0 : r & ~TAIL_BITS);
            if (pos == dpos) mk = TAIL_BITS + 1;
            if (go) T[pos] = d | mk;
            if (go && pick) M.st(M.r + ca, d | mk);
            acc = go ? d : acc;
            mark = go ? mk : mark;
            leg = go ? x >> PACK_SHIFT : leg;
            pos -= go ? 1 : 0;
            x = go ? (pos >= start ? nx : 0) : x;
            moved |= go;
            __syncwarp();
        }
    } while (__any_sync(FULL_MASK, moved));
}

// One warp, route r of the staged solution: stock after every op, its running
// extremes (the start counts, at 0) and the extremes from every op on, packed
// as shorts; the route's extremes, start load and length into the CTA's words.
struct LsRoutes {
    int mn[32], mx[32], load[32], len[32];
};
__device__ __forceinline__ int pack_range(int mn, int mx) { return (mn & 0xffff) | (mx << 16); }
__device__ __forceinline__ int range_lo(int p) { return static_cast<int>(static_cast<short>(p & 0xffff)); }
__device__ __forceinline__ int range_hi(int p) { return p >> 16; }

__device__ void ls_scan_route(const AlnsTeam& t, const Smem& s, int r, int* S, int* PM, int* SM, LsRoutes* R) {
    const int lane = threadIdx.x & 31, st = s.sWoff[r], en = s.sWoff[r + 1];
    int carry = 0, cmin = 0, cmax = 0, len = 0;
    for (int base = st; base < en; base += 32) {
        const int k = base + lane;
        const bool in = k < en;
        const int x = in ? s.sW[k] : 0;
        int v = in ? ((x & 1) ? 1 : -1) : 0;
        len += x >> PACK_SHIFT;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL_MASK, v, o);
            if (lane >= o) v += y;
        }
        const int sv = carry + v;
        int mn = in ? sv : INT32_MAX, mx = in ? sv : INT32_MIN;
        for (int o = 1; o < 32; o <<= 1) {
            const int y1 = __shfl_up_sync(FULL_MASK, mn, o), y2 = __shfl_up_sync(FULL_MASK, mx, o);
            if (lane >= o) { mn = min(mn, y1); mx = max(mx, y2); }
        }
        mn = min(mn, cmin);
        mx = max(mx, cmax);
        if (in) { S[k] = sv; PM[k] = pack_range(mn, mx); }
        carry = __shfl_sync(FULL_MASK, sv, 31);
        cmin = __shfl_sync(FULL_MASK, mn, 31);
        cmax = __shfl_sync(FULL_MASK, mx, 31);
    }
    __syncwarp();
    int smn = INT32_MAX, smx = INT32_MIN;
    for (int top = en - 1; top >= st; top -= 32) {
        const int k = top - lane;
        const bool in = k >= st;
        const int sv = in ? S[k] : 0;
        int mn = in ? sv : INT32_MAX, mx = in ? sv : INT32_MIN;
        for (int o = 1; o < 32; o <<= 1) {
            const int y1 = __shfl_up_sync(FULL_MASK, mn, o), y2 = __shfl_up_sync(FULL_MASK, mx, o);
            if (lane >= o) { mn = min(mn, y1); mx = max(mx, y2); }
        }
        mn = min(mn, smn);
        mx = max(mx, smx);
        if (in) SM[k] = pack_range(mn, mx);
        smn = __shfl_sync(FULL_MASK, mn, 31);
        smx = __shfl_sync(FULL_MASK, mx, 31);
    }
    len = __reduce_add_sync(FULL_MASK, len);
    if (lane == 0) {
        R->mn[r] = cmin;
        R->mx[r] = cmax;
        R->load[r] = t.load_full ? t.Q : -cmin;
        R->len[r] = len + (en > st ? Dx(t, s, (s.sW[en - 1] & PACK_MASK) >> 1, 0) : 0);
    }
}

// A move's key: makespan and travel, then customer, drop gap and pickup gap
// (route and place in the solution without the customer; the order of gaps by
// flat index).
struct LsBest {
    unsigned long long hi = KEY_NONE, lo = KEY_NONE;
    __device__ __forceinline__ void take(int z, int tr, int c, int a, int ia, int b, int jb) {
        const unsigned long long h = (static_cast<unsigned long long>(static_cast<unsigned>(z)) << 32) | static_cast<unsigned>(tr);
        const unsigned long long l = (static_cast<unsigned long long>(c) << 34) |
                                     (static_cast<unsigned long long>((a << 12) | ia) << 17) |
                                     static_cast<unsigned long long>((b << 12) | jb);
        least(h, l);
    }
    __device__ __forceinline__ void least(unsigned long long h, unsigned long long l) {
        if (h < hi || (h == hi && l < lo)) { hi = h; lo = l; }
    }
};
// Gaps and pairs of gaps of one pass, per thread: decided by the formula or by a
// bound, decided through a shortcut gap, and of the first those scored.  What a
// bound rules out depends on how far the other CTAs are; the first two do not.
struct LsCounts {
    unsigned long long entries = 0, shortcut = 0;
    unsigned scored = 0;
};
// The least of all threads' keys, in thread 0 (sh: 2 u64 per warp).
__device__ void ls_block_least(LsBest& b, unsigned long long* sh) {
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long h = __shfl_xor_sync(FULL_MASK, b.hi, o), l = __shfl_xor_sync(FULL_MASK, b.lo, o);
        b.least(h, l);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        sh[2 * (threadIdx.x >> 5)] = b.hi;
        sh[2 * (threadIdx.x >> 5) + 1] = b.lo;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < ALNS_WARPS; ++w) b.least(sh[2 * w], sh[2 * w + 1]);
    __syncthreads();
}

// One candidate of pickup repositioning, the whole CTA.
__device__ void ls_pickup_item(const AlnsTeam& t, const Smem& s, int* scr, LsRoutes* rt, int c, LsBest& best,
                               LsCounts& count) {
    const int n = t.n, m = t.m, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, N0 = 2 * n;
    const int rw = ((n + 1) + 3) & ~3;
    const uint16_t* place = reinterpret_cast<const uint16_t*>(t.gains);
    const int pd = place[2 * c], pp = place[2 * c + 1], zcur = t.ctl->z_cur;
    int *H = scr, *T = H + N0, *S = T + N0, *PM = S + N0, *SM = PM + N0, *list = SM + N0;   // (an empty route has no shortcut gap: at most 2N)
    int* sh = s.misc + 32;                     // makespan, shortcut gaps
    __syncthreads();                           // the previous item is done with the staged solution
    stage_without(t, s, pp, -1);
    const int N = N0 - 1, G = N + m, d1 = pd - (pp < pd ? 1 : 0);
    if (tid == 0) sh[1] = 0;
    if (warp == 0) {
        const int z = walk_heads(t, s, s.rdy, H);
        if (lane == 0) sh[0] = z;
    } else if (warp == 1) {
        walk_tails(t, s, s.rdy + rw, T, c, d1);
    } else {
        for (int r = warp - 2; r < m; r += ALNS_WARPS - 2) ls_scan_route(t, s, r, S, PM, SM, rt);
    }
    __syncthreads();
    const int z1 = sh[0], hp = H[d1] + s.sp[c];
    int a = 0, p = 0, sumL = 0, len = 0;
    for (int v = 0; v < m; ++v) {
        if (t.cur_off[v] <= pd) a = v;
        if (t.cur_off[v] <= pp) p = v;
        sumL += rt->load[v];
        len += rt->len[v];
    }
    const int ia = pd - t.cur_off[a];
    int tmp = 0;
    const bool okA = cap_ok(t, rt->mn[a], rt->mx[a], tmp);
    // the pickup's old route, left over capacity, has to take it back
    const int only = p != a && !cap_ok(t, rt->mn[p], rt->mx[p], tmp) ? p : -1;
    auto gap_of = [&](int g, int* pos) {
        int lo = 0, hi = m;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s.sWoff[mid] + mid <= g) lo = mid; else hi = mid;
        }
        *pos = g - (s.sWoff[lo] + lo);
        return lo;
    };
    auto cust = [&](int k) { return (s.sW[k] & PACK_MASK) >> 1; };
    for (int g = tid; g < G; g += ALNS_THREADS) {
        int pos;
        const int r = gap_of(g, &pos), off = s.sWoff[r], L = s.sWoff[r + 1] - off;
        if ((only >= 0 && r != only) || (r == a && off + pos <= d1) || (r != a && !okA)) continue;
        const int xo = pos > 0 ? off + pos - 1 : -1, yo = pos < L ? off + pos : -1;
        const int Ty = yo >= 0 ? T[yo] : 0;
        if (Ty > TAIL_BITS) continue;          // the pickup would come before an op that leads to its drop
        const int pm = xo >= 0 ? PM[xo] : 0, sb = xo >= 0 ? S[xo] : 0;
        int mn = range_lo(pm), mx = max(range_hi(pm), sb + 1);
        if (yo >= 0) {
            const int sm = SM[yo];
            mn = min(mn, range_lo(sm) + 1);
            mx = max(mx, range_hi(sm) + 1);
        }
        int lb = 0;
        if (!cap_ok(t, mn, mx, lb) || sumL - rt->load[r] + lb > t.R) continue;
        const int x = xo >= 0 ? cust(xo) : 0, y = yo >= 0 ? cust(yo) : 0;
        const int dxc = Dx(t, s, x, c), dcy = Dx(t, s, c, y), w = L == 0 ? 0 : Dx(t, s, x, y);
        if (dxc + dcy < w) {
            list[atomicAdd(&sh[1], 1)] = g;
            continue;
        }
        ++count.entries;
        ++count.scored;
        const int zn = max(z1, max((xo >= 0 ? H[xo] : 0) + dxc, hp) + dcy + Ty);
        if (zn < zcur) best.take(zn, len + dxc + dcy - w, c, a, ia, r, pos - (r == a ? 1 : 0));
    }
    __syncthreads();
    const int ns = sh[1];
    int* rdy = s.rdy + warp * rw;
    for (int k = warp; k < ns; k += ALNS_WARPS) {
        int pos;
        const int r = gap_of(list[k], &pos), off = s.sWoff[r], L = s.sWoff[r + 1] - off;
        for (int q = lane; q <= n; q += 32) rdy[q] = UNRES;
        __syncwarp();
        const int zn = walk_fwd(t, s, rdy, r, pos, 2 * c + 1, -1, 0, 0, nullptr, nullptr);
        const int x = pos > 0 ? cust(off + pos - 1) : 0, y = pos < L ? cust(off + pos) : 0;
        if (lane == 0) {
            ++count.shortcut;
            if (zn < zcur)
                best.take(zn, len + Dx(t, s, x, c) + Dx(t, s, c, y) - Dx(t, s, x, y), c, a, ia, r, pos - (r == a ? 1 : 0));
        }
    }
}

// One candidate of relocation onto the vehicles part, part + split, ..., the whole CTA.
__device__ void ls_relocate_item(const AlnsTeam& t, const Smem& s, int* scr, LsRoutes* rt, int c, int part, int split,
                                 LsBest& best, LsCounts& count) {
    const int n = t.n, m = t.m, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, N0 = 2 * n;
    const int rw = ((n + 1) + 3) & ~3;
    const uint16_t* place = reinterpret_cast<const uint16_t*>(t.gains);
    const int pd = place[2 * c], pp = place[2 * c + 1], zcur = t.ctl->z_cur, bott = t.ctl->ls_bott, pc = s.sp[c];
    int *H = scr, *T = H + N0, *S = T + N0, *PM = S + N0, *SM = PM + N0, *gC = SM + N0, *list = gC + N0 + 4;
    constexpr int SCUT = INT32_MIN;            // gC: a shortcut gap; SKIPV: one that cannot matter; else its path
    int* sh = s.misc + 32;                     // makespan, largest shortcut, gaps that matter, their least travel, bound, shortcut gaps
    // what the whole team's moves of this pass have reached: nothing above it
    // can be the pass's move
    volatile unsigned long long* bound = &t.ctl->ls_bound;
    unsigned long long published = best.hi;
    auto publish = [&]() {
        if (best.hi < published) {
            published = best.hi;
            atomicMin(&t.ctl->ls_bound, published);
        }
    };
    __syncthreads();                           // the previous item is done with the staged solution
    stage_without(t, s, min(pd, pp), max(pd, pp));
    if (warp == 0) {
        const int z = walk_heads(t, s, s.rdy, H);
        if (lane == 0) sh[0] = z;
    } else if (warp == 1) {
        walk_tails(t, s, s.rdy + rw, T, 0, -1);
    } else {
        for (int r = warp - 2; r < m; r += ALNS_WARPS - 2) ls_scan_route(t, s, r, S, PM, SM, rt);
    }
    __syncthreads();
    const int z = sh[0], dcc = Dx(t, s, c, c);
    int sumL = 0, len = 0;
    unsigned bad = 0;
    for (int v = 0; v < m; ++v) {
        int l = 0;
        sumL += rt->load[v];
        len += rt->len[v];
        if (!cap_ok(t, rt->mn[v], rt->mx[v], l)) bad |= 1u << v;
    }
    auto cust = [&](int k) { return (s.sW[k] & PACK_MASK) >> 1; };
    int* rdy_ = s.rdy + warp * rw;
    volatile int* rdy = rdy_;
    for (int v = part; v < m; v += split) {
        if (v == bott || (bad & ~(1u << v)) != 0u) continue;   // uniform over the CTA
        const int off = s.sWoff[v], L = s.sWoff[v + 1] - off;
        struct Gap { int Hx, Ty, dxc, dcy, w; };
        auto gap = [&](int i) {
            Gap g;
            const int x = i > 0 ? cust(off + i - 1) : 0, y = i < L ? cust(off + i) : 0;
            g.Hx = i > 0 ? H[off + i - 1] : 0;
            g.Ty = i < L ? T[off + i] : 0;
            g.dxc = Dx(t, s, x, c);
            g.dcy = Dx(t, s, c, y);
            g.w = L == 0 ? 0 : Dx(t, s, x, y);
            return g;
        };
        auto fits = [&](int mn, int mx) {
            int l = 0;
            return cap_ok(t, mn, mx, l) && sumL - rt->load[v] + l <= t.R;
        };
        // both ops into gap i
        auto fits_adjacent = [&](int i) {
            const int pm = i > 0 ? PM[off + i - 1] : 0, sb = i > 0 ? S[off + i - 1] : 0;
            int mn = min(range_lo(pm), sb - 1), mx = range_hi(pm);
            if (i < L) {
                mn = min(mn, range_lo(SM[off + i]));
                mx = max(mx, range_hi(SM[off + i]));
            }
            return fits(mn, mx);
        };
        __syncthreads();                       // the previous route is done with gC, the list and the words
        if (tid == 0) {
            sh[1] = 0;
            sh[2] = 0;
            sh[3] = INT32_MAX;
            sh[4] = static_cast<int>(min(*bound >> 32, 0x7fffffffull));
            sh[5] = 0;
        }
        __syncthreads();
        for (int i = tid; i <= L; i += ALNS_THREADS) {
            const Gap g = gap(i);
            const int cut = g.w - g.dxc - g.dcy;
            if (cut > 0) {
                atomicMax(&sh[1], cut);
                atomicAdd(&sh[5], 1);
            }
            gC[i] = cut > 0 ? SCUT : g.Hx + g.dxc + g.dcy + g.Ty;
        }
        __syncthreads();
        if (tid == 0) {                        // every pair of the route's gaps, whatever a bound leaves out below
            const unsigned long long gaps = L + 1, plain = gaps - sh[5];
            count.entries += plain * (plain + 1) / 2;
            count.shortcut += gaps * (gaps + 1) / 2 - plain * (plain + 1) / 2;
        }
        // a path through two shortcut gaps loses at most both
        const int cut = sh[1];
        if (z - 2 * cut >= zcur || z - 2 * cut > sh[4]) continue;
        for (int i = tid; i <= L; i += ALNS_THREADS) {
            const int gc = gC[i];
            const Gap g = gap(i);
            if (gc != SCUT) {
                const int zn = max(z, g.Hx + g.dxc + max(dcc, pc) + g.dcy + g.Ty);
                ++count.scored;
                if (zn < zcur && fits_adjacent(i)) best.take(zn, len + g.dxc + dcc + g.dcy - g.w, c, v, i, v, i);
                if (gc - cut >= zcur) {
                    gC[i] = SKIPV;
                    continue;
                }
            }
            list[atomicAdd(&sh[2], 1)] = i;
            atomicMin(&sh[3], g.dxc + g.dcy - g.w);
        }
        publish();
        __syncthreads();
        const int nv = sh[2], least = sh[3];
        for (int k = warp; k < nv; k += ALNS_WARPS) {
            const int i = list[k];
            const bool si = gC[i] == SCUT;
            const Gap gi = gap(i);
            // no entry of this row is below (row's path less a shortcut, its travel and
            // the least of another gap)
            const int floor_z = max(z - 2 * cut, si ? 0 : gC[i] - cut);
            const int floor_t = max(0, len + gi.dxc + gi.dcy - gi.w + (si ? min(least, 0) : least));
            const unsigned long long reached = __shfl_sync(FULL_MASK, *bound, 0);
            if (((static_cast<unsigned long long>(static_cast<unsigned>(max(0, floor_z))) << 32) |
                 static_cast<unsigned>(floor_t)) > reached)
                continue;
            const int pmi = i > 0 ? PM[off + i - 1] : 0, sbi = i > 0 ? S[off + i - 1] : 0;
            bool walk = false;
            for (int q = 0; q < nv; ++q) {
                const int j = list[q];
                if (j < i || (j == i && !si)) continue;
                const int gc = gC[j];
                if (!si && gc != SCUT) { walk = true; continue; }
                // a shortcut on either side: simulated
                const Gap gj = gap(j);
                bool ok;
                if (i == j) {
                    ok = fits_adjacent(i);
                } else {
                    int mn = INT32_MAX, mx = INT32_MIN;
                    for (int e = off + i + lane; e < off + j; e += 32) { mn = min(mn, S[e]); mx = max(mx, S[e]); }
                    mn = __reduce_min_sync(FULL_MASK, mn);
                    mx = __reduce_max_sync(FULL_MASK, mx);
                    mn = min(min(range_lo(pmi), sbi - 1), mn - 1);
                    mx = max(max(range_hi(pmi), mx - 1), S[off + j - 1]);
                    if (j < L) {
                        mn = min(mn, range_lo(SM[off + j]));
                        mx = max(mx, range_hi(SM[off + j]));
                    }
                    ok = fits(mn, mx);
                }
                if (!ok) continue;
                const int zn = walk_insert(t, s, rdy_, c, v, i, v, j);
                if (lane == 0) {
                    const int di = gi.dxc + gi.dcy - gi.w;
                    if (zn < zcur)
                        best.take(zn, len + (i == j ? gi.dxc + dcc + gi.dcy - gi.w : di + gj.dxc + gj.dcy - gj.w), c, v, i, v, j);
                }
            }
            if (!walk) continue;
            // W from op y_i on: the longest path from it to every op of the route
            const int u = off + i, row = max(z, gC[i]);
            for (int q = lane; q <= n; q += 32) rdy[q] = UNRES;
            __syncwarp();
            int pos = lane < m ? s.sWoff[lane] : 0, val = NEG, sv = sbi, mn = INT32_MAX, mx = INT32_MIN;
            const int end = lane < m ? s.sWoff[lane + 1] : 0;
            int x = pos < end ? s.sW[pos] : 0;
            for (;;) {
                const bool on = pos < end, at = pos == u;
                const int cc = (x & PACK_MASK) >> 1, nx = pos + 1 < end ? s.sW[pos + 1] : 0;
                const bool pick = (x & 1) != 0;
                const int r = on && pick && !at ? rdy[cc] : 0;
                const bool go = on && (!pick || at || r != UNRES);
                if (go) {
                    val = at ? 0 : max(val == NEG ? NEG : val + (x >> PACK_SHIFT), pick ? r : NEG);
                    if (!pick) rdy[cc] = val == NEG ? NEG : val + s.sp[cc];
                    if (lane == v && pos >= u) {
                        sv += pick ? 1 : -1;
                        mn = min(mn, sv);
                        mx = max(mx, sv);
                        const int j = pos + 1 - off, gc = gC[j];
                        if (gc != SCUT && gc != SKIPV) {
                            const Gap gj = gap(j);
                            ++count.scored;
                            const int zn = max(max(row, gc), max(gi.Hx + gi.dxc + pc + gj.dcy + gj.Ty,
                                                                 gi.Hx + gi.dxc + gi.dcy + val + gj.dxc + gj.dcy + gj.Ty));
                            if (zn < zcur) {
                                int lo = min(min(range_lo(pmi), sbi - 1), mn - 1), hi = max(max(range_hi(pmi), mx - 1), sv);
                                if (j < L) {
                                    lo = min(lo, range_lo(SM[off + j]));
                                    hi = max(hi, range_hi(SM[off + j]));
                                }
                                if (fits(lo, hi))
                                    best.take(zn, len + gi.dxc + gi.dcy - gi.w + gj.dxc + gj.dcy - gj.w, c, v, i, v, j);
                            }
                        }
                    }
                    x = nx;
                    ++pos;
                }
                __syncwarp();
                if (!__any_sync(FULL_MASK, go) || __shfl_sync(FULL_MASK, pos >= end, v)) break;
            }
            publish();
        }
    }
}

// One pass, every CTA of the team between two barriers: its share of the
// candidates, the CTA's least key to its record.
__device__ __noinline__ void ls_pass(const AlnsTeam& t, const Smem& s, int rank, int team_blocks, int mode) {
    const int active = ls_active(t, team_blocks);
    if (rank >= active) return;
    AlnsCtl* ctl = t.ctl;
    const int ncand = *reinterpret_cast<volatile int*>(&ctl->ls_ncand);
    int* scr = ls_scratch(t, rank);
    LsRoutes* rt = reinterpret_cast<LsRoutes*>(s.rowv);
    LsBest best;
    LsCounts count;
    if (mode == LS_PICKUP) {
        for (int k = rank; k < ncand; k += active) ls_pickup_item(t, s, scr, rt, t.lscand[k], best, count);
    } else {
        const int split = max(1, min(t.m - 1, active / max(ncand, 1)));
        for (int k = rank; k < ncand * split; k += active)
            ls_relocate_item(t, s, scr, rt, t.lscand[k / split], k % split, split, best, count);
    }
    unsigned long long we = count.entries, wf = count.shortcut, ws = count.scored;
    for (int o = 16; o > 0; o >>= 1) {
        we += __shfl_xor_sync(FULL_MASK, we, o);
        wf += __shfl_xor_sync(FULL_MASK, wf, o);
        ws += __shfl_xor_sync(FULL_MASK, ws, o);
    }
    if ((threadIdx.x & 31) == 0) {             // (thread 0 holds a route's entries, the others their scores: modulo 2^64)
        if (we) atomicAdd(&ctl->entries, we);
        if (we != ws) atomicAdd(&ctl->pruned, we - ws);
        if (wf) atomicAdd(&ctl->fallback_entries, wf);
    }
    ls_block_least(best, reinterpret_cast<unsigned long long*>(s.colv));
    if (threadIdx.x == 0) {
        unsigned long long* rec = reinterpret_cast<unsigned long long*>(t.scpair) + 2 * rank;
        rec[0] = best.hi;
        rec[1] = best.lo;
    }
}

// Rank 0 at the end of a pass: apply the least move (all in the records lower
// the makespan).
__device__ __noinline__ void ls_apply(const AlnsTeam& t, const Smem& s, int team_blocks) {
    AlnsCtl* ctl = t.ctl;
    const int active = ls_active(t, team_blocks);
    const unsigned long long* rec = reinterpret_cast<const unsigned long long*>(t.scpair);
    LsBest best;
    for (int k = threadIdx.x; k < active; k += ALNS_THREADS) best.least(__ldcg(rec + 2 * k), __ldcg(rec + 2 * k + 1));
    unsigned long long* sh = reinterpret_cast<unsigned long long*>(s.colv);
    ls_block_least(best, sh);
    if (threadIdx.x == 0) { sh[0] = best.hi; sh[1] = best.lo; }
    __syncthreads();
    const unsigned long long hi = sh[0], lo = sh[1];
    const bool go = hi != KEY_NONE;
    if (go) {
        const int c = static_cast<int>(lo >> 34), drop = static_cast<int>(lo >> 17) & 0x1ffff, pick = static_cast<int>(lo) & 0x1ffff;
        for (int x = threadIdx.x; x <= t.n; x += blockDim.x) s.flags[x] = x == c ? 1 : 0;
        if (threadIdx.x == 0) ctl->wsel = 0;
        __syncthreads();
        build_W_from_cur(t, s);
        stage_W(t, s);
        __syncthreads();
        insert_staged(t, s, c, drop >> 12, drop & 0xfff, pick >> 12, pick & 0xfff, t.cur_ops, t.cur_off);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        ctl->ls_moved = go ? 1 : 0;
        if (go) {
            ctl->z_cur = static_cast<int>(hi >> 32);
            ctl->ls_moves += 1;
        }
    }
    __syncthreads();
}

// Rank 0 after the local search of iteration it: the trace and the best solution.
__device__ __noinline__ void ls_finish(const AlnsTeam& t, const Smem& s, int it) {
    AlnsCtl* ctl = t.ctl;
    int* flag = s.misc;
    if (threadIdx.x == 0) {
        flag[0] = ctl->z_cur < ctl->z_best ? 1 : 0;
        if (flag[0]) {
            ctl->z_best = ctl->z_cur;
            ctl->stagnation = 0;
            ctl->ls_new_best += 1;
        }
        if (t.trace && it > 0) t.trace[it - 1] = ctl->z_cur;
    }
    __syncthreads();
    if (flag[0]) {
        for (int k = threadIdx.x; k < 2 * t.n; k += blockDim.x) t.best_ops[k] = t.cur_ops[k];
        for (int v = threadIdx.x; v <= t.m; v += blockDim.x) t.best_off[v] = t.cur_off[v];
    }
    __syncthreads();
}

// The local search of one iteration (it = 0: outside the iterations), every
// CTA of the team: up to three passes of each mode in lsm, pickup
// repositioning first.  False when a team barrier gave up.
__device__ __noinline__ bool ls_block(const AlnsTeam& t, const Smem& s, int rank, int team_blocks, unsigned& gen, int lsm, int it) {
    AlnsCtl* ctl = t.ctl;
    for (int mode = LS_PICKUP; mode <= LS_RELOCATE; ++mode) {
        if (!(lsm & mode)) continue;
        for (int pass = 0; pass < 3; ++pass) {
            if (rank == 0) ls_candidates(t, s, mode);
            if (!team_barrier(ctl, team_blocks, gen)) return false;
            ls_pass(t, s, rank, team_blocks, mode);
            if (!team_barrier(ctl, team_blocks, gen)) return false;
            if (rank == 0) ls_apply(t, s, team_blocks);
            if (!team_barrier(ctl, team_blocks, gen)) return false;
            if (!*reinterpret_cast<volatile int*>(&ctl->ls_moved)) break;
        }
    }
    if (rank == 0) ls_finish(t, s, it);
    return team_barrier(ctl, team_blocks, gen);
}

// The team barrier after the matrix phase, with the selection folded in: the
// CTA that arrives last (every tile and shortcut item of the step is then
// done and visible) selects and applies the insertion before it releases the
// others, so a greedy step crosses one barrier here instead of two.  Bounded
// like team_barrier; false when a wait gave up.
__device__ bool team_barrier_select(const AlnsTeam& t, const Smem& s, int team_blocks, unsigned& gen) {
    AlnsCtl* ctl = t.ctl;
    __syncthreads();
    if (team_blocks == 1) {
        phase_select(t, s);
        __syncthreads();
        return *reinterpret_cast<volatile int*>(&ctl->err) == 0;
    }
    const bool last = __syncthreads_or(threadIdx.x == 0 && arrive_last(ctl, team_blocks));
    bool failed = false;
    if (last) {
        phase_select(t, s);
        __syncthreads();
        if (threadIdx.x == 0) failed = !release_team(ctl, gen);
    } else if (threadIdx.x == 0) {
        failed = !await_release(ctl, gen);
    }
    gen += 1u;
    return !__syncthreads_or(failed);
}

__global__ void __launch_bounds__(ALNS_THREADS, 3) alns_kernel(AlnsTeam* teams, int team_blocks) {
    extern __shared__ __align__(16) int smem_alns[];
    __shared__ AlnsTeam team_s;
    const int team = blockIdx.x / team_blocks, rank = blockIdx.x - team * team_blocks;
    if (threadIdx.x == 0) team_s = teams[team];
    __syncthreads();
    const AlnsTeam& t = team_s;
    AlnsCtl* ctl = t.ctl;
    const Smem s = carve(smem_alns, t.n, t.m);   // coordinates follow the flags when staged
    for (int c = threadIdx.x; c <= t.n; c += blockDim.x) s.sp[c] = t.p[c];
    if (t.coords)
        for (int i = threadIdx.x; i < 2 * (t.n + 1); i += blockDim.x) s.xy[i] = t.coords[i];
    if (threadIdx.x < 4) s.counts[threadIdx.x] = 0ull;
    unsigned gen = 0, ggen = 0;
    __syncthreads();

    if (t.mode == 1) {
        // one-customer matrix dump on the partial solution already in W[0]
        if (!team_barrier(ctl, team_blocks, gen)) return;
        phase_prep(t, s, rank, team_blocks, false, true);
        if (!team_barrier(ctl, team_blocks, gen)) return;
        phase_gaps(t, s, rank, team_blocks);
        team_arrive(ctl, team_blocks, gen);
        gap_walks(t, s, rank, team_blocks);
        if (!team_wait(ctl, team_blocks, gen)) return;
        if (!phase_matrix(t, s, rank, team_blocks)) return;
        team_barrier(ctl, team_blocks, gen);
        return;
    }
    if (t.mode == 3) {
        // repair steps on the partial solution already in W[0] (the search's
        // own step: prep, incrementally after a non-shortcut insertion, gaps,
        // shortcut walks, matrix, selection), then the matrix of the first
        // customer still to insert written out as in mode 1
        if (!team_barrier(ctl, team_blocks, gen)) return;
        for (int step = 0; step <= t.dump_steps; ++step) {
            if (*reinterpret_cast<volatile int*>(&ctl->repair_fail) || *reinterpret_cast<volatile int*>(&ctl->nrem) == 0)
                return;
            const bool incr = *reinterpret_cast<volatile int*>(&ctl->incr) != 0;
            if (rank == 0 && threadIdx.x == 0) {
                if (incr) ctl->steps_incr += 1; else ctl->steps_full += 1;
            }
            phase_prep(t, s, rank, team_blocks, incr, step == 0);
            if (incr) {
                __syncthreads();
                if (threadIdx.x == 0) {
                    int* q = team_s.H; team_s.H = team_s.H2; team_s.H2 = q;
                    q = team_s.T; team_s.T = team_s.T2; team_s.T2 = q;
                    q = team_s.Ms; team_s.Ms = team_s.Ms2; team_s.Ms2 = q;
                }
                __syncthreads();
            }
            if (!team_barrier(ctl, team_blocks, gen)) return;
            phase_gaps(t, s, rank, team_blocks);
            team_arrive(ctl, team_blocks, gen);
            gap_walks(t, s, rank, team_blocks);
            if (!team_wait(ctl, team_blocks, gen)) return;
            if (step == t.dump_steps) {
                __syncthreads();
                if (threadIdx.x == 0) team_s.mode = 1;
                __syncthreads();
                if (!phase_matrix(t, s, rank, team_blocks)) return;
                team_barrier(ctl, team_blocks, gen);
                return;
            }
            if (!phase_matrix(t, s, rank, team_blocks)) return;
            if (!team_barrier_select(t, s, team_blocks, gen)) return;
        }
        return;
    }
    // start: W = cur, evaluate
    if (rank == 0) {
        for (int k = threadIdx.x; k < 2 * t.n; k += blockDim.x) t.W_ops[0][k] = t.cur_ops[k];
        for (int v = threadIdx.x; v <= t.m; v += blockDim.x) t.W_off[0][v] = t.cur_off[v];
        if (threadIdx.x == 0) ctl->wsel = 0;
        __syncthreads();
        phase_end(t, s, true);
        if (t.mode == 0 && (t.destroy_mask & (1 << D_WORST))) worst_weights(t, s);
    }
    if (!team_barrier(ctl, team_blocks, gen)) return;
    if (t.mode == 2) {
        // refinement of a start solution: local-search rounds until one moves nothing
        for (int round = 0; round < t.refine_rounds; ++round) {
            const int before = *reinterpret_cast<volatile int*>(&ctl->ls_moves);
            if (!ls_block(t, s, rank, team_blocks, gen, LS_PICKUP | LS_RELOCATE, 0)) return;
            if (*reinterpret_cast<volatile int*>(&ctl->ls_moves) == before) break;
        }
        return;
    }
    // wall time per phase, read by rank 0 at each barrier exit
    uint64_t tmark = global_ns();
    auto mark = [&](int ph) {
        if (rank == 0 && threadIdx.x == 0) {
            const uint64_t now = global_ns();
            ctl->phase_ns[ph] += now - tmark;
            tmark = now;
        }
    };
    for (int it = 1; it <= t.iterations; ++it) {
        if (*reinterpret_cast<volatile int*>(&ctl->di) == D_WORST) {
            // worst removal needs every customer's removal gain: a team phase
            phase_gains(t, s, rank, team_blocks);
            if (!team_barrier(ctl, team_blocks, gen)) return;
        }
        if (rank == 0) {
            if (threadIdx.x == 0) ctl->iter = it;
            __syncthreads();
            phase_begin(t, s);
        }
        if (!team_barrier(ctl, team_blocks, gen)) return;
        mark(0);
        bool fresh = true;
        while (true) {
            const int nrem = *reinterpret_cast<volatile int*>(&ctl->nrem);
            const int fail = *reinterpret_cast<volatile int*>(&ctl->repair_fail);
            const bool incr = *reinterpret_cast<volatile int*>(&ctl->incr) != 0;
            if (nrem == 0 || fail) break;
            if (rank == 0 && threadIdx.x == 0) {
                if (incr) ctl->steps_incr += 1; else ctl->steps_full += 1;
            }
            phase_prep(t, s, rank, team_blocks, incr, fresh);
            fresh = false;
            if (incr) {
                // every CTA swaps its own copy of the pointers: the update wrote the second buffers
                __syncthreads();
                if (threadIdx.x == 0) {
                    int* q = team_s.H; team_s.H = team_s.H2; team_s.H2 = q;
                    q = team_s.T; team_s.T = team_s.T2; team_s.T2 = q;
                    q = team_s.Ms; team_s.Ms = team_s.Ms2; team_s.Ms2 = q;
                }
                __syncthreads();
            }
            if (!team_barrier(ctl, team_blocks, gen)) return;
            mark(1);
            phase_gaps(t, s, rank, team_blocks);
            team_arrive(ctl, team_blocks, gen);
            gap_walks(t, s, rank, team_blocks);
            if (!team_wait(ctl, team_blocks, gen)) return;
            mark(2);
            if (!phase_matrix(t, s, rank, team_blocks)) return;
            if (!team_barrier_select(t, s, team_blocks, gen)) return;   // select runs inside
            mark(3);
            mark(4);
        }
        if (rank == 0) phase_end(t, s, false);
        if (!team_barrier(ctl, team_blocks, gen)) return;
        mark(5);
        const int lsm = (t.ls_pickup > 0 && it % t.ls_pickup == 0 ? LS_PICKUP : 0) |
                        (t.ls_relocate > 0 && it % t.ls_relocate == 0 ? LS_RELOCATE : 0);
        if (lsm) {
            if (!ls_block(t, s, rank, team_blocks, gen, lsm, it)) return;
            mark(6);
        }
        if (t.nreplicas > 1 && t.sync_every > 0 && it % t.sync_every == 0) {
            if (!grid_barrier(t, ggen)) return;
            if (rank == 0) replica_import(t, s);
            if (!grid_barrier(t, ggen)) return;
        }
    }
    if (threadIdx.x == 0) {
        if (s.counts[0]) atomicAdd(&ctl->entries, s.counts[0]);
        if (s.counts[1]) atomicAdd(&ctl->pruned, s.counts[1]);
        if (s.counts[2]) atomicAdd(&ctl->tiles, s.counts[2]);
        if (s.counts[3]) atomicAdd(&ctl->tiles_pruned, s.counts[3]);
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct DevBuf {
    char* base = nullptr;
    size_t used = 0, cap = 0;
    template <class T>
    T* take(size_t count) {
        size_t bytes = (count * sizeof(T) + 255) & ~static_cast<size_t>(255);
        T* p = reinterpret_cast<T*>(base + used);
        used += bytes;
        return p;
    }
};

static size_t team_bytes(int n, int m, int qmax, int iterations, bool dump) {
    const size_t N = 2ull * n, G = N + m;
    int levels = 1;
    while ((1ull << levels) <= N) ++levels;
    size_t w = 0;
    auto add = [&](size_t count, size_t sz) { w += (count * sz + 255) & ~static_cast<size_t>(255); };
    add(1, sizeof(AlnsCtl));
    add(N, 4); add(m + 1, 4); add(N, 4); add(m + 1, 4);
    add(N + 2, 4); add(m + 1, 4); add(N + 2, 4); add(m + 1, 4);
    add(std::max<size_t>(n + 1, qmax), 4);
    add(N, 4); add(N, 4); add(N * N, 4);
    add(N, 4); add(N, 4); add(N * N, 4);
    for (int i = 0; i < 5; ++i) add(N, 4);
    add(levels * N, 4); add(levels * N, 4);
    for (int i = 0; i < 10; ++i) add(G, 4);
    add(m, 4);
    add(G * 16, 4); add(G * 12, 4);
    add(static_cast<size_t>(qmax) * G, 16); add(static_cast<size_t>(qmax) * G, 16);
    if (dump) add(static_cast<size_t>(qmax) * G, 8);
    add(static_cast<size_t>(qmax) * G, 8);
    add(static_cast<size_t>(qmax) * 32, 8);
    add(static_cast<size_t>(qmax) * 4, 8);
    add(static_cast<size_t>(qmax) * ((G + 31) / 32), 16);
    add(tile_words(static_cast<int>(G)), 4);
    add(static_cast<size_t>(qmax) * G, 1);
    add(static_cast<size_t>(qmax) * G, 4);
    add(static_cast<size_t>(qmax) * G, 4);
    add(static_cast<size_t>(SC_CAP) * (4 * N + 8), 4);
    add(static_cast<size_t>(SC_CAP) * SC_CAP, 4);
    add(std::max(iterations, 1), 4);
    add(n + 1, 8);
    add(n + 1, 4);
    add(n + 1, 4);
    if (dump) { add(G * G, 4); add(G * G, 4); }
    return w;
}

static void carve_team(AlnsTeam& t, DevBuf& B, int n, int m, int qmax, int iterations, bool dump) {
    const size_t N = 2ull * n, G = N + m;
    int levels = 1;
    while ((1ull << levels) <= N) ++levels;
    t.ctl = B.take<AlnsCtl>(1);
    t.cur_ops = B.take<int>(N); t.cur_off = B.take<int>(m + 1);
    t.best_ops = B.take<int>(N); t.best_off = B.take<int>(m + 1);
    t.W_ops[0] = B.take<int>(N + 2); t.W_off[0] = B.take<int>(m + 1);
    t.W_ops[1] = B.take<int>(N + 2); t.W_off[1] = B.take<int>(m + 1);
    t.rem = B.take<int>(std::max(n + 1, qmax));
    t.H = B.take<int>(N); t.T = B.take<int>(N); t.Ms = B.take<int>(N * N);
    t.H2 = B.take<int>(N); t.T2 = B.take<int>(N); t.Ms2 = B.take<int>(N * N);
    t.S_ = B.take<int>(N); t.PMINp = B.take<int>(N); t.PMAXp = B.take<int>(N);
    t.SMINs = B.take<int>(N); t.SMAXs = B.take<int>(N);
    t.spmin = B.take<int>(levels * N); t.spmax = B.take<int>(levels * N);
    t.log_levels = levels;
    t.gx = B.take<int>(G); t.gy = B.take<int>(G);
    t.gw = B.take<int>(G); t.gsb = B.take<int>(G); t.gpmin = B.take<int>(G); t.gpmax = B.take<int>(G);
    t.gsmin = B.take<int>(G); t.gsmax = B.take<int>(G); t.groute = B.take<int>(G); t.gpos = B.take<int>(G);
    t.rload = B.take<int>(m);
    t.growc = B.take<int>(G * 16); t.gcolc = B.take<int>(G * 12);
    t.vrow = B.take<int4>(static_cast<size_t>(qmax) * G); t.vcol = B.take<int4>(static_cast<size_t>(qmax) * G);
    t.vadj = dump ? B.take<int2>(static_cast<size_t>(qmax) * G) : nullptr;
    t.keys = B.take<unsigned long long>(static_cast<size_t>(qmax) * G);
    t.rkeys = B.take<unsigned long long>(static_cast<size_t>(qmax) * 32);
    t.gmin = B.take<unsigned long long>(static_cast<size_t>(qmax) * 4);
    t.band_stride = qmax;
    t.bands = B.take<int4>(static_cast<size_t>(qmax) * ((G + 31) / 32));
    t.tmask = B.take<unsigned>(tile_words(static_cast<int>(G)));
    t.sc = B.take<unsigned char>(static_cast<size_t>(qmax) * G);
    t.slist = B.take<int>(static_cast<size_t>(qmax) * G);
    t.scix = B.take<int>(static_cast<size_t>(qmax) * G);
    t.scw_stride = static_cast<int>(4 * N + 8);
    t.graph_warps = graph_warps(n);
    t.scw = B.take<int>(static_cast<size_t>(SC_CAP) * (4 * N + 8));
    t.scpair = B.take<int>(static_cast<size_t>(SC_CAP) * SC_CAP);
    t.trace = B.take<int>(std::max(iterations, 1));
    t.pw = B.take<double>(n + 1);
    t.gains = B.take<int>(n + 1);
    t.lscand = B.take<int>(n + 1);
    t.dump_delta = dump ? B.take<int>(G * G) : nullptr;
    t.dump_travel = dump ? B.take<int>(G * G) : nullptr;
}

// Rows of the per-customer buffers: a route removal takes a whole route, so
// with that operator on, up to n customers wait for reinsertion at once.
int alns_row_cap(int n, int m, int qmax, const vrprpd_alns_params* P) {
    int cap = (P->destroy_mask & (1 << D_ROUTE)) ? n : qmax;
    return std::max(cap, 1);
}

// ALNS CTAs one SM holds for an instance of n customers and m vehicles (its
// shared memory with staged coordinates, the larger layout); 0 if none fits.
int alns_blocks_per_sm(int n, int m) {
    if (ensure_smem_limit(reinterpret_cast<const void*>(&alns_kernel))) return 0;
    int occ = 0;
    const size_t smem = alns_smem_words(n, m, true) * 4;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, alns_kernel, ALNS_THREADS, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return occ;
}

size_t alns_device_bytes(int n, int m, int qmax, const vrprpd_alns_params* P, int iterations) {
    const size_t R = static_cast<size_t>(std::max(1, P->replicas));
    return R * (team_bytes(n, m, alns_row_cap(n, m, qmax, P), iterations, false) + sizeof(AlnsTeam)) + 8192;
}

bool alns_supported(const vrprpd_instance* I, std::string* why) {
    if (I->m > 32) { *why = "ALNS needs m <= 32"; return false; }
    if (2 * I->n + I->m > 4096) { *why = "ALNS needs 2n + m <= 4096"; return false; }
    if (I->maxd >= (1 << 17)) { *why = "ALNS needs max d < 2^17"; return false; }
    // every schedule time of every insertion the matrix scores stays below
    // 2^27, so sums of three of them next to the exclusion sentinel fit int32
    const long long bound = (2ll * I->n + 1) * I->maxd + static_cast<long long>(I->n) * I->maxp;
    if (bound >= (1ll << 27)) { *why = "ALNS needs (2n+1)*max(d) + n*max(p) < 2^27"; return false; }
    return true;
}

static int choose_team_blocks(const vrprpd_instance* I, int requested, size_t smem, int nteams, int* out) {
    int occ = 0;
    { int rc_ = ensure_smem_limit(reinterpret_cast<const void*>(&alns_kernel)); if (rc_) return rc_; }
    VRP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, alns_kernel, ALNS_THREADS, smem));
    VRP_CHECK(occ > 0, VRPRPD_EINVAL, "ALNS block does not fit on an SM (n=%d)", I->n);
    // every CTA of every team is resident at once (a cooperative launch)
    const int maxb = occ * I->num_sms / nteams;
    VRP_CHECK(maxb >= 1, VRPRPD_EINVAL, "%d replicas exceed the %d resident ALNS blocks of this GPU", nteams,
              occ * I->num_sms);
    int tb = requested;
    if (tb <= 0) {
        // about one tile of the first step's matrix per CTA, at least one CTA
        const long long G = 2ll * I->n + I->m;
        const long long tiles = ((G + TR - 1) / TR) * ((G + TC - 1) / TC);
        tb = static_cast<int>(std::min<long long>(tiles, maxb));
        if (G < 64) tb = 1;
    }
    *out = std::max(1, std::min(tb, maxb));
    return VRPRPD_OK;
}

static int launch_alns(const vrprpd_instance* I, AlnsTeam* d_teams, int nteams, int team_blocks, size_t smem,
                       cudaStream_t stream) {
    void* args[] = {&d_teams, &team_blocks};
    const int grid = nteams * team_blocks;
    if (grid > 1) {
        VRP_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&alns_kernel), dim3(grid),
                                             dim3(ALNS_THREADS), args, smem, stream));
    } else {
        alns_kernel<<<grid, ALNS_THREADS, smem, stream>>>(d_teams, team_blocks);
        VRP_CUDA(cudaGetLastError());
    }
    return VRPRPD_OK;
}

}  // namespace vrp

using namespace vrp;

extern "C" void vrprpd_alns_params_default(vrprpd_alns_params* P) {
    if (!P) return;
    P->T0 = 0.30;
    P->alpha = 0.9998;
    P->reheat = 0.50;
    P->r = 0.1;
    P->stagnation = 2000;
    P->tau = 100;
    P->sigma1 = 33;
    P->sigma2 = 9;
    P->sigma3 = 13;
    P->w_min = 0.1;
    P->q_min = 0;
    P->q_max = 0;
    P->iterations = 1000;
    P->repair_mask = 3;
    P->team_blocks = 0;
    P->destroy_mask = 1;
    P->ls_pickup_every = 200;
    P->ls_relocate_every = 500;
    P->replicas = 1;
    P->sync_every = 1000;
    P->init_mode = 1;
    P->init_refine_rounds = 10;
    P->wait_limit_ns = 2000000000ll;
}

// exact angular order around the depot: half plane, then cross product, then id
static bool angle_less(const std::vector<int32_t>& xy, int a, int b) {
    const long long ax = xy[2 * a] - xy[0], ay = xy[2 * a + 1] - xy[1];
    const long long bx = xy[2 * b] - xy[0], by = xy[2 * b + 1] - xy[1];
    const int ha = (ay < 0 || (ay == 0 && ax < 0)) ? 1 : 0, hb = (by < 0 || (by == 0 && bx < 0)) ? 1 : 0;
    if (ha != hb) return ha < hb;
    const long long cr = ax * by - ay * bx;
    if (cr != 0) return cr > 0;
    return a < b;
}

extern "C" int vrprpd_initial_solution(const vrprpd_instance* I, vrprpd_solution* out) {
    VRP_CHECK(I && out && out->ops && out->off, VRPRPD_EINVAL, "NULL argument");
    VRP_CHECK(I->R >= 1 && I->Q >= 1, VRPRPD_EINVAL, "initial solution needs R >= 1 and Q >= 1");
    const int n = I->n, m = I->m, N1 = n + 1;
    std::vector<int> order(n);
    for (int k = 0; k < n; ++k) order[k] = k + 1;
    if (I->has_coords)
        std::sort(order.begin(), order.end(), [&](int a, int b) { return angle_less(I->h_coords, a, b); });
    const int mact = std::min(m, I->R);
    const int b = std::max(1, std::min(I->Q, I->R / mact));
    long long W = 0;
    for (int k = 0; k < n; ++k) W += 2ll * I->h_d[order[k]] + I->h_p[order[k]];
    std::vector<int> sector(n);
    long long cum = 0;
    for (int k = 0; k < n; ++k) {
        const long long w = 2ll * I->h_d[order[k]] + I->h_p[order[k]];
        long long s = W > 0 ? ((2 * cum + w) * mact) / (2 * W) : (static_cast<long long>(k) * mact) / n;
        sector[k] = static_cast<int>(std::min<long long>(s, mact - 1));
        cum += w;
    }
    (void)N1;
    int w = 0;
    out->off[0] = 0;
    for (int v = 0; v < m; ++v) {
        std::vector<int> mine;
        for (int k = 0; k < n; ++k)
            if (sector[k] == v) mine.push_back(order[k]);
        for (size_t s = 0; s < mine.size(); s += b) {
            const size_t e = std::min(mine.size(), s + b);
            for (size_t q = s; q < e; ++q) out->ops[w++] = 2 * mine[q];
            for (size_t q = s; q < e; ++q) out->ops[w++] = 2 * mine[q] + 1;
        }
        out->off[v + 1] = w;
    }
    out->makespan = 0;
    out->status = 0;
    return VRPRPD_OK;
}

// Mode 3 (repair steps, then a matrix dump): the customers to insert, the
// repair operator, the steps, and where the partial solution goes afterwards.
struct RepairDump {
    int steps, op, count;
    const int32_t* removed;
    int32_t* out_ops;
    int32_t* out_off;
};

static int run_team(const vrprpd_instance* I, const vrprpd_solution* init, const vrprpd_alns_params* P,
                    uint64_t seed, int mode, int dump_c, const int32_t* dump_ops, const int32_t* dump_off,
                    vrprpd_solution* best, vrprpd_solution* current, vrprpd_alns_stats* stats, int32_t* trace,
                    int32_t* dump_delta, int32_t* dump_travel, cudaStream_t stream, int refine_rounds = 0,
                    const RepairDump* rd = nullptr) {
    std::string why;
    VRP_CHECK(alns_supported(I, &why), VRPRPD_EINVAL, "%s", why.c_str());
    const int n = I->n, m = I->m;
    int qmin = P->q_min, qmax = P->q_max;
    if (qmin <= 0 || qmax <= 0) {
        qmax = std::max(4, static_cast<int>(static_cast<long long>(n) * 5 / 100));
        qmin = std::max(4, qmax / 2);
    }
    qmax = std::min(qmax, n);
    qmin = std::min(qmin, qmax);
    VRP_CHECK(qmin >= 1 && qmax <= 1024, VRPRPD_EINVAL, "removal size must lie in [1, 1024] (q_min=%d q_max=%d)",
              qmin, qmax);
    const int iters = mode == 0 ? P->iterations : 0;
    VRP_CHECK(iters >= 0 && iters <= (1 << 24), VRPRPD_EINVAL, "iterations out of range");
    VRP_CHECK(P->tau >= 1, VRPRPD_EINVAL, "tau must be >= 1");
    VRP_CHECK(P->ls_pickup_every >= 0 && P->ls_relocate_every >= 0, VRPRPD_EINVAL,
              "local-search periods must be >= 0 (0 = off)");
    const bool dump = mode == 1 || mode == 3;
    const int R = mode != 0 ? 1 : std::max(1, P->replicas);
    VRP_CHECK(R <= 1024, VRPRPD_EINVAL, "replicas must lie in [0, 1024] (%d)", R);
    VRP_CHECK(P->sync_every >= 0, VRPRPD_EINVAL, "sync_every must be >= 0 (0 = never)");
    const int qcap = mode == 3 ? std::max(1, rd->count) : dump ? 1 : alns_row_cap(n, m, qmax, P);
    DevBuf B;
    const size_t per_team = team_bytes(n, m, qcap, iters, dump);
    B.cap = per_team * R + 4096;
    VRP_CUDA(pool_alloc(reinterpret_cast<void**>(&B.base), B.cap, stream));
    auto cleanup = [&]() { cudaFreeAsync(B.base, stream); };
    unsigned* gbar = B.take<unsigned>(4);
    AlnsTeam* d_team = nullptr;
    cudaError_t e = pool_alloc(reinterpret_cast<void**>(&d_team), sizeof(AlnsTeam) * R, stream);
    if (e != cudaSuccess) { cleanup(); set_error("alns setup: %s", cudaGetErrorString(e)); return VRPRPD_ECUDA; }
    AlnsTeam t{};
    t.n = n;
    t.m = m;
    t.R = I->R;
    t.Q = I->Q;
    t.load_full = (I->flags & VRPRPD_LOAD_FULL) != 0;
    t.d32 = I->d32;
    t.p = I->p;
    t.coords = coords_exact_small(I) ? I->coords : nullptr;
    t.T0 = P->T0;
    t.alpha = P->alpha;
    t.reheat = P->reheat;
    t.r = P->r;
    t.w_min = P->w_min;
    t.stagnation_limit = P->stagnation;
    t.tau = P->tau;
    t.sigma1 = P->sigma1;
    t.sigma2 = P->sigma2;
    t.sigma3 = P->sigma3;
    t.q_min = qmin;
    t.q_max = qmax;
    t.iterations = iters;
    t.repair_mask = P->repair_mask & 15;
    t.destroy_mask = P->destroy_mask & 63;
    t.ls_pickup = dump ? 0 : P->ls_pickup_every;
    t.ls_relocate = dump ? 0 : P->ls_relocate_every;
    auto fail_all = [&](int code) { cleanup(); cudaFreeAsync(d_team, stream); return code; };
    if (t.destroy_mask == 0) { set_error("destroy_mask enables no destroy operator"); return fail_all(VRPRPD_EINVAL); }
    if (t.repair_mask == 0) { set_error("repair_mask enables no repair operator"); return fail_all(VRPRPD_EINVAL); }
    t.mode = mode;
    t.refine_rounds = refine_rounds;
    t.dump_c = dump_c;
    t.dump_steps = mode == 3 ? rd->steps : 0;
    t.nreplicas = R;
    t.sync_every = P->sync_every;
    t.gbar = gbar;
    t.sib = d_team;
    // replica r draws from its own stream: the single-run stream for r = 0,
    // else a draw of it far past any iteration's counters
    const uint64_t key0 = stream_key(seed, RNG_STREAM_ALNS);
    std::vector<AlnsTeam> ts(R, t);
    for (int r = 0; r < R; ++r) {
        ts[r].replica = r;
        ts[r].key = r == 0 ? key0 : draw(key0, (0xFFFFFFFFull << 32) + static_cast<uint64_t>(r));
        carve_team(ts[r], B, n, m, qcap, iters, dump);
    }
    AlnsCtl ctl{};
    ctl.wait_ns = P->wait_limit_ns > 0 ? static_cast<unsigned long long>(P->wait_limit_ns) : 2000000000ull;
    for (int i = 0; i < 8; ++i) ctl.wd[i] = 1.0;
    ctl.wr[0] = ctl.wr[1] = ctl.wr[2] = ctl.wr[3] = 1.0;
    if (dump) {
        ctl.nrem = mode == 3 ? rd->count : 1;
        ctl.rj = mode == 3 ? rd->op : 0;
        ctl.wsel = 0;
    }
    e = cudaMemsetAsync(gbar, 0, 16, stream);
    for (int r = 0; r < R && e == cudaSuccess; ++r) e = cudaMemcpyAsync(ts[r].ctl, &ctl, sizeof(ctl), cudaMemcpyHostToDevice, stream);
    std::vector<int32_t> init_ops(2 * n), init_off(m + 1);
    if (!dump) {
        if (init) {
            std::memcpy(init_ops.data(), init->ops, 2 * n * 4);
            std::memcpy(init_off.data(), init->off, (m + 1) * 4);
        } else {
            vrprpd_solution s0{init_ops.data(), init_off.data(), 0, 0};
            const int rc = P->init_mode == 1
                               ? initial_solution_paper_tb(I, P->init_refine_rounds, &s0, stream, P->team_blocks)
                               : vrprpd_initial_solution(I, &s0);
            if (rc) return fail_all(rc);
        }
        for (int r = 0; r < R && e == cudaSuccess; ++r) {
            e = cudaMemcpyAsync(ts[r].cur_ops, init_ops.data(), 2 * n * 4, cudaMemcpyHostToDevice, stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(ts[r].cur_off, init_off.data(), (m + 1) * 4, cudaMemcpyHostToDevice, stream);
        }
    } else {
        const int Nops = dump_off[m];
        if (e == cudaSuccess) e = cudaMemcpyAsync(ts[0].W_ops[0], dump_ops, std::max(Nops, 1) * 4, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(ts[0].W_off[0], dump_off, (m + 1) * 4, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess)
            e = mode == 3 ? cudaMemcpyAsync(ts[0].rem, rd->removed, rd->count * 4, cudaMemcpyHostToDevice, stream)
                          : cudaMemcpyAsync(ts[0].rem, &dump_c, 4, cudaMemcpyHostToDevice, stream);
        const size_t G = static_cast<size_t>(Nops) + (mode == 3 ? 2 * rd->steps : 0) + m;
        if (e == cudaSuccess) e = cudaMemsetAsync(ts[0].dump_delta, 0xff, G * G * 4, stream);
    }
    // recompute distances from staged coordinates only when that costs no resident CTAs
    size_t smem = alns_smem_words(n, m, false) * 4;
    if (t.coords) {
        const size_t smem_c = alns_smem_words(n, m, true) * 4;
        int occ0 = 0, occ1 = 0;
        ensure_smem_limit(reinterpret_cast<const void*>(&alns_kernel));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ0, alns_kernel, ALNS_THREADS, smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ1, alns_kernel, ALNS_THREADS, smem_c);
        if (occ1 >= occ0 && smem_c <= I->smem_optin) smem = smem_c;
        else for (auto& x : ts) x.coords = nullptr;
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_team, ts.data(), sizeof(AlnsTeam) * R, cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) {
        set_error("alns setup: %s", cudaGetErrorString(e));
        return fail_all(VRPRPD_ECUDA);
    }
    if (smem > I->smem_optin) {
        set_error("ALNS shared memory %zu exceeds the limit", smem);
        return fail_all(VRPRPD_EINVAL);
    }
    int tb = 1;
    int rc = choose_team_blocks(I, P->team_blocks, smem, R, &tb);
    if (rc) return fail_all(rc);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, stream);
    rc = launch_alns(I, d_team, R, tb, smem, stream);
    cudaEventRecord(e1, stream);
    if (rc) return fail_all(rc);
    e = cudaStreamSynchronize(stream);
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    std::vector<AlnsCtl> out(R);
    for (int r = 0; r < R && e == cudaSuccess; ++r) e = cudaMemcpyAsync(&out[r], ts[r].ctl, sizeof(AlnsCtl), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
        set_error("alns run: %s", cudaGetErrorString(e));
        return fail_all(VRPRPD_ECUDA);
    }
    for (int r = 0; r < R; ++r) {
        if (out[r].err != 0) {
            set_error("alns device error %d (%s)", out[r].err,
                      out[r].err == DEV_TIMEOUT_BARRIER ? "team barrier timed out" : "inconsistent state");
            return fail_all(out[r].err == DEV_TIMEOUT_BARRIER ? VRPRPD_ETIMEOUT : VRPRPD_ECUDA);
        }
    }
    // the best of all replicas, the lowest index on ties; replica 0 reports
    // the current solution, the temperature and the weights
    int g = 0;
    for (int r = 1; r < R; ++r)
        if (out[r].z_best < out[g].z_best) g = r;
    if (mode == 3 && out[0].repair_fail) {
        set_error("a customer has no feasible insertion during the repair steps");
        return fail_all(VRPRPD_EINVAL);
    }
    if (dump) {
        const int Nout = dump_off[m] + (mode == 3 ? 2 * rd->steps : 0);
        const size_t G = static_cast<size_t>(Nout) + m;
        e = cudaMemcpyAsync(dump_delta, ts[0].dump_delta, G * G * 4, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess && mode == 3) {
            const int w = out[0].wsel;
            e = cudaMemcpyAsync(rd->out_ops, ts[0].W_ops[w], std::max(Nout, 1) * 4, cudaMemcpyDeviceToHost, stream);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(rd->out_off, ts[0].W_off[w], (m + 1) * 4, cudaMemcpyDeviceToHost, stream);
        }
        if (e == cudaSuccess && dump_travel) e = cudaMemcpyAsync(dump_travel, ts[0].dump_travel, G * G * 4, cudaMemcpyDeviceToHost, stream);
    } else {
        if (best) {
            e = cudaMemcpyAsync(best->ops, ts[g].best_ops, 2 * n * 4, cudaMemcpyDeviceToHost, stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(best->off, ts[g].best_off, (m + 1) * 4, cudaMemcpyDeviceToHost, stream);
            best->makespan = out[g].z_best;
            best->status = 0;
        }
        if (current && e == cudaSuccess) {
            e = cudaMemcpyAsync(current->ops, ts[0].cur_ops, 2 * n * 4, cudaMemcpyDeviceToHost, stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(current->off, ts[0].cur_off, (m + 1) * 4, cudaMemcpyDeviceToHost, stream);
            current->makespan = out[0].z_cur;
            current->status = 0;
        }
        for (int r = 0; r < R && trace && e == cudaSuccess && iters > 0; ++r)
            e = cudaMemcpyAsync(trace + static_cast<size_t>(r) * iters, ts[r].trace, iters * 4, cudaMemcpyDeviceToHost, stream);
    }
    if (stats) {
        std::memset(stats, 0, sizeof(*stats));
        stats->iterations = iters;
        for (int r = 0; r < R; ++r) {
            const AlnsCtl& o = out[r];
            stats->accepted += o.accepted;
            stats->improved += o.improved;
            stats->new_best += o.new_best;
            stats->reheats += o.reheats;
            stats->rejected_infeasible += o.rejected;
            stats->matrix_entries += static_cast<int64_t>(o.entries);
            stats->fallback_entries += static_cast<int64_t>(o.fallback_entries);
            stats->pruned_entries += static_cast<int64_t>(o.pruned);
            stats->tiles += static_cast<int64_t>(o.tiles);
            stats->tiles_pruned += static_cast<int64_t>(o.tiles_pruned);
            stats->incremental_steps += static_cast<int64_t>(o.steps_incr);
            stats->full_steps += static_cast<int64_t>(o.steps_full);
            stats->ls_moves += o.ls_moves;
            stats->ls_new_best += o.ls_new_best;
            stats->imports += o.imports;
        }
        stats->z_init = out[0].z_init;
        stats->z_best = out[g].z_best;
        stats->z_current = out[0].z_cur;
        stats->T_final = out[0].T;
        for (int i = 0; i < 8; ++i) stats->w_destroy[i] = i < ND_OPS ? out[0].wd[i] : 0.0;
        for (int i = 0; i < 4; ++i) stats->w_repair[i] = out[0].wr[i];
        stats->device_ms = ms;
        stats->team_blocks = tb;
        for (int i = 0; i < 6; ++i) stats->phase_ms[i] = static_cast<double>(out[0].phase_ns[i]) * 1e-6;
        stats->ls_ms = static_cast<double>(out[0].phase_ns[6]) * 1e-6;
        stats->replicas = R;
        stats->best_replica = g;
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    cleanup();
    cudaFreeAsync(d_team, stream);
    if (e != cudaSuccess) {
        set_error("alns copy-out: %s", cudaGetErrorString(e));
        return VRPRPD_ECUDA;
    }
    return VRPRPD_OK;
}

extern "C" int vrprpd_initial_solution_paper(const vrprpd_instance* I, int32_t refine_rounds, vrprpd_solution* out,
                                             void* stream_) {
    return initial_solution_paper_tb(I, refine_rounds, out, static_cast<cudaStream_t>(stream_), 0);
}

namespace vrp {

int initial_solution_paper_tb(const vrprpd_instance* I, int32_t refine_rounds, vrprpd_solution* out,
                              cudaStream_t stream, int team_blocks) {
    VRP_CHECK(I && out && out->ops && out->off, VRPRPD_EINVAL, "NULL argument");
    VRP_CHECK(refine_rounds >= 0, VRPRPD_EINVAL, "refine_rounds must be >= 0");
    std::string why;
    VRP_CHECK(alns_supported(I, &why), VRPRPD_EINVAL, "%s", why.c_str());
    const int n = I->n, m = I->m;
    int32_t* dops = nullptr;
    VRP_CUDA(pool_alloc(reinterpret_cast<void**>(&dops), (2 * n + m + 1) * 4, stream));
    int32_t* doff = dops + 2 * n;
    int rc = construct_paper_device(I, dops, doff, stream);
    cudaError_t e = cudaSuccess;
    if (!rc) {
        e = cudaMemcpyAsync(out->ops, dops, 2 * n * 4, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(out->off, doff, (m + 1) * 4, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    }
    cudaFreeAsync(dops, stream);
    if (rc) return rc;
    if (e != cudaSuccess) {
        set_error("initial solution: %s", cudaGetErrorString(e));
        return VRPRPD_ECUDA;
    }
    // evaluation and refinement in the ALNS kernel (refine-only mode)
    vrprpd_alns_params P;
    vrprpd_alns_params_default(&P);
    P.team_blocks = team_blocks;
    std::vector<int32_t> io(out->ops, out->ops + 2 * n), of(out->off, out->off + m + 1);
    vrprpd_solution start{io.data(), of.data(), 0, 0};
    return run_team(I, &start, &P, 0, 2, 0, nullptr, nullptr, nullptr, out, nullptr, nullptr, nullptr, nullptr,
                    stream, refine_rounds);
}

}  // namespace vrp

extern "C" int vrprpd_alns_run(const vrprpd_instance* I, const vrprpd_solution* init, const vrprpd_alns_params* P,
                               uint64_t seed, vrprpd_solution* best, vrprpd_solution* current,
                               vrprpd_alns_stats* stats, int32_t* z_trace, void* stream) {
    VRP_CHECK(I && P && best && best->ops && best->off, VRPRPD_EINVAL, "NULL argument");
    int rc = run_team(I, init, P, seed, 0, 0, nullptr, nullptr, best, current, stats, z_trace, nullptr, nullptr,
                      static_cast<cudaStream_t>(stream));
    return rc;
}

extern "C" int vrprpd_repair_then_matrix(const vrprpd_instance* I, const int32_t* ops, const int32_t* off,
                                         const int32_t* removed, int32_t count, int32_t repair_op, int32_t steps,
                                         int32_t team_blocks, int32_t* out_ops, int32_t* out_off, int32_t* delta,
                                         int32_t* travel, int64_t* incremental_steps, void* stream) {
    VRP_CHECK(I && ops && off && removed && out_ops && out_off && delta, VRPRPD_EINVAL, "NULL argument");
    const int m = I->m, n = I->n;
    VRP_CHECK(count >= 1 && count <= 1024, VRPRPD_EINVAL, "count must lie in [1, 1024]");
    VRP_CHECK(steps >= 0 && steps < count, VRPRPD_EINVAL, "steps must lie in [0, count)");
    VRP_CHECK(repair_op >= 0 && repair_op <= 3, VRPRPD_EINVAL, "repair_op must lie in [0, 3]");
    VRP_CHECK(off[0] == 0 && off[m] == 2 * (n - count), VRPRPD_EINVAL, "the partial solution must hold 2(n - count) ops");
    for (int v = 0; v < m; ++v) VRP_CHECK(off[v + 1] >= off[v], VRPRPD_EINVAL, "offsets decrease");
    std::vector<char> seen(2 * n + 2, 0);
    for (int k = 0; k < off[m]; ++k) {
        const int o = ops[k];
        VRP_CHECK(o >= 2 && o <= 2 * n + 1 && !seen[o], VRPRPD_EINVAL, "bad or repeated op %d", o);
        seen[o] = 1;
    }
    for (int k = 0; k < count; ++k) {
        const int c = removed[k];
        VRP_CHECK(c >= 1 && c <= n && (k == 0 || c > removed[k - 1]), VRPRPD_EINVAL,
                  "removed customers must be ascending ids in [1, n]");
        VRP_CHECK(!seen[2 * c] && !seen[2 * c + 1], VRPRPD_EINVAL, "customer %d is in the partial solution", c);
    }
    for (int q = 1; q <= n; ++q) VRP_CHECK(seen[2 * q] == seen[2 * q + 1], VRPRPD_EINVAL, "customer %d half present", q);
    vrprpd_alns_params P;
    vrprpd_alns_params_default(&P);
    P.team_blocks = team_blocks;
    RepairDump rd{steps, repair_op, count, removed, out_ops, out_off};
    vrprpd_alns_stats st;
    const int rc = run_team(I, nullptr, &P, 0, 3, 0, ops, off, nullptr, nullptr, &st, nullptr, delta, travel,
                            static_cast<cudaStream_t>(stream), 0, &rd);
    if (rc == VRPRPD_OK && incremental_steps) *incremental_steps = st.incremental_steps;
    return rc;
}

extern "C" int vrprpd_insertion_matrix(const vrprpd_instance* I, const int32_t* ops, const int32_t* off, int32_t c,
                                       int32_t* delta, int32_t* travel, void* stream) {
    VRP_CHECK(I && ops && off && delta, VRPRPD_EINVAL, "NULL argument");
    VRP_CHECK(c >= 1 && c <= I->n, VRPRPD_EINVAL, "customer %d out of range", c);
    const int m = I->m;
    VRP_CHECK(off[0] == 0 && off[m] >= 0 && off[m] <= 2 * I->n - 2, VRPRPD_EINVAL, "bad partial offsets");
    for (int v = 0; v < m; ++v) VRP_CHECK(off[v + 1] >= off[v], VRPRPD_EINVAL, "offsets decrease");
    std::vector<char> seen(2 * I->n + 2, 0);
    for (int k = 0; k < off[m]; ++k) {
        const int o = ops[k];
        VRP_CHECK(o >= 2 && o <= 2 * I->n + 1 && !seen[o], VRPRPD_EINVAL, "bad or repeated op %d", o);
        VRP_CHECK((o >> 1) != c, VRPRPD_EINVAL, "customer %d is already in the partial solution", c);
        seen[o] = 1;
    }
    for (int q = 1; q <= I->n; ++q) VRP_CHECK(seen[2 * q] == seen[2 * q + 1], VRPRPD_EINVAL, "customer %d half present", q);
    vrprpd_alns_params P;
    vrprpd_alns_params_default(&P);
    return run_team(I, nullptr, &P, 0, 1, c, ops, off, nullptr, nullptr, nullptr, nullptr, delta, travel,
                    static_cast<cudaStream_t>(stream));
}
