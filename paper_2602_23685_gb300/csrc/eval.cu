// Batched candidate evaluation (the repair's timing evaluation of Section
// 4.2.3 and the decoder's schedule simulation of Section 4.4.2, done exactly
// on the semantics of Section 3.1, Eqs. 7-23).
//
// Batched form: a persistent launch; the block stages the instance (distances
// or points, and the ready-row template) in shared memory with TMA bulk
// copies, and every warp owns a tile of candidates, one or two routes per lane
// (eval_tile below).
// Plain form: one thread per candidate, Kahn order over routes, scratch in
// global memory, distances from global memory.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "device_common.cuh"
#include "internal.h"

namespace vrp {

// Internal distance mode of VRPRPD_DIST_COORDS when every squared leg is below
// EUC2D_HALF2_LIMIT: points as pairs of fp16 integers.
constexpr int DIST_HALF2 = 6;

// Warps per block at most, by routes per lane (register budget 64 and 128).
__host__ __device__ constexpr int max_warps(int V) { return V == 1 ? 32 : 16; }

struct EvalArgs {
    const int32_t* ops;
    const uint16_t* ops16;   // the 16-bit form (ops/off unused then)
    const uint16_t* off16;
    const int32_t* off;
    int32_t* z;
    uint32_t* st;
    const int32_t* d32;
    const uint16_t* d16;
    const int32_t* coords;
    const uint32_t* xy;      // points as fp16 pairs (row_words of them), or null
    const int32_t* rowt;     // ready-row template, row_words words
    int* err;
    long long num;
    int n, m, R, Q;
    int load_full;
    int pool_full;    // load_full: the m full loads exceed R
    int prefetch;     // candidates in device memory: fetch the next tile's codes into L2
    int N;            // n + 1
    int K;            // candidates per tile
    int row_words;    // words of one ready row: n + 2 rounded up to 4
    // shared-memory layout, in 32-bit words
    int shared_words; // per-block instance data (distances or points, ready-row template)
    int dist_words;
    int a_words, ready_words, off_words, warp_words;
    int pts;          // many-instance launches: where the warp's region keeps the tile's points
};

// ---------------------------------------------------------------------------
// The walk.  A warp owns a tile of K candidates and walks all their routes in
// lock step, V routes per lane (32 V >= K m).  Shared memory per warp: the
// tile's op codes as 16 bits, one row of ready slots per candidate, the route
// offsets and four words of results per candidate.
//
//   stage   codes by 16-byte loads whatever the alignment (four in flight per
//           lane), saturated to [0, 2n+2] and packed to 16 bits; ready rows
//           copied from the block's template;
//   walk    one op per route and round; see below;
//   check   every customer's slot must have ended PICKED;
//   reduce  makespan, start loads and flags per candidate by shared atomics.
//
// What bounds it.  At n=1000 m=20 a candidate takes 1475 wavefronts of shared
// memory with one route per lane (1208 with two) and 6.1 k warp instructions
// (4.0 k), where the earlier kernels issued 9.9 k and 8.4 k: one route per lane
// runs at 81% of the issue slots and 72% of the shared-memory pipe, two routes
// at 54% and 61%, short of warps.  262144 candidates: 2861 us before (its best
// walk and shape), 1415 us now; n=100 m=4, 65536: 89 to 42 us; n=499 m=19,
// 65536, a quarter of them blocked: 348 to 179 us; 32 instances of 17 to 500
// customers, 4096 each: 298 to 137 us.
// Tried at n=1000: the round's loads a round earlier, between the two routes'
// steps (21% more instructions, 446 us against 365 us for 65536 candidates);
// legs computed after the round's loads (385); groups of two warps with a
// shared progress count in place of two routes per lane (365, and 187 against
// 172 us at n=499); eight code chunks in flight at 64 registers (spills, 486).
//
// Ready slots.  Slot c holds -(p_c + 1) until c's drop, the pickup-ready time
// T_drop + p_c until its pickup, then PICKED for good: a drop that finds PICKED
// stores nothing.  The slots of the depot (c = 0) and of code 2n+2 (c = n+1,
// where every code out of range ends up) start as PICKED, so nothing on them is
// ever ready.  A lane past its route's end holds code 1, "pick up at the depot":
// it never goes, its point is the depot, so the leg it computes is the way home,
// and no lane state says whether the route is still going on.
//
// A round with no progress in the whole warp ends the walk: every write of
// earlier rounds was visible to this one, so nothing can go later either.
// Routes that have not ended then are blocked.
//
// Validation without bookkeeping in the walk.  Let a candidate's offsets be in
// order (checked first).  If no route of it is blocked, 2n ops were walked.  A
// slot becomes PICKED only by a pickup of its customer, and a pickup goes only
// after a drop of the same customer: a drop stores nd - 1 - r, which is
// T_drop + p_c over the slot's first state and between -1 and nd over a ready
// time (nd >= r then; -1 is the first state of p_c = 0), and no nd + p_c wraps.
// (Every leg is one of the instance's, also to and from the point of code 2n+2,
// and no path through the walked ops passes one twice or adds a p_c twice, so
// times stay within the (2n+1) max d + n max p that an instance keeps below
// 2^31 - 1.)  So if every customer's slot ends PICKED, the 2n ops hold a drop
// and a pickup of each of the n customers and nothing else: a permutation.  If
// some slot does not, an op is repeated or out of range.  (Over PICKED the
// drop's sum would wrap, to a ready time or, a drop later, even to PICKED: with
// such drops stored, 2 3 2 3 4 6 passed for three customers at the depot with
// p = 0, 1, 1.)  A candidate with a blocked route gets the full check (range and
// a duplicate bitmap), which tells MALFORMED from CYCLE.  Whatever a repeated or
// foreign code does to the slots on the way stays inside its own candidate, and
// every route still ends: each round that goes on takes at least one op.
//
// Stock.  One word holds 2^14 - s above 2^14 + s (s the stock relative to the
// start, |s| <= 2n < 2^13), so one add moves both and one packed maximum keeps
// max(-s) and max(s).
// ---------------------------------------------------------------------------
constexpr int PICKED = static_cast<int>(0x80000000u);   // ready slot of a customer already picked up

constexpr unsigned STOCK0 = 0x40004000u;
constexpr int NOTE_NONE = (1 << 26) - 1;                 // a drop whose vehicle has no next op

__device__ __forceinline__ int lds_s32(unsigned addr) {
    int v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_s32_if(bool on, unsigned addr, int v) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %0, 0;\n\t"
        "@p st.shared.b32 [%1], %2;\n\t}" ::"r"(static_cast<unsigned>(on)),
        "r"(addr), "r"(v)
        : "memory");
}
// the 16-bit code at addr, or past the end code 1, a pickup at the depot
__device__ __forceinline__ int code_or_idle(unsigned addr, unsigned end) {
    int v;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.lt.u32 p, %1, %2;\n\t"
        "mov.u32 %0, 1;\n\t"
        "@p ld.shared.u16 %0, [%1];\n\t}"
        : "=&r"(v)
        : "r"(addr), "r"(end)
        : "memory");
    return v;
}
__device__ __forceinline__ unsigned pack_sat_u16(int lo, int hi) {
    unsigned r;
    asm("cvt.pack.sat.u16.s32 %0, %1, %2;" : "=r"(r) : "r"(hi), "r"(lo));
    return r;
}
__device__ __forceinline__ unsigned min_u16x2(unsigned a, unsigned b) {
    unsigned r;
    asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ unsigned max_u16x2(unsigned a, unsigned b) {
    unsigned r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// Where a route stands, and the leg to the next stop.  leg() returns the
// travel time plus BIAS (the fp32 form's rounding constant, folded into the
// departure time instead of subtracted per leg).
template <int DM>
struct Place {
    static constexpr int BIAS = 0;
    int row;                                   // c (n+1)
    static __device__ __forceinline__ Place of(const EvalArgs& a, const int32_t*, int c) {
        // code 2n+2 stands one past the matrix: the last customer's row and column will
        // do, its candidate is malformed
        return {min(c, a.n) * a.N};
    }
    static __device__ __forceinline__ int leg(const EvalArgs& a, const int32_t* sh, const Place& x, const Place&,
                                              int c) {
        const int at = x.row + min(c, a.n);
        if constexpr (DM == VRPRPD_DIST_SMEM32) return sh[at];
        else if constexpr (DM == VRPRPD_DIST_SMEM16) return reinterpret_cast<const uint16_t*>(sh)[at];
        else if constexpr (DM == VRPRPD_DIST_GLOBAL16) return __ldg(a.d16 + at);
        else return __ldg(a.d32 + at);
    }
};
template <>
struct Place<VRPRPD_DIST_COORDS> {             // any coordinates with squared legs below 2^24
    static constexpr int BIAS = 0;
    int2 p;
    static __device__ __forceinline__ Place of(const EvalArgs&, const int32_t* sh, int c) {
        return {reinterpret_cast<const int2*>(sh)[c]};
    }
    static __device__ __forceinline__ int leg(const EvalArgs&, const int32_t*, const Place& x, const Place& y, int) {
        return euc2d_small(x.p.x, x.p.y, y.p.x, y.p.y);
    }
};
template <>
struct Place<DIST_HALF2> {                     // squared legs below 2^21: see euc2d_half2
    static constexpr int BIAS = EUC2D_BIAS;
    unsigned p;                                // x, y as two fp16 integers
    static __device__ __forceinline__ Place of(const EvalArgs&, const int32_t* sh, int c) {
        return {reinterpret_cast<const unsigned*>(sh)[c]};
    }
    static __device__ __forceinline__ int leg(const EvalArgs&, const int32_t*, const Place& x, const Place& y, int) {
        return euc2d_half2(x.p, y.p);
    }
};

// A tile's codes on their way from global to shared memory: `total` of them
// (the first `head`, fewer than a 16-byte chunk holds, belong to what lies
// before the tile) from the 16-byte boundary `base`, as 16-byte loads; the
// first and last chunk code by code.  Shared memory gets them saturated to
// [0, 2n+2] and packed to 16 bits, head included.  A batch is SB chunks per
// lane, all in flight together.
template <bool W16, int SB>
struct CodeBatch {
    static constexpr int CPC = W16 ? 8 : 4;    // codes per chunk
    int4 raw[SB] = {};
    __device__ __forceinline__ void load(const char* base, int head, int total, int first) {
        const int lane = threadIdx.x & 31, chunks = (total + CPC - 1) / CPC;
#pragma unroll
        for (int u = 0; u < SB; ++u) {
            const int ck = first + 32 * u + lane;
            if (ck >= chunks) continue;
            if ((ck > 0 || head == 0) && (ck + 1) * CPC <= total) {
                raw[u] = __ldg(reinterpret_cast<const int4*>(base) + ck);
            } else {
                unsigned w[4] = {0, 0, 0, 0};
#pragma unroll
                for (int e = 0; e < CPC; ++e) {
                    const int i = ck * CPC + e;
                    if (i < head || i >= total) continue;
                    if constexpr (W16) w[e >> 1] |= static_cast<unsigned>(__ldg(reinterpret_cast<const uint16_t*>(base) + i)) << (16 * (e & 1));
                    else w[e] = __ldg(reinterpret_cast<const int32_t*>(base) + i);
                }
                raw[u] = make_int4(w[0], w[1], w[2], w[3]);
            }
        }
    }
    __device__ __forceinline__ void store(unsigned A, unsigned lim2, int total, int first) {
        const int lane = threadIdx.x & 31, chunks = (total + CPC - 1) / CPC;
#pragma unroll
        for (int u = 0; u < SB; ++u) {
            const int ck = first + 32 * u + lane;
            if (ck >= chunks) continue;
            if constexpr (W16) {
                const unsigned x = min_u16x2(raw[u].x, lim2), y = min_u16x2(raw[u].y, lim2);
                const unsigned z = min_u16x2(raw[u].z, lim2), w = min_u16x2(raw[u].w, lim2);
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(A + 16u * ck), "r"(x), "r"(y), "r"(z),
                             "r"(w) : "memory");
            } else {
                const unsigned x = min_u16x2(pack_sat_u16(raw[u].x, raw[u].y), lim2);
                const unsigned y = min_u16x2(pack_sat_u16(raw[u].z, raw[u].w), lim2);
                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(A + 8u * ck), "r"(x), "r"(y) : "memory");
            }
        }
    }
};

// One tile of up to K candidates of one instance, walked by one warp.  W is
// the warp's shared-memory region, sh the instance's distances or points and
// rowt the ready-row template (shared memory, or for many-instance launches
// global memory).
// COUNT: the coordination counts instead of makespan and status.  A drop also
// leaves, beside its ready slot, its vehicle and how much later than the ready
// time its vehicle reaches its next op (both known the moment it goes), so the
// pickup settles its customer by itself: 32768 candidates at n=200 m=6 in 92 us,
// where the kernel with one candidate per warp, four words per customer and
// legs from L2 (metrics.cu) takes 317 us.
template <int DM, bool W16, int V, bool COUNT>
__device__ __forceinline__ void eval_tile(const EvalArgs& a, const int32_t* sh, const int32_t* rowt, int32_t* W,
                                          long long t, long long next) {
    using P = Place<DM>;
    const int lane = threadIdx.x & 31;
    const int n = a.n, m = a.m, two_n = 2 * n, K = a.K, str4 = a.row_words >> 2;
    int32_t* ready = W + a.a_words;
    int32_t* soff = ready + (COUNT ? 2 : 1) * a.ready_words;
    int32_t* res = soff + a.off_words;         // [4][K]: return, load + 2^16 per overfull route, malformed, blocked
                                               // (COUNT: cross, interleaved, malformed, blocked)
    const unsigned note = 4u * static_cast<unsigned>(a.ready_words);   // from a ready slot to the drop's note
    const long long first = t * K;
    const int kt = static_cast<int>(min(static_cast<long long>(K), a.num - first));
    const unsigned lim2 = static_cast<unsigned>(two_n + 2) * 0x10001u;

    // ---- codes, offsets, result words, ready rows ----
    const void* src = W16 ? static_cast<const void*>(a.ops16 + first * two_n) : static_cast<const void*>(a.ops + first * two_n);
    const int head = static_cast<int>(reinterpret_cast<uintptr_t>(src) & 15u) / (W16 ? 2 : 4);
    const char* base = static_cast<const char*>(src) - head * (W16 ? 2 : 4);
    const int total = head + kt * two_n;
    const unsigned Abase = smem_u32(W), A = Abase + 2u * head;
    constexpr int SB = V == 1 ? 4 : 8;         // one-route kernels run at 64 registers, the others at 128
    CodeBatch<W16, SB> codes;
    codes.load(base, head, total, 0);
    for (int i = lane; i < kt * (m + 1); i += 32)
        soff[i] = W16 ? static_cast<int32_t>(__ldg(a.off16 + first * (m + 1) + i)) : __ldg(a.off + first * (m + 1) + i);
    for (int i = lane; i < 4 * K; i += 32) res[i] = 0;
    {
        const int4* from = reinterpret_cast<const int4*>(rowt);
        int4* dst = reinterpret_cast<int4*>(ready);
        if (str4 >= 32) {
            for (int i = lane; i < str4; i += 32) {
                const int4 v = from[i];
                for (int g = 0; g < kt; ++g) dst[g * str4 + i] = v;
            }
        } else {
            int s = lane % str4;
            const int step = 32 % str4;
            for (int i = lane; i < kt * str4; i += 32) {
                dst[i] = from[s];
                s += step;
                s -= s >= str4 ? str4 : 0;
            }
        }
    }
    for (int b = 0;;) {
        codes.store(Abase, lim2, total, b);
        b += 32 * SB;
        if (b * CodeBatch<W16, SB>::CPC >= total) break;
        codes.load(base, head, total, b);
    }
    if (next >= 0 && lane == 0) {
        // the next tile's codes on their way into L2 while this one is walked
        const uintptr_t p0 = reinterpret_cast<uintptr_t>(W16 ? static_cast<const void*>(a.ops16 + next * K * two_n)
                                                             : static_cast<const void*>(a.ops + next * K * two_n));
        const long long left = min(static_cast<long long>(K), a.num - next * K) * two_n * (W16 ? 2 : 4);
        const uintptr_t lo = (p0 + 15) & ~static_cast<uintptr_t>(15), hi = (p0 + left) & ~static_cast<uintptr_t>(15);
        if (hi > lo) l2_prefetch_bulk(lo, static_cast<unsigned>(hi - lo));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(W16 ? static_cast<const void*>(a.off16 + next * K * (m + 1))
                                                          : static_cast<const void*>(a.off + next * K * (m + 1))));
    }
    __syncwarp();

    // ---- the walk ----
    // Per route: the op in hand (code, its slot's address, its point, the leg
    // into it), the code after it, and where the one after that lies (ca).
    int dep[V], leg[V], code[V], ncode[V], cand[V];
    unsigned stock[V], ext[V], rbase[V], ca[V], ce[V], ad[V];
    int veh[V], prev[V], cross[V], inter[V];   // COUNT only
    bool live[V];
    P at[V];
#pragma unroll
    for (int s = 0; s < V; ++s) {
        const int vl = lane + 32 * s, c = vl / m, v = vl - c * m;
        live[s] = c < kt;
        cand[s] = live[s] ? c : 0;
        veh[s] = v;
        prev[s] = cross[s] = inter[s] = 0;
        int lo = 0, hi = 0;
        if (live[s]) {
            lo = soff[c * (m + 1) + v];
            hi = soff[c * (m + 1) + v + 1];
            if (lo < 0 || hi > two_n || lo > hi || (v == 0 && lo != 0) || (v == m - 1 && hi != two_n)) {
                res[2 * K + c] = 1;
                lo = hi = 0;
            }
        }
        rbase[s] = smem_u32(ready + cand[s] * a.row_words);
        const unsigned cbase = A + 2u * static_cast<unsigned>(cand[s] * two_n);
        ca[s] = cbase + 2u * static_cast<unsigned>(lo);
        ce[s] = cbase + 2u * static_cast<unsigned>(hi);
        dep[s] = -P::BIAS;
        stock[s] = ext[s] = STOCK0;
        const P depot = P::of(a, sh, 0);
        code[s] = code_or_idle(ca[s], ce[s]);
        ncode[s] = code_or_idle(ca[s] + 2u, ce[s]);
        ca[s] += 4u;
        const int c1 = code[s] >> 1;
        at[s] = P::of(a, sh, c1);
        leg[s] = P::leg(a, sh, depot, at[s], c1);
        ad[s] = rbase[s] + 4u * static_cast<unsigned>(c1);
    }
    for (;;) {
        bool any = false;
        int r[V], acode[V];
        P nat[V];
#pragma unroll
        for (int s = 0; s < V; ++s) {
            // every load of the round at its start: whether the op in hand is
            // ready, the next op's point, the code after that
            r[s] = lds_s32(ad[s]);
            nat[s] = P::of(a, sh, ncode[s] >> 1);
            acode[s] = code_or_idle(ca[s], ce[s]);
        }
#pragma unroll
        for (int s = 0; s < V; ++s) {
            // this round's op: a drop goes at once, a pickup once it is ready.  A
            // drop's slot is negative, so the same maximum serves both
            const bool pick = (code[s] & 1) != 0;
            const bool go = !pick || r[s] >= 0;
            const int nd = __viaddmax_s32(dep[s], leg[s], r[s]);
            const int c1 = ncode[s] >> 1;
            const int nleg = P::leg(a, sh, at[s], nat[s], c1);
            if constexpr (COUNT) {
                // (next arrival - ready) << 5 | vehicle; the arrival is T_drop + the
                // next leg, the ready time T_drop + p and the slot still -(p + 1)
                if (!pick) {
                    const int late = ncode[s] == 1 ? NOTE_NONE : nleg - P::BIAS + 1 + r[s];
                    sts_s32_if(true, ad[s] + note, static_cast<int>(static_cast<unsigned>(late) << 5) | veh[s]);
                } else if (go) {
                    const int w = lds_s32(ad[s] + note), late = w >> 5;
                    const bool same = (w & 31) == veh[s];
                    cross[s] += same ? 0 : 1;
                    inter[s] += (same ? prev[s] != (code[s] ^ 1) : late != NOTE_NONE && r[s] + late < nd) ? 1 : 0;
                }
                prev[s] = go ? code[s] : prev[s];
            }
            sts_s32_if(go && r[s] != PICKED, ad[s], pick ? PICKED : static_cast<int>(static_cast<unsigned>(nd) - 1u - static_cast<unsigned>(r[s])));
            any = any || go;
            if (go) {
                dep[s] = nd - P::BIAS;
                if constexpr (!COUNT) stock[s] += pick ? 0xffff0001u : 0x0000ffffu;
                code[s] = ncode[s];
                ncode[s] = acode[s];
                at[s] = nat[s];
                leg[s] = nleg;
                ad[s] = rbase[s] + 4u * static_cast<unsigned>(c1);
                ca[s] += 2u;
            }
            if constexpr (!COUNT) ext[s] = max_u16x2(ext[s], stock[s]);
        }
        __syncwarp();
        if (!__any_sync(FULL_MASK, any)) break;
    }
    bool some_blocked = false;
#pragma unroll
    for (int s = 0; s < V; ++s) {
        const bool blocked = ca[s] - 4u < ce[s];
        if (blocked) {
            some_blocked = true;
            res[3 * K + cand[s]] = 1;
            if constexpr (!COUNT)              // finish the stock of a blocked route
                for (unsigned q = ca[s] - 4u; q < ce[s]; q += 2u) {
                    stock[s] += (code_or_idle(q, ce[s]) & 1) ? 0xffff0001u : 0x0000ffffu;
                    ext[s] = max_u16x2(ext[s], stock[s]);
                }
        }
        if constexpr (COUNT) {
            if (cross[s]) atomicAdd(&res[cand[s]], cross[s]);
            if (inter[s]) atomicAdd(&res[K + cand[s]], inter[s]);
        } else if (live[s]) {
            const int up = static_cast<int>(ext[s] & 0xffffu) - 0x4000, down = static_cast<int>(ext[s] >> 16) - 0x4000;
            const bool over = a.load_full ? (down > a.Q || up > 0) : (down + up > a.Q);
            atomicMax(&res[cand[s]], dep[s] + leg[s]);
            atomicAdd(&res[K + cand[s]], (a.load_full ? 0 : down) + (over ? 0x10000 : 0));
        }
    }

    // ---- every customer picked up? ----
    {
        const int4* rows = reinterpret_cast<const int4*>(ready);
        for (int i = lane; i < kt * str4; i += 32) {
            const int4 v = rows[i];
            if (max(max(v.x, v.y), max(v.z, v.w)) != PICKED) res[2 * K + i / str4] |= 2;
        }
    }
    __syncwarp();
    if (__any_sync(FULL_MASK, some_blocked)) {
        // the full check of candidates with a blocked route, on the staged codes
        for (int g = 0; g < kt; ++g) {
            if (!res[3 * K + g] || (res[2 * K + g] & 1)) continue;   // uniform over the warp
            uint32_t* seen = reinterpret_cast<uint32_t*>(ready + g * a.row_words);
            for (int i = lane; i < (two_n + 2 + 31) / 32; i += 32) seen[i] = 0u;
            __syncwarp();
            bool bad = false;
            for (int e = lane; e < two_n; e += 32) {
                const int o = code_or_idle(A + 2u * static_cast<unsigned>(g * two_n + e), ~0u);
                bool dup = o < 2 || o > two_n + 1;
                if (!dup) {
                    const unsigned bit = 1u << (o & 31);
                    dup = (atomicOr(&seen[o >> 5], bit) & bit) != 0u;
                }
                bad = bad || dup;
            }
            bad = __any_sync(FULL_MASK, bad);
            if (lane == 0) res[2 * K + g] = bad ? 1 : 0;
            __syncwarp();
            if constexpr (COUNT) {
                // the cross count of a cycle: both vehicles of every customer by
                // its ops' places, now in the candidate's row
                if (bad) continue;
                int32_t* both = ready + g * a.row_words;
                const int32_t* F = soff + g * (m + 1);
                for (int c = lane; c <= n; c += 32) both[c] = 0;
                if (lane == 0) res[g] = 0;
                __syncwarp();
                for (int e = lane; e < two_n; e += 32) {
                    const int o = code_or_idle(A + 2u * static_cast<unsigned>(g * two_n + e), ~0u);
                    int lo = 0, hi = m;
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (F[mid] <= e) lo = mid; else hi = mid;
                    }
                    atomicXor(&both[o >> 1], lo);
                }
                __syncwarp();
                int nc = 0;
                for (int c = 1 + lane; c <= n; c += 32) nc += both[c] != 0 ? 1 : 0;
                nc = __reduce_add_sync(FULL_MASK, nc);
                if (lane == 0) res[g] = nc;
                __syncwarp();
            }
        }
    }

    // ---- results ----
    for (int g = lane; g < kt; g += 32) {
        if constexpr (COUNT) {
            const bool bad = res[2 * K + g] != 0;
            a.z[first + g] = bad ? -1 : res[g];
            a.st[first + g] = static_cast<uint32_t>(bad || res[3 * K + g] ? -1 : res[K + g]);
            continue;
        }
        const int load = res[K + g];
        int z = res[g], f = 0;
        if (load >> 16) f |= VRPRPD_VEH_CAP;
        if (a.load_full ? a.pool_full != 0 : (load & 0xffff) > a.R) f |= VRPRPD_POOL;
        if (res[3 * K + g]) { f |= VRPRPD_CYCLE; z = 0x7fffffff; }
        if (res[2 * K + g]) { z = 0x7fffffff; f = VRPRPD_MALFORMED; }
        a.z[first + g] = z;
        a.st[first + g] = static_cast<uint32_t>(f);
    }
    __syncwarp();
}

template <int DM, bool W16, int V, bool COUNT>
__global__ void __launch_bounds__(32 * max_warps(V)) eval_tiles_kernel(EvalArgs a) {
    extern __shared__ __align__(16) int32_t smem[];
    __shared__ __align__(8) uint64_t block_bar;
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;

    // ---- block-wide staging of the instance (TMA bulk copies) ----
    int32_t* sh = smem;                        // distances or points
    int32_t* rowt = smem + a.dist_words;       // ready-row template
    if (threadIdx.x == 0) {
        mbar_init(&block_bar, 1);
        unsigned dist_bytes = 0;
        if constexpr (DM == VRPRPD_DIST_SMEM32) dist_bytes = ((a.N * a.N * 4) + 15) & ~15;
        if constexpr (DM == VRPRPD_DIST_SMEM16) dist_bytes = ((a.N * a.N * 2) + 15) & ~15;
        if constexpr (DM == VRPRPD_DIST_COORDS) dist_bytes = ((a.N * 8) + 8 + 15) & ~15;
        const unsigned row_bytes = a.row_words * 4u;
        if constexpr (DM == DIST_HALF2) dist_bytes = row_bytes;
        mbar_arrive_expect_tx(&block_bar, dist_bytes + row_bytes);
        if constexpr (DM == VRPRPD_DIST_SMEM32) tma_bulk_g2s(sh, a.d32, dist_bytes, &block_bar);
        if constexpr (DM == VRPRPD_DIST_SMEM16) tma_bulk_g2s(sh, a.d16, dist_bytes, &block_bar);
        if constexpr (DM == VRPRPD_DIST_COORDS) tma_bulk_g2s(sh, a.coords, dist_bytes, &block_bar);
        if constexpr (DM == DIST_HALF2) tma_bulk_g2s(sh, a.xy, dist_bytes, &block_bar);
        tma_bulk_g2s(rowt, a.rowt, row_bytes, &block_bar);
    }
    __syncthreads();
    if (!mbar_wait_bounded(&block_bar, 0)) {
        if (threadIdx.x == 0) atomicExch(a.err, DEV_TIMEOUT_TMA);
        mbar_wait_bounded(&block_bar, 0);      // give copies in flight one more bounded chance
        return;
    }
    int32_t* W = smem + a.shared_words + warp * a.warp_words;
    const long long ntiles = (a.num + a.K - 1) / a.K;
    const long long gw = static_cast<long long>(blockIdx.x) * nwarps + warp;
    const long long nw = static_cast<long long>(gridDim.x) * nwarps;
    for (long long t = gw; t < ntiles; t += nw)
        eval_tile<DM, W16, V, COUNT>(a, sh, rowt, W, t, a.prefetch && t + nw < ntiles ? t + nw : -1);
}

// Many instances of uneven size in one persistent launch: tile t of the
// whole job belongs to the instance whose tile prefix brackets it.  Distances
// come from the instance's points, copied into the warp's region per tile
// (DIST_HALF2), or from its matrix in global memory (L2-resident).  Every warp
// region is sized for the largest instance.
template <int DM, int V>
__global__ void __launch_bounds__(32 * max_warps(V)) eval_multi_kernel(const EvalArgs* __restrict__ insts,
                                                          const long long* __restrict__ tile_prefix, int n_inst,
                                                          int warp_words) {
    extern __shared__ __align__(16) int32_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    int32_t* W = smem + warp * warp_words;
    const long long total = tile_prefix[n_inst];
    const long long gw = static_cast<long long>(blockIdx.x) * nwarps + warp;
    const long long nw = static_cast<long long>(gridDim.x) * nwarps;
    int have = -1;                              // the instance whose points the region holds
    for (long long t = gw; t < total; t += nw) {
        int lo = 0, hi = n_inst;                // prefix[lo] <= t < prefix[lo+1]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(tile_prefix + mid) <= t) lo = mid; else hi = mid;
        }
        const EvalArgs a = insts[lo];
        const int32_t* sh = nullptr;
        if constexpr (DM == DIST_HALF2) {
            sh = W + a.pts;
            if (have != lo) {
                const int4* src = reinterpret_cast<const int4*>(a.xy);
                int4* dst = reinterpret_cast<int4*>(W + a.pts);
                for (int i = lane; i < a.row_words / 4; i += 32) dst[i] = __ldg(src + i);
                have = lo;
            }
        }
        eval_tile<DM, false, V, false>(a, sh, a.rowt, W, t - __ldg(tile_prefix + lo), -1);
    }
}

// ---------------------------------------------------------------------------
// Plain form: thread per candidate, global scratch, Kahn order.
// scratch per thread: ready[n+1], pos[m], dep[m], loc[m], seen[(2n+2+31)/32]
// ---------------------------------------------------------------------------
__global__ void eval_plain_kernel(const int32_t* __restrict__ ops, const int32_t* __restrict__ off,
                                  long long num, int n, int m, int R, int Q, int load_full,
                                  const int32_t* __restrict__ d, const int32_t* __restrict__ p,
                                  int32_t* __restrict__ zout, uint32_t* __restrict__ stout,
                                  int32_t* __restrict__ scratch, int scratch_words) {
    const long long tid = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    const long long nthreads = static_cast<long long>(gridDim.x) * blockDim.x;
    const int N = n + 1, two_n = 2 * n, sw = (two_n + 2 + 31) / 32;
    int32_t* ready = scratch + tid * static_cast<long long>(scratch_words);
    int32_t* pos = ready + (n + 1);
    int32_t* dep = pos + m;
    int32_t* loc = dep + m;
    uint32_t* seen = reinterpret_cast<uint32_t*>(loc + m);
    for (long long i = tid; i < num; i += nthreads) {
        const int32_t* o = ops + i * two_n;
        const int32_t* f = off + i * (m + 1);
        uint32_t st = 0;
        if (f[0] != 0 || f[m] != two_n) st = VRPRPD_MALFORMED;
        for (int v = 0; v < m && !st; ++v)
            if (f[v + 1] < f[v]) st = VRPRPD_MALFORMED;
        for (int w = 0; w < sw; ++w) seen[w] = 0u;
        for (int k2 = 0; k2 < two_n && !st; ++k2) {
            const int op = o[k2];
            if (op < 2 || op > two_n + 1) { st = VRPRPD_MALFORMED; break; }
            const uint32_t bit = 1u << (op & 31);
            if (seen[op >> 5] & bit) { st = VRPRPD_MALFORMED; break; }
            seen[op >> 5] |= bit;
        }
        if (st) { zout[i] = 0x7fffffff; stout[i] = st; continue; }
        for (int c = 0; c <= n; ++c) ready[c] = UNRESOLVED;
        for (int v = 0; v < m; ++v) { pos[v] = f[v]; dep[v] = 0; loc[v] = 0; }
        bool progress = true;
        while (progress) {
            progress = false;
            for (int v = 0; v < m; ++v) {
                while (pos[v] < f[v + 1]) {
                    const int op = o[pos[v]], c = op >> 1;
                    const bool pick = op & 1;
                    if (pick && ready[c] < 0) break;
                    const int arr = dep[v] + d[static_cast<long long>(loc[v]) * N + c];
                    if (!pick) { dep[v] = arr; ready[c] = arr + p[c]; }
                    else dep[v] = max(arr, ready[c]);
                    loc[v] = c;
                    ++pos[v];
                    progress = true;
                }
            }
        }
        int z = 0;
        long long pool = 0;
        for (int v = 0; v < m; ++v) {
            if (pos[v] < f[v + 1]) st |= VRPRPD_CYCLE;
            if (f[v + 1] > f[v]) z = max(z, dep[v] + d[static_cast<long long>(loc[v]) * N]);
            int s = 0, smin = 0, smax = 0;
            for (int k2 = f[v]; k2 < f[v + 1]; ++k2) {
                s += (o[k2] & 1) ? 1 : -1;
                smin = min(smin, s);
                smax = max(smax, s);
            }
            if (load_full) {
                if (smin < -Q || smax > 0) st |= VRPRPD_VEH_CAP;
                pool += Q;
            } else {
                if (-smin + smax > Q) st |= VRPRPD_VEH_CAP;
                pool += -smin;
            }
        }
        if (pool > R) st |= VRPRPD_POOL;
        if (st & VRPRPD_CYCLE) z = 0x7fffffff;
        zout[i] = z;
        stout[i] = st;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int round4(long long w) { return static_cast<int>((w + 3) & ~3ll); }

// Shared memory of an SM, and what the system keeps of it per block.
constexpr long long SM_SHARED_BYTES = 228 << 10, BLOCK_SHARED_BYTES = 1 << 10;

struct Plan {
    int dm = 0;          // the kernel's distance mode (DIST_HALF2 for small coordinates)
    int warps = 0, blocks = 0;
    bool w16 = false;    // 16-bit op codes and offsets
    bool count = false;  // coordination counts instead of makespan and status
    int V = 1;           // routes per lane
    size_t smem = 0;
    EvalArgs args{};
};

bool coords_exact_small(const vrprpd_instance* I) { return I->coords24; }

bool batched_supported(const vrprpd_instance* I) {
    return I->m <= 32 && 2 * I->n + 1 < (1 << PACK_SHIFT) && I->maxd < (1 << 19);
}

static bool dist_mode_available(const vrprpd_instance* I, int dm) {
    switch (dm) {
        case VRPRPD_DIST_SMEM32: return true;
        case VRPRPD_DIST_SMEM16: return I->has_d16;
        case VRPRPD_DIST_GLOBAL16: return I->has_d16;
        case VRPRPD_DIST_GLOBAL32: return true;
        case VRPRPD_DIST_COORDS: return I->coords24;
    }
    return false;
}

// What the entry points accept, in words of shared memory: the shapes of
// vrprpd_eval_config mean a block of `warps` warps, each with a region for
// floor(32/m) candidates (staged), or each group of G warps with one for
// floor(32 G/m) (streamed; codes not kept), beside the instance data.  The
// kernel's own regions are at most as large, or hold fewer candidates.
static long long accepted_shared_words(const vrprpd_instance* I, int dm) {
    const long long N = I->n + 1;
    long long w = 0;
    if (dm == VRPRPD_DIST_SMEM32) w = N * N;
    if (dm == VRPRPD_DIST_SMEM16) w = (N * N + 1) / 2;
    if (dm == VRPRPD_DIST_COORDS) w = 2 * N;
    return round4(w) + round4(N);
}
static long long accepted_staged_words(int n, int m) {
    const long long k = 32 / m, N = n + 1, sw = (2ll * n + 2 + 31) / 32;
    return round4((k * 2 * n + 1) / 2 + 2) + round4(k * N) + round4(k * sw) + round4(k * (m + 1)) + round4(k) + 100;
}
static long long accepted_streamed_words(int n, int m, int G) {
    const long long K = 32ll * G / m, N = n + 1;
    return round4(K * N) + round4(K * (m + 1)) + round4(K) + round4(2 * K) + 96ll * G;
}
static bool shape_accepted(const vrprpd_instance* I, int dm, int warps, int walk, int G) {
    long long words = accepted_shared_words(I, dm);
    if (walk == VRPRPD_WALK_STREAMED) {
        if ((G != 1 && G != 2) || warps % G != 0 || (G > 1 && warps / G > 15) || 32 * G < I->m) return false;
        words += warps / G * accepted_streamed_words(I->n, I->m, G);
    } else {
        words += warps * accepted_staged_words(I->n, I->m);
    }
    return words * 4 + 64 <= static_cast<long long>(I->smem_optin);
}

// The layout for (distance mode, warps per block, routes per lane): as many
// candidates per tile as the lanes take (32 V / m), fewer where the block's
// shared memory does not hold them or a warp's region would pass `cap` words.
// False if not even one fits.
static bool make_plan(const vrprpd_instance* I, int dm, int warps, int V, long long num, Plan* P, int cap = INT32_MAX) {
    EvalArgs& a = P->args;
    a = EvalArgs{};
    a.n = I->n;
    a.m = I->m;
    a.R = I->R;
    a.Q = I->Q;
    a.N = I->n + 1;
    a.load_full = (I->flags & VRPRPD_LOAD_FULL) != 0;
    a.pool_full = static_cast<long long>(I->m) * I->Q > I->R;
    a.d32 = I->d32;
    a.d16 = I->d16;
    a.coords = I->coords;
    a.xy = I->xy;
    a.rowt = I->rowt;
    a.row_words = I->row_words;
    a.err = I->err;
    a.num = num;
    const long long N = a.N;
    if (dm == VRPRPD_DIST_COORDS && I->xy) dm = DIST_HALF2;
    long long dist_words = 0;
    if (dm == VRPRPD_DIST_SMEM32) dist_words = N * N;
    if (dm == VRPRPD_DIST_SMEM16) dist_words = (N * N + 1) / 2;
    if (dm == VRPRPD_DIST_COORDS) dist_words = 2 * (N + 1);   // the point of code 2n+2 with them
    if (dm == DIST_HALF2) dist_words = a.row_words;
    a.dist_words = round4(dist_words);
    a.shared_words = a.dist_words + a.row_words;
    for (int K = 32 * V / I->m; K >= 1; --K) {
        a.K = K;
        a.a_words = round4(static_cast<long long>(K) * I->n) + 8;   // codes, shifted by up to 7 and padded to 16 bytes
        a.ready_words = K * a.row_words;
        a.off_words = round4(static_cast<long long>(K) * (I->m + 1));
        a.warp_words = a.a_words + a.ready_words + a.off_words + round4(4ll * K) + (P->count ? a.ready_words : 0);
        P->smem = static_cast<size_t>(a.shared_words + static_cast<long long>(warps) * a.warp_words) * 4;
        if (P->smem + 64 <= I->smem_optin && (K == 1 || a.warp_words <= cap)) {
            P->dm = dm;
            P->warps = warps;
            P->V = V;
            return true;
        }
    }
    return false;
}

template <bool W16, int V, bool COUNT = false>
static const void* kernel_for(int dm) {
    switch (dm) {
        case VRPRPD_DIST_SMEM32: return reinterpret_cast<const void*>(&eval_tiles_kernel<VRPRPD_DIST_SMEM32, W16, V, COUNT>);
        case VRPRPD_DIST_SMEM16: return reinterpret_cast<const void*>(&eval_tiles_kernel<VRPRPD_DIST_SMEM16, W16, V, COUNT>);
        case VRPRPD_DIST_GLOBAL16: return reinterpret_cast<const void*>(&eval_tiles_kernel<VRPRPD_DIST_GLOBAL16, W16, V, COUNT>);
        case VRPRPD_DIST_GLOBAL32: return reinterpret_cast<const void*>(&eval_tiles_kernel<VRPRPD_DIST_GLOBAL32, W16, V, COUNT>);
        case DIST_HALF2: return reinterpret_cast<const void*>(&eval_tiles_kernel<DIST_HALF2, W16, V, COUNT>);
        default: return reinterpret_cast<const void*>(&eval_tiles_kernel<VRPRPD_DIST_COORDS, W16, V, COUNT>);
    }
}

static const void* plan_kernel(const Plan& P) {
    if (P.count) return P.V == 2 ? kernel_for<false, 2, true>(P.dm) : kernel_for<false, 1, true>(P.dm);
    if (P.V == 2) return P.w16 ? kernel_for<true, 2>(P.dm) : kernel_for<false, 2>(P.dm);
    return P.w16 ? kernel_for<true, 1>(P.dm) : kernel_for<false, 1>(P.dm);
}

static int finalize_plan(const vrprpd_instance* I, int blocks_per_sm, Plan* P) {
    const void* fn = plan_kernel(*P);
    { int rc_ = ensure_smem_limit(fn); if (rc_) return rc_; }
    int occ = 0;
    VRP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, P->warps * 32, P->smem));
    VRP_CHECK(occ > 0, VRPRPD_EINVAL, "evaluation layout does not fit on an SM");
    if (blocks_per_sm > 0) occ = std::min(occ, blocks_per_sm);
    const long long ntiles = (P->args.num + P->args.K - 1) / P->args.K;
    const long long want = (ntiles + P->warps - 1) / P->warps;
    const long long blocks = std::min<long long>(static_cast<long long>(occ) * I->num_sms, want);
    P->blocks = static_cast<int>(std::max<long long>(blocks, 1));
    return VRPRPD_OK;
}

// The plan of a configured or tuned shape: its warps per block, or the most
// that fit.
static int plan_shape(const vrprpd_instance* I, const EvalTuning& T, long long num, Plan* P) {
    VRP_CHECK(dist_mode_available(I, T.dist_mode), VRPRPD_EINVAL, "configured distance mode unavailable");
    const int V = T.walk == VRPRPD_WALK_STREAMED ? T.group_warps : 1;
    for (int warps = std::min(T.warps_per_block, max_warps(V)); warps >= 1; --warps)
        if (make_plan(I, T.dist_mode, warps, V, num, P)) return finalize_plan(I, T.blocks_per_sm, P);
    set_error("configured evaluation layout exceeds shared memory");
    return VRPRPD_EINVAL;
}

// What a batch costs whose distances are gathered from L2, by shape (in lane
// reads that miss the L1).  The L1 is what the blocks' shared memory leaves of an
// SM's 256 KB, and how much of the matrix it catches decides: a turn of the SMs
// takes a round's latency or its lanes' reads, whichever is longer.  The three
// numbers were fitted to 2800 timings (n 240 to 1400, m 5 to 30, 512 to 32768
// candidates, one and two routes per lane, 4 to 32 warps): the shape of the
// least cost is 4% from the fastest one on average; the most routes in flight,
// as for the other forms, is 18% from it (n=500 m=20, 32768 candidates: two
// routes in 196 KB of shared memory 249 us, the shape of the least cost 182).
static double gather_cost(const EvalArgs& a, long long resident, long long shared, double matrix, int sms) {
    int kb = 228;
    for (int step : {196, 164, 132, 100, 64, 32, 16, 8})
        if (shared <= static_cast<long long>(step) << 10) kb = step;
    const double misses = 1.0 / 12 + 1.0 - std::min(1.0, std::pow((256 - kb) * 1024.0 / matrix, 0.2));
    auto turn = [&](double warps) { return std::max(160.0, warps * a.K * a.m * misses); };
    const long long tiles = (a.num + a.K - 1) / a.K, all = resident * sms;
    const double rest = static_cast<double>(tiles % all);
    return static_cast<double>(tiles / all) * turn(static_cast<double>(resident)) + (rest > 0 ? turn(rest / sms) : 0.0);
}

// The plan when nothing is configured.
static int auto_plan(const vrprpd_instance* I, long long num, Plan* P) {
    // Distances: points as fp16 pairs when the instance has them (a leg is 7
    // instructions from one 4-byte gather); else the 16-bit matrix in shared
    // memory while it takes at most half of it, recomputed integer legs, and
    // the matrix in L2 last.
    int dm = VRPRPD_DIST_GLOBAL32;
    if (I->xy) dm = VRPRPD_DIST_COORDS;
    else if (I->has_d16 && accepted_shared_words(I, VRPRPD_DIST_SMEM16) * 8 <= static_cast<long long>(I->smem_optin)) dm = VRPRPD_DIST_SMEM16;
    else if (accepted_shared_words(I, VRPRPD_DIST_SMEM32) * 8 <= static_cast<long long>(I->smem_optin)) dm = VRPRPD_DIST_SMEM32;
    else if (I->coords24) dm = VRPRPD_DIST_COORDS;
    else if (I->has_d16) dm = VRPRPD_DIST_GLOBAL16;
    const bool gathers = dm == VRPRPD_DIST_GLOBAL16 || dm == VRPRPD_DIST_GLOBAL32;
    const double matrix = static_cast<double>(I->n + 1) * (I->n + 1) * (dm == VRPRPD_DIST_GLOBAL16 ? 2 : 4);
    Plan best;
    double least = 0;                          // its cost; 0: none yet
    long long resident = 0;                    // its warps on an SM
    // Warps per block: most routes in flight on an SM, the smallest block on
    // ties (n=200 m=6: 4 warps 72 us, 24 warps 76 us), or the least gather_cost.
    auto take = [&](int V) {
        for (int warps : {4, 8, 12, 16, 20, 24, 28, 32, 2, 1}) {
            if (warps > max_warps(V) || (warps < 4 && least != 0) || (warps == 20 && !gathers)) continue;
            Plan C;
            C.w16 = P->w16;
            C.count = P->count;
            if (!make_plan(I, dm, warps, V, num, &C)) continue;
            const long long bytes = static_cast<long long>(C.smem + BLOCK_SHARED_BYTES);
            const long long blocks = std::min<long long>(SM_SHARED_BYTES / bytes, max_warps(V) / warps);
            const double cost = gathers ? gather_cost(C.args, warps * blocks, blocks * bytes, matrix, I->num_sms)
                                        : 1.0 / static_cast<double>(warps * blocks * C.args.K);
            if (least != 0 && cost >= least) continue;
            least = cost;
            best = C;
            resident = warps * blocks;
        }
    };
    auto tiles = [&]() { return (num + best.args.K - 1) / best.args.K; };
    // Two routes per lane when that uses the lanes better by a fifth or more
    // (m = 11, 12 and 17..21): n=499 m=19 (57 of 64 lane slots against 19 of
    // 32) 172 us against 223 us for 65536 candidates, n=1000 m=20 368 against
    // 377; but n=200 m=6 (30 of 32 both ways) 78 us against 72 us.  The counts
    // keep two rows per candidate, and two routes per lane take 1.1 to 2 times as
    // long there (n=200 m=20, 8192: 37.8 us against 30.3), unless that saves a
    // second turn of the SMs (n=60 m=20, 5120: 10.9 us against 12.7).
    const int m = I->m;
    const bool two = 5 * (64 / m) * m >= 6 * 2 * (32 / m) * m;
    if (gathers || P->count || !two) take(1);
    if (gathers ? !P->count : !P->count && two) take(2);
    if (P->count && !gathers && two && resident && tiles() > resident * I->num_sms) {
        const Plan one = best;
        const long long before = resident;
        least = 0;
        take(2);
        if (least == 0 || tiles() > resident * I->num_sms) {
            best = one;
            resident = before;
        }
    }
    if (!resident) {
        set_error("no evaluation layout fits shared memory (n=%d, m=%d)", I->n, I->m);
        return VRPRPD_EINVAL;
    }
    // few tiles are spread over the SMs first
    const long long ntiles = tiles();
    best.warps = static_cast<int>(std::max<long long>(1, std::min<long long>(best.warps, (ntiles + I->num_sms - 1) / I->num_sms)));
    best.smem = static_cast<size_t>(best.args.shared_words + static_cast<long long>(best.warps) * best.args.warp_words) * 4;
    *P = best;
    return finalize_plan(I, 0, P);
}

static int choose_plan(const vrprpd_instance* I, long long num, Plan* P) {
    if (I->tune.dist_mode != VRPRPD_DIST_AUTO && I->tune.warps_per_block > 0) return plan_shape(I, I->tune, num, P);
    if (!shape_accepted(I, VRPRPD_DIST_GLOBAL32, 1, VRPRPD_WALK_STAGED, 1)) {
        set_error("no evaluation layout fits shared memory (n=%d, m=%d)", I->n, I->m);
        return VRPRPD_EINVAL;
    }
    return auto_plan(I, num, P);
}

static int launch_plan(const Plan& P, cudaStream_t stream) {
    EvalArgs args = P.args;
    void* params[] = {&args};
    VRP_CUDA(cudaLaunchKernel(plan_kernel(P), dim3(P.blocks), dim3(P.warps * 32), params, P.smem, stream));
    return VRPRPD_OK;
}

static int check_batch(const vrprpd_instance* I, const vrprpd_batch* b, const void* z, const void* st) {
    VRP_CHECK(I && b && z && st, VRPRPD_EINVAL, "NULL argument");
    VRP_CHECK(b->num >= 0, VRPRPD_EINVAL, "negative batch size");
    VRP_CHECK(b->num == 0 || (b->ops && b->off), VRPRPD_EINVAL, "NULL ops/off");
    VRP_CHECK((reinterpret_cast<uintptr_t>(b->ops) & 3u) == 0 && (reinterpret_cast<uintptr_t>(b->off) & 3u) == 0,
              VRPRPD_EINVAL, "ops/off must be 4-byte aligned");
    return VRPRPD_OK;
}

int evaluate_device(const vrprpd_instance* I, const int32_t* ops, const int32_t* off, long long num,
                    int32_t* z, uint32_t* st, cudaStream_t stream, bool host_mapped = false) {
    if (num == 0) return VRPRPD_OK;
    if (!batched_supported(I)) {
        set_error("batched evaluation needs m <= 32, 2n+1 < 4096 and max d < 2^19 (use the plain form)");
        return VRPRPD_EINVAL;
    }
    Plan P;
    int rc = choose_plan(I, num, &P);
    if (rc) return rc;
    P.args.prefetch = host_mapped ? 0 : 1;
    P.args.ops = ops;
    P.args.off = off;
    P.args.z = z;
    P.args.st = st;
    return launch_plan(P, stream);
}

// The same evaluation from 16-bit op codes and offsets.
static int evaluate_device16(const vrprpd_instance* I, const uint16_t* ops, const uint16_t* off, long long num,
                             int32_t* z, uint32_t* st, cudaStream_t stream, bool host_mapped = false) {
    if (num == 0) return VRPRPD_OK;
    if (!batched_supported(I)) {
        set_error("batched evaluation needs m <= 32, 2n+1 < 4096 and max d < 2^19 (use the plain form)");
        return VRPRPD_EINVAL;
    }
    Plan P;
    P.w16 = true;
    int rc = choose_plan(I, num, &P);
    if (rc) return rc;
    P.args.prefetch = host_mapped ? 0 : 1;
    P.args.ops16 = ops;
    P.args.off16 = off;
    P.args.z = z;
    P.args.st = st;
    return launch_plan(P, stream);
}

// Coordination counts by the same walk, for instances its words hold: true
// when launched (*rc is its result), false when the caller has to.
bool coordination_walk(const vrprpd_instance* I, const int32_t* ops, const int32_t* off, long long num,
                       int32_t* cross, int32_t* interleaved, cudaStream_t stream, int* rc) {
    if (!batched_supported(I) || I->maxp >= (1 << 25)) return false;
    Plan P;
    P.count = true;
    *rc = auto_plan(I, num, &P);
    if (*rc) return false;
    P.args.prefetch = 1;
    P.args.ops = ops;
    P.args.off = off;
    P.args.z = cross;
    P.args.st = reinterpret_cast<uint32_t*>(interleaved);
    *rc = launch_plan(P, stream);
    return true;
}

static int check_batch16(const vrprpd_instance* I, const vrprpd_batch16* b, const void* z, const void* st) {
    VRP_CHECK(I && b && z && st, VRPRPD_EINVAL, "NULL argument");
    VRP_CHECK(b->num >= 0, VRPRPD_EINVAL, "negative batch size");
    VRP_CHECK(b->num == 0 || (b->ops && b->off), VRPRPD_EINVAL, "NULL ops/off");
    VRP_CHECK((reinterpret_cast<uintptr_t>(b->ops) & 3u) == 0 && (reinterpret_cast<uintptr_t>(b->off) & 1u) == 0,
              VRPRPD_EINVAL, "ops must be 4-byte and off 2-byte aligned");
    return VRPRPD_OK;
}

// Host buffers (ops/off of esz bytes per value): pinned ones are read by the
// kernel in place over the host link (each op is read once, by coalesced
// loads), pageable ones are copied to the device first; the results come back
// to z_host/st_host before the call returns.
static int evaluate_host_impl(vrprpd_instance* I, const void* ops, const void* off, int esz, long long num,
                              int32_t* z_host, uint32_t* st_host, cudaStream_t stream) {
    if (num == 0) return VRPRPD_OK;
    auto run = [&](const void* o, const void* f, int32_t* dz, uint32_t* dst, bool mapped) {
        return esz == 2 ? evaluate_device16(I, static_cast<const uint16_t*>(o), static_cast<const uint16_t*>(f), num,
                                            dz, dst, stream, mapped)
                        : evaluate_device(I, static_cast<const int32_t*>(o), static_cast<const int32_t*>(f), num, dz,
                                          dst, stream, mapped);
    };
    auto grow = [&](size_t need) -> int {
        if (need > I->stage_bytes) {
            if (I->stage) cudaFree(I->stage);
            I->stage = nullptr;
            I->stage_bytes = 0;
            VRP_CUDA(cudaMalloc(&I->stage, need));
            I->stage_bytes = need;
        }
        return VRPRPD_OK;
    };
    const size_t ops_b = static_cast<size_t>(num) * 2 * I->n * esz, off_b = static_cast<size_t>(num) * (I->m + 1) * esz;
    const size_t res_b = (static_cast<size_t>(num) * 4 + 255) & ~static_cast<size_t>(255);
    const void* ops_dev = nullptr;
    const void* off_dev = nullptr;
    {
        cudaPointerAttributes pa{}, pb{};
        if (cudaPointerGetAttributes(&pa, ops) == cudaSuccess && pa.type == cudaMemoryTypeHost &&
            cudaPointerGetAttributes(&pb, off) == cudaSuccess && pb.type == cudaMemoryTypeHost) {
            ops_dev = pa.devicePointer;
            off_dev = pb.devicePointer;
        }
        cudaGetLastError();                    // a pageable pointer is not an error here
    }
    int32_t* d_z;
    int rc;
    if (ops_dev && off_dev) {
        if ((rc = grow(2 * res_b))) return rc;
        d_z = reinterpret_cast<int32_t*>(I->stage);
        rc = run(ops_dev, off_dev, d_z, reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(d_z) + res_b), true);
    } else {
        const size_t ops_r = (ops_b + 255) & ~static_cast<size_t>(255), off_r = (off_b + 255) & ~static_cast<size_t>(255);
        if ((rc = grow(ops_r + off_r + 2 * res_b))) return rc;
        char* base = reinterpret_cast<char*>(I->stage);
        VRP_CUDA(cudaMemcpyAsync(base, ops, ops_b, cudaMemcpyHostToDevice, stream));
        VRP_CUDA(cudaMemcpyAsync(base + ops_r, off, off_b, cudaMemcpyHostToDevice, stream));
        d_z = reinterpret_cast<int32_t*>(base + ops_r + off_r);
        rc = run(base, base + ops_r, d_z, reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(d_z) + res_b), false);
    }
    if (rc) return rc;
    VRP_CUDA(cudaMemcpyAsync(z_host, d_z, num * 4, cudaMemcpyDeviceToHost, stream));
    VRP_CUDA(cudaMemcpyAsync(st_host, reinterpret_cast<char*>(d_z) + res_b, num * 4, cudaMemcpyDeviceToHost, stream));
    VRP_CUDA(cudaStreamSynchronize(stream));
    return VRPRPD_OK;
}

}  // namespace vrp

using namespace vrp;

extern "C" int vrprpd_evaluate(const vrprpd_instance* I, const vrprpd_batch* b, int32_t* z, uint32_t* st,
                               void* stream) {
    int rc = check_batch(I, b, z, st);
    if (rc) return rc;
    return evaluate_device(I, b->ops, b->off, b->num, z, st, static_cast<cudaStream_t>(stream));
}

extern "C" int vrprpd_evaluate_host(const vrprpd_instance* I_, const vrprpd_batch* b, int32_t* z_host,
                                    uint32_t* st_host, void* stream) {
    vrprpd_instance* I = const_cast<vrprpd_instance*>(I_);
    int rc = check_batch(I, b, z_host, st_host);
    if (rc) return rc;
    return evaluate_host_impl(I, b->ops, b->off, 4, b->num, z_host, st_host, static_cast<cudaStream_t>(stream));
}

extern "C" int vrprpd_evaluate16(const vrprpd_instance* I, const vrprpd_batch16* b, int32_t* z, uint32_t* st,
                                 void* stream) {
    int rc = check_batch16(I, b, z, st);
    if (rc) return rc;
    return evaluate_device16(I, b->ops, b->off, b->num, z, st, static_cast<cudaStream_t>(stream));
}

extern "C" int vrprpd_evaluate16_host(const vrprpd_instance* I_, const vrprpd_batch16* b, int32_t* z_host,
                                      uint32_t* st_host, void* stream) {
    vrprpd_instance* I = const_cast<vrprpd_instance*>(I_);
    int rc = check_batch16(I, b, z_host, st_host);
    if (rc) return rc;
    return evaluate_host_impl(I, b->ops, b->off, 2, b->num, z_host, st_host, static_cast<cudaStream_t>(stream));
}

extern "C" int vrprpd_evaluate_plain(const vrprpd_instance* I_, const vrprpd_batch* b, int32_t* z, uint32_t* st,
                                     void* stream) {
    vrprpd_instance* I = const_cast<vrprpd_instance*>(I_);
    int rc = check_batch(I, b, z, st);
    if (rc) return rc;
    if (b->num == 0) return VRPRPD_OK;
    const int threads = 128;
    const long long want = (b->num + threads - 1) / threads;
    const int blocks = static_cast<int>(std::min<long long>(want, 512));
    const int words = (I->n + 1) + 3 * I->m + (2 * I->n + 2 + 31) / 32;
    const size_t need = static_cast<size_t>(blocks) * threads * words;
    if (need > I->plain_scratch_words) {
        cudaFree(I->plain_scratch);
        I->plain_scratch = nullptr;
        I->plain_scratch_words = 0;
        VRP_CUDA(cudaMalloc(&I->plain_scratch, need * 4));
        I->plain_scratch_words = need;
    }
    eval_plain_kernel<<<blocks, threads, 0, static_cast<cudaStream_t>(stream)>>>(
        b->ops, b->off, b->num, I->n, I->m, I->R, I->Q, (I->flags & VRPRPD_LOAD_FULL) != 0, I->d32, I->p, z, st,
        I->plain_scratch, words);
    VRP_CUDA(cudaGetLastError());
    return VRPRPD_OK;
}

extern "C" int vrprpd_eval_set_config(vrprpd_instance* I, const vrprpd_eval_config* cfg) {
    VRP_CHECK(I && cfg, VRPRPD_EINVAL, "NULL argument");
    if (cfg->dist_mode == VRPRPD_DIST_AUTO) {
        I->tune = EvalTuning{};
        return VRPRPD_OK;
    }
    VRP_CHECK(cfg->dist_mode >= VRPRPD_DIST_SMEM32 && cfg->dist_mode <= VRPRPD_DIST_COORDS, VRPRPD_EINVAL,
              "bad dist_mode %d", cfg->dist_mode);
    VRP_CHECK(dist_mode_available(I, cfg->dist_mode), VRPRPD_EINVAL, "distance mode %d unavailable here",
              cfg->dist_mode);
    VRP_CHECK(cfg->warps_per_block >= 1 && cfg->warps_per_block <= 32, VRPRPD_EINVAL, "bad warps_per_block");
    VRP_CHECK(cfg->walk == VRPRPD_WALK_STAGED || cfg->walk == VRPRPD_WALK_STREAMED, VRPRPD_EINVAL, "bad walk %d",
              cfg->walk);
    VRP_CHECK(shape_accepted(I, cfg->dist_mode, cfg->warps_per_block, cfg->walk, cfg->group_warps), VRPRPD_EINVAL,
              cfg->walk == VRPRPD_WALK_STREAMED
                  ? "streamed layout does not fit (group_warps must be 1 or 2, divide warps_per_block, leave at "
                    "most 15 groups and cover m lanes)"
                  : "layout exceeds shared memory");
    I->tune.dist_mode = cfg->dist_mode;
    I->tune.warps_per_block = cfg->warps_per_block;
    I->tune.blocks_per_sm = cfg->blocks_per_sm;
    I->tune.walk = cfg->walk;
    I->tune.group_warps = cfg->walk == VRPRPD_WALK_STREAMED ? cfg->group_warps : 1;
    return VRPRPD_OK;
}

extern "C" int vrprpd_eval_get_config(const vrprpd_instance* I, vrprpd_eval_config* cfg) {
    VRP_CHECK(I && cfg, VRPRPD_EINVAL, "NULL argument");
    Plan P;
    int rc = choose_plan(I, 1 << 20, &P);
    if (rc) return rc;
    const bool set = I->tune.dist_mode != VRPRPD_DIST_AUTO;
    cfg->dist_mode = P.dm == DIST_HALF2 ? VRPRPD_DIST_COORDS : P.dm;
    cfg->warps_per_block = set ? I->tune.warps_per_block : P.warps;
    cfg->blocks_per_sm = I->tune.blocks_per_sm;
    cfg->walk = set ? I->tune.walk : P.V == 2 ? VRPRPD_WALK_STREAMED : VRPRPD_WALK_STAGED;
    cfg->group_warps = set ? I->tune.group_warps : P.V;
    return VRPRPD_OK;
}

extern "C" int vrprpd_autotune(vrprpd_instance* I, const vrprpd_batch* b, void* stream_, vrprpd_eval_config* chosen) {
    VRP_CHECK(I && b && b->num > 0, VRPRPD_EINVAL, "autotune needs a non-empty batch");
    if (!batched_supported(I)) {
        set_error("batched evaluation unsupported for this instance");
        return VRPRPD_EINVAL;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int32_t* z = nullptr;
    uint32_t* st = nullptr;
    VRP_CUDA(cudaMalloc(&z, b->num * 4));
    VRP_CUDA(cudaMalloc(&st, b->num * 4));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best_ms = 1e30f;
    EvalTuning best{};
    const EvalTuning saved = I->tune;
    const int modes[] = {VRPRPD_DIST_SMEM32, VRPRPD_DIST_SMEM16, VRPRPD_DIST_COORDS, VRPRPD_DIST_GLOBAL16,
                         VRPRPD_DIST_GLOBAL32};
    for (int dm : modes) {
        if (!dist_mode_available(I, dm)) continue;
        for (int V : {1, 2}) {
            const int walk = V == 2 ? VRPRPD_WALK_STREAMED : VRPRPD_WALK_STAGED;
            for (int warps : {4, 8, 12, 16, 24, 28, 32}) {
                Plan P;
                if (warps > max_warps(V) || !shape_accepted(I, dm, warps, walk, V) || !make_plan(I, dm, warps, V, b->num, &P)) continue;
                I->tune = EvalTuning{dm, warps, 0, walk, V};
                float ms_min = 1e30f;
                for (int rep = 0; rep < 4; ++rep) {
                    cudaEventRecord(e0, stream);
                    int rc = evaluate_device(I, b->ops, b->off, b->num, z, st, stream);
                    cudaEventRecord(e1, stream);
                    if (rc) break;
                    cudaEventSynchronize(e1);
                    float ms = 0;
                    cudaEventElapsedTime(&ms, e0, e1);
                    if (rep > 0) ms_min = std::min(ms_min, ms);
                }
                if (ms_min < best_ms) {
                    best_ms = ms_min;
                    best = I->tune;
                }
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(z);
    cudaFree(st);
    if (best.dist_mode == VRPRPD_DIST_AUTO) {
        I->tune = saved;
        set_error("autotune found no runnable configuration");
        return VRPRPD_EINVAL;
    }
    I->tune = best;
    if (chosen) {
        chosen->dist_mode = best.dist_mode;
        chosen->warps_per_block = best.warps_per_block;
        chosen->blocks_per_sm = best.blocks_per_sm;
        chosen->walk = best.walk;
        chosen->group_warps = best.group_warps;
    }
    VRP_CUDA(cudaGetLastError());
    return VRPRPD_OK;
}

// ---------------------------------------------------------------------------
// many instances, one persistent launch
// ---------------------------------------------------------------------------
// Words of one warp's region per route a lane walks, at most (unless a single
// candidate needs more): every region is sized for the largest instance, and
// this leaves 26 warps per SM.
constexpr int MULTI_CAP_WORDS = 2048;

struct vrprpd_multi {
    int n_inst = 0, device = 0, num_sms = 0;
    size_t smem_optin = 0;
    bool all16 = true, all_xy = true;
    // what the entry points accept: the largest instance's region per warp, staged and streamed
    long long accepted_words[2] = {0, 0};
    // for one and two routes per lane: per-instance arguments and tile prefix
    std::vector<EvalArgs> args[2];
    std::vector<long long> prefix[2];
    EvalArgs* d_args[2] = {nullptr, nullptr};
    long long* d_prefix[2] = {nullptr, nullptr};
    int V = 1;
    int dm = VRPRPD_DIST_GLOBAL16, warps = 8, blocks = 0, warp_words = 0;
    size_t smem = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t graph_stream = nullptr;
};

namespace vrp {

template <int V>
static const void* multi_kernel(int dm) {
    if (dm == DIST_HALF2) return reinterpret_cast<const void*>(&eval_multi_kernel<DIST_HALF2, V>);
    return dm == VRPRPD_DIST_GLOBAL16 ? reinterpret_cast<const void*>(&eval_multi_kernel<VRPRPD_DIST_GLOBAL16, V>)
                                      : reinterpret_cast<const void*>(&eval_multi_kernel<VRPRPD_DIST_GLOBAL32, V>);
}
static const void* multi_kernel(const vrprpd_multi* M) { return M->V == 2 ? multi_kernel<2>(M->dm) : multi_kernel<1>(M->dm); }

static int multi_layout(vrprpd_multi* M, int dm, int warps, int V) {
    int ww = 0;
    for (auto& a : M->args[V - 1]) ww = std::max(ww, a.warp_words);
    for (warps = std::min(warps, max_warps(V)); warps >= 1; --warps)
        if (static_cast<size_t>(warps) * ww * 4 + 64 <= M->smem_optin) break;
    if (warps < 1) return VRPRPD_EINVAL;
    M->V = V;
    M->dm = dm;
    M->warps = warps;
    M->warp_words = ww;
    M->smem = static_cast<size_t>(warps) * ww * 4;
    const void* fn = multi_kernel(M);
    { int rc_ = ensure_smem_limit(fn); if (rc_) return rc_; }
    int occ = 0;
    VRP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, warps * 32, M->smem));
    if (occ <= 0) return VRPRPD_EINVAL;
    const long long total = M->prefix[V - 1].back();
    M->blocks = static_cast<int>(std::max<long long>(1, std::min<long long>(static_cast<long long>(occ) * M->num_sms,
                                                                         (total + warps - 1) / warps)));
    if (M->exec) { cudaGraphExecDestroy(M->exec); M->exec = nullptr; }
    if (M->graph) { cudaGraphDestroy(M->graph); M->graph = nullptr; }
    return VRPRPD_OK;
}

static int multi_launch(vrprpd_multi* M, cudaStream_t s) {
    const EvalArgs* args = M->d_args[M->V - 1];
    const long long* prefix = M->d_prefix[M->V - 1];
    void* params[] = {&args, &prefix, &M->n_inst, &M->warp_words};
    VRP_CUDA(cudaLaunchKernel(multi_kernel(M), dim3(M->blocks), dim3(M->warps * 32), params, M->smem, s));
    return VRPRPD_OK;
}

}  // namespace vrp

extern "C" int vrprpd_multi_create(const vrprpd_instance* const* insts, const vrprpd_batch* batches,
                                   int32_t* const* makespan, uint32_t* const* status, int32_t n_inst,
                                   vrprpd_multi** out) {
    VRP_CHECK(insts && batches && makespan && status && out && n_inst >= 1, VRPRPD_EINVAL, "bad arguments");
    *out = nullptr;
    vrprpd_multi* M = new vrprpd_multi();
    M->n_inst = n_inst;
    M->prefix[0].assign(1, 0);
    M->prefix[1].assign(1, 0);
    for (int i = 0; i < n_inst; ++i) {
        const vrprpd_instance* I = insts[i];
        int rc = check_batch(I, &batches[i], makespan[i], status[i]);
        if (rc) { delete M; return rc; }
        if (!batched_supported(I)) {
            delete M;
            set_error("instance %d: batched evaluation needs m <= 32, 2n+1 < 4096, max d < 2^19", i);
            return VRPRPD_EINVAL;
        }
        if (i == 0) {
            M->device = I->device;
            M->num_sms = I->num_sms;
            M->smem_optin = I->smem_optin;
        } else if (I->device != M->device) {
            delete M;
            set_error("instances live on different devices");
            return VRPRPD_EINVAL;
        }
        M->all16 = M->all16 && I->has_d16;
        M->all_xy = M->all_xy && I->xy != nullptr;
        M->accepted_words[0] = std::max(M->accepted_words[0], accepted_staged_words(I->n, I->m));
        M->accepted_words[1] = std::max(M->accepted_words[1], accepted_streamed_words(I->n, I->m, 1));
        // no block-wide instance data; the points (if used) follow the warp's region
        for (int w = 0; w < 2; ++w) {
            Plan P;
            make_plan(I, VRPRPD_DIST_GLOBAL32, 1, w + 1, batches[i].num, &P, MULTI_CAP_WORDS * (w + 1));
            EvalArgs a = P.args;
            a.shared_words = 0;
            a.dist_words = 0;
            a.pts = a.warp_words;
            a.warp_words += I->xy ? a.row_words : 0;
            a.ops = batches[i].ops;
            a.off = batches[i].off;
            a.z = makespan[i];
            a.st = status[i];
            M->args[w].push_back(a);
            M->prefix[w].push_back(M->prefix[w].back() + (a.num + a.K - 1) / a.K);
        }
    }
    cudaError_t e = cudaSuccess;
    for (int w = 0; w < 2 && e == cudaSuccess; ++w) {
        e = cudaMalloc(&M->d_args[w], sizeof(EvalArgs) * n_inst);
        if (e == cudaSuccess) e = cudaMalloc(&M->d_prefix[w], sizeof(long long) * (n_inst + 1));
        if (e == cudaSuccess)
            e = cudaMemcpy(M->d_args[w], M->args[w].data(), sizeof(EvalArgs) * n_inst, cudaMemcpyHostToDevice);
        if (e == cudaSuccess)
            e = cudaMemcpy(M->d_prefix[w], M->prefix[w].data(), sizeof(long long) * (n_inst + 1),
                           cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
        set_error("multi_create: %s", cudaGetErrorString(e));
        vrprpd_multi_destroy(M);
        return VRPRPD_ECUDA;
    }
    int rc = VRPRPD_EINVAL;
    if (M->accepted_words[0] * 4 + 64 <= static_cast<long long>(M->smem_optin)) {
        // one or two routes per lane as for a single instance, by the lane
        // steps of the whole job (a tile walks about 2n/m rounds of V routes)
        double steps[2] = {0, 0};
        for (int w = 0; w < 2; ++w)
            for (auto& a : M->args[w]) steps[w] += static_cast<double>((a.num + a.K - 1) / a.K) * (w + 1) * a.n / a.m;
        const int dm = M->all_xy ? DIST_HALF2 : M->all16 ? VRPRPD_DIST_GLOBAL16 : VRPRPD_DIST_GLOBAL32;
        rc = multi_layout(M, dm, 4, 1.2 * steps[1] <= steps[0] ? 2 : 1);
    }
    if (rc) {
        set_error("multi_create: no layout fits shared memory");
        vrprpd_multi_destroy(M);
        return rc;
    }
    *out = M;
    return VRPRPD_OK;
}

extern "C" int vrprpd_multi_evaluate(vrprpd_multi* M, void* stream_) {
    VRP_CHECK(M, VRPRPD_EINVAL, "NULL plan");
    cudaStream_t s = static_cast<cudaStream_t>(stream_);
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (s != nullptr) VRP_CUDA(cudaStreamIsCapturing(s, &cs));
    if (s == nullptr || cs != cudaStreamCaptureStatusNone) return multi_launch(M, s);
    if (!M->exec || M->graph_stream != s) {
        if (M->exec) { cudaGraphExecDestroy(M->exec); M->exec = nullptr; }
        if (M->graph) { cudaGraphDestroy(M->graph); M->graph = nullptr; }
        VRP_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
        int rc = multi_launch(M, s);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(s, &g);
        if (rc) { if (g) cudaGraphDestroy(g); return rc; }
        VRP_CHECK(e == cudaSuccess, VRPRPD_ECUDA, "capture failed: %s", cudaGetErrorString(e));
        M->graph = g;
        VRP_CUDA(cudaGraphInstantiate(&M->exec, g, 0));
        M->graph_stream = s;
    }
    VRP_CUDA(cudaGraphLaunch(M->exec, s));
    return VRPRPD_OK;
}

extern "C" int vrprpd_multi_autotune(vrprpd_multi* M, void* stream_, vrprpd_eval_config* chosen) {
    VRP_CHECK(M, VRPRPD_EINVAL, "NULL plan");
    cudaStream_t s = static_cast<cudaStream_t>(stream_);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int bdm = M->dm, bw = M->warps, bV = M->V;
    for (int V : {1, 2}) {
        for (int dm : {DIST_HALF2, static_cast<int>(VRPRPD_DIST_GLOBAL16), static_cast<int>(VRPRPD_DIST_GLOBAL32)}) {
            if ((dm == DIST_HALF2 && !M->all_xy) || (dm == VRPRPD_DIST_GLOBAL16 && !M->all16)) continue;
            for (int warps : {4, 8, 12, 16, 24, 32, 2, 1}) {
                if (warps < 4 && best < 1e30f) continue;      // only where no larger block fits
                if (M->accepted_words[V - 1] * 4 * warps + 64 > static_cast<long long>(M->smem_optin)) continue;
                if (multi_layout(M, dm, warps, V) != VRPRPD_OK) continue;
                float ms_min = 1e30f;
                for (int rep = 0; rep < 3; ++rep) {
                    cudaEventRecord(e0, s);
                    multi_launch(M, s);
                    cudaEventRecord(e1, s);
                    cudaEventSynchronize(e1);
                    float ms = 0;
                    cudaEventElapsedTime(&ms, e0, e1);
                    if (rep > 0) ms_min = std::min(ms_min, ms);
                }
                if (ms_min < best) { best = ms_min; bdm = dm; bw = warps; bV = V; }
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    int rc = multi_layout(M, bdm, bw, bV);
    if (rc) return rc;
    if (chosen) {
        chosen->dist_mode = bdm == DIST_HALF2 ? VRPRPD_DIST_COORDS : bdm;
        chosen->warps_per_block = bw;
        chosen->blocks_per_sm = 0;
        chosen->walk = bV == 2 ? VRPRPD_WALK_STREAMED : VRPRPD_WALK_STAGED;
        chosen->group_warps = bV;
    }
    VRP_CUDA(cudaGetLastError());
    return VRPRPD_OK;
}

extern "C" int vrprpd_multi_set_config(vrprpd_multi* M, const vrprpd_eval_config* cfg) {
    VRP_CHECK(M && cfg, VRPRPD_EINVAL, "NULL argument");
    VRP_CHECK(cfg->dist_mode == VRPRPD_DIST_GLOBAL16 || cfg->dist_mode == VRPRPD_DIST_GLOBAL32 ||
                  cfg->dist_mode == VRPRPD_DIST_COORDS, VRPRPD_EINVAL,
              "many-instance plans take distances from points or L2: dist_mode must be COORDS, GLOBAL16 or GLOBAL32");
    VRP_CHECK(cfg->walk == VRPRPD_WALK_STAGED ||
                  (cfg->walk == VRPRPD_WALK_STREAMED && (cfg->group_warps == 1 || cfg->group_warps == 2)),
              VRPRPD_EINVAL, "walk must be staged, or streamed with group_warps 1 or 2");
    VRP_CHECK(cfg->dist_mode != VRPRPD_DIST_COORDS || M->all_xy, VRPRPD_EINVAL,
              "an instance has no points, or points too far apart");
    if (cfg->dist_mode == VRPRPD_DIST_GLOBAL16)
        for (auto& a : M->args[0]) VRP_CHECK(a.d16 != nullptr, VRPRPD_EINVAL, "an instance has no 16-bit matrix");
    VRP_CHECK(cfg->warps_per_block >= 1 && cfg->warps_per_block <= 32, VRPRPD_EINVAL, "bad warps_per_block");
    const bool streamed = cfg->walk == VRPRPD_WALK_STREAMED;
    VRP_CHECK(M->accepted_words[streamed] * 4 * cfg->warps_per_block + 64 <= static_cast<long long>(M->smem_optin),
              VRPRPD_EINVAL, "this layout does not fit shared memory");
    const int rc = multi_layout(M, cfg->dist_mode == VRPRPD_DIST_COORDS ? DIST_HALF2 : cfg->dist_mode,
                                cfg->warps_per_block, streamed ? cfg->group_warps : 1);
    VRP_CHECK(rc == VRPRPD_OK, rc, "this layout does not fit shared memory");
    return VRPRPD_OK;
}

extern "C" void vrprpd_multi_destroy(vrprpd_multi* M) {
    if (!M) return;
    if (M->exec) cudaGraphExecDestroy(M->exec);
    if (M->graph) cudaGraphDestroy(M->graph);
    for (int w = 0; w < 2; ++w) {
        cudaFree(M->d_args[w]);
        cudaFree(M->d_prefix[w]);
    }
    delete M;
}

// ---------------------------------------------------------------------------
// Plain evaluation without any device allocation.
//
// Some callers cannot let the library allocate device memory: code that is
// recording a CUDA graph (an allocation there is not part of the capture and
// breaks it), serving processes that reserve their whole memory budget up
// front and must not grow, and processes whose framework caching allocator
// already holds the free device memory, so a fresh cudaMalloc would fail.
// For them this entry point runs the plain one-thread-per-candidate kernel
// with its per-thread scratch (ready times, route cursors, the op bitmap)
// carved from a fixed array that is part of the library image: 16 MiB on each
// GPU that loads the library, held until the process exits.
// ---------------------------------------------------------------------------
namespace vrp {
constexpr long long NOALLOC_SCRATCH_WORDS = 4ll << 20;   // 4 Mi int32 = 16 MiB
static __device__ __align__(256) int32_t g_noalloc_scratch[NOALLOC_SCRATCH_WORDS];
}  // namespace vrp

extern "C" int vrprpd_evaluate_plain_noalloc_shape(int32_t n, int32_t m, int64_t num, int32_t* blocks,
                                                   int32_t* threads) {
    VRP_CHECK(n >= 1 && m >= 1 && num >= 0 && blocks && threads, VRPRPD_EINVAL, "bad arguments");
    const long long words = (n + 1ll) + 3ll * m + (2ll * n + 2 + 31) / 32;
    const long long max_threads = NOALLOC_SCRATCH_WORDS / words;
    VRP_CHECK(max_threads >= 32, VRPRPD_EINVAL,
              "instance needs %lld scratch words per thread; the fixed %lld-word scratch fits fewer than 32 "
              "threads (use vrprpd_evaluate_plain)", words, NOALLOC_SCRATCH_WORDS);
    // a block of up to 128 threads, a multiple of 32, and only as many
    // blocks as the scratch holds: every launched thread owns its words
    const long long tpb = std::min<long long>(128, max_threads / 32 * 32);
    const long long want = std::max<long long>(1, (num + tpb - 1) / tpb);
    const long long nb = std::max<long long>(1, std::min<long long>(want, max_threads / tpb));
    if (nb * tpb > max_threads) {
        set_error("internal: launch shape exceeds the fixed scratch");
        return VRPRPD_EINVAL;
    }
    *blocks = static_cast<int32_t>(nb);
    *threads = static_cast<int32_t>(tpb);
    return VRPRPD_OK;
}

extern "C" int vrprpd_evaluate_plain_noalloc(const vrprpd_instance* I, const vrprpd_batch* b, int32_t* z,
                                             uint32_t* st, void* stream) {
    int rc = check_batch(I, b, z, st);
    if (rc) return rc;
    if (b->num == 0) return VRPRPD_OK;
    int32_t blocks = 0, threads = 0;
    rc = vrprpd_evaluate_plain_noalloc_shape(I->n, I->m, b->num, &blocks, &threads);
    if (rc) return rc;
    const long long words = (I->n + 1) + 3ll * I->m + (2ll * I->n + 2 + 31) / 32;
    // the array's address on the current device, looked up on every call (the
    // lookup allocates nothing): a cached address would dangle after a
    // device reset reloads the module
    void* scratch = nullptr;
    VRP_CUDA(cudaGetSymbolAddress(&scratch, g_noalloc_scratch));
    eval_plain_kernel<<<blocks, threads, 0, static_cast<cudaStream_t>(stream)>>>(
        b->ops, b->off, b->num, I->n, I->m, I->R, I->Q, (I->flags & VRPRPD_LOAD_FULL) != 0, I->d32, I->p, z, st,
        static_cast<int32_t*>(scratch), static_cast<int>(words));
    VRP_CUDA(cudaGetLastError());
    return VRPRPD_OK;
}
