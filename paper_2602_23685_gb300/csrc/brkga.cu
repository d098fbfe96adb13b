// BRKGA on the device (Section 4.4): random-key chromosomes, the multi-pass
// decoder of Algorithm 2, elite preservation, mutants, biased crossover and
// the ALNS warm start (Section 4.4.4).
//
// Per generation (captured once as a CUDA graph, replayed):
//   decode   one warp per chromosome: warp bitonic sort of (key, op index)
//            pairs in shared memory -- the segmented key sort -- then the
//            multi-pass decode with one lane per vehicle; SelectVehicle is a
//            warp argmin of (arrival, vehicle-key rank);
//   evaluate the decoded routes go through the batched evaluator (same
//            makespans by construction; disagreements are counted), beside the
//            two steps that follow;
//   rank     by (fitness, index), recording the generation's best;
//   evolve   elites copied, children by biased crossover, mutants drawn.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "device_common.cuh"
#include "internal.h"

namespace vrp {

int evaluate_device(const vrprpd_instance* I, const int32_t* ops, const int32_t* off, long long num, int32_t* z,
                    uint32_t* st, cudaStream_t stream, bool host_mapped = false);
bool batched_supported(const vrprpd_instance* I);

constexpr int DEC_WARPS = 4;
constexpr long long PENALTY = 1000000;

struct BrkgaCtl {
    int gen;            // generation being built
    int sel;            // which key buffer is current
    int mismatches;     // decoder makespan != evaluator makespan (complete decodes)
    int pad;
};

struct DecArgs {
    const float* keys;   // num x L (or two buffers selected by ctl->sel when keys2 != nullptr)
    const float* keys2;
    const BrkgaCtl* ctl;
    int num, n, m, R, Q, load_full, L, P;   // P = power of two >= 2n
    int layout;          // VRPRPD_LAYOUT_VKEYS (2n+m keys) or VRPRPD_LAYOUT_HINTS (4n keys)
    const int32_t* d32;
    const int32_t* p;
    int smem_dist;       // 1 = distance matrix staged in shared memory as int32, 2 = as uint16
    int pack;            // every schedule time is below 2^22: SelectVehicle is one 32-bit reduction
    const uint16_t* d16; // the 16-bit copy (max d < 65536) or null
    int* err;
    int32_t* ops;
    int32_t* off;
    int32_t* z;
    int32_t* unsched;
    long long* fitness;
};

__host__ __device__ inline int pow2_at_least(int x) {
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

constexpr int SORT_REGS_MAX = 1024;   // ops (a power of two) that a warp sorts in registers

__host__ __device__ inline size_t dec_warp_words(int n, int P) {
    // op list (beyond SORT_REGS_MAX the u64 sort buffer it comes from) + tdrop +
    // log of the scheduled ops + per-op hinted vehicle (bytes)
    const int list = P > SORT_REGS_MAX ? 2 * P : P > 32 ? P : 32;
    return static_cast<size_t>(list) + (((n + 1) + 3) & ~3) + (((2 * n) + 3) & ~3) + ((((2 * n + 3) / 4) + 3) & ~3);
}

// The vehicle an assignment hint names: floor(m * alpha), capped to [0, m - 1].
// The product rounded down lies at or above an integer exactly when the product
// does (integers up to 32 are floats), so fp32 gives the floor of the exact
// product; an fp64 product, also exact, costs a tenth of the decode here.
__device__ inline int hint_vehicle(float alpha, int m) {
    const int h = __float2int_rd(__fmul_rd(alpha, static_cast<float>(m)));
    return max(min(h, m - 1), 0);
}

// The ops in priority order into list: stable argsort of the 2n keys, as a
// bitonic sort of (key bits, op index) by one warp.  Lane l holds elements
// l EPL .. l EPL + EPL - 1 in registers, so of the 45 steps for 512 elements 30
// stay inside a lane and 15 are shuffles (in shared memory every step was a
// pass over the buffer and a barrier).
__device__ __forceinline__ unsigned long long sort_entry(const float* kk, int two_n, int i) {
    if (i >= two_n) return ~0ull;                                     // padding sorts last
    const float f = __fadd_rn(__ldg(kk + i), 0.0f);                  // -0 -> +0
    return (static_cast<unsigned long long>(__float_as_uint(f)) << 32) | static_cast<unsigned>(i);
}
template <int EPL>
__device__ __noinline__ void sort_ops(const float* kk, int two_n, int* list) {
    const int lane = threadIdx.x & 31;
    unsigned long long x[EPL];
#pragma unroll
    for (int r = 0; r < EPL; ++r) x[r] = sort_entry(kk, two_n, lane * EPL + r);
    auto exchange = [&](int i, int j, bool asc) {
        const unsigned long long a = x[i], b = x[j];
        const bool swap = (a > b) == asc;
        x[i] = swap ? b : a;
        x[j] = swap ? a : b;
    };
#pragma unroll
    for (int size = 2; size < EPL; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1)
#pragma unroll
            for (int r = 0; r < EPL; ++r)
                if (!(r & stride)) exchange(r, r | stride, (r & size) == 0);
    for (int size = EPL > 1 ? EPL : 2; size <= 32 * EPL; size <<= 1) {
        const bool asc = ((lane * EPL) & size) == 0;
        for (int far = size / (2 * EPL); far > 0; far >>= 1) {
            const bool least = ((lane & far) == 0) == asc;
#pragma unroll
            for (int r = 0; r < EPL; ++r) {
                const unsigned long long o = __shfl_xor_sync(FULL_MASK, x[r], far);
                x[r] = (o < x[r]) == least ? o : x[r];
            }
        }
#pragma unroll
        for (int stride = EPL >> 1; stride > 0; stride >>= 1)
#pragma unroll
            for (int r = 0; r < EPL; ++r)
                if (!(r & stride)) exchange(r, r | stride, asc);
    }
#pragma unroll
    for (int r = 0; r < EPL; ++r) list[lane * EPL + r] = static_cast<int>(x[r] & 0xffffffffu);
    __syncwarp();
}
// The same beyond SORT_REGS_MAX, through a shared buffer that list shares.
__device__ __noinline__ void sort_ops_shared(const float* kk, int two_n, int P, unsigned long long* sb, int* list) {
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < P; i += 32) sb[i] = sort_entry(kk, two_n, i);
    __syncwarp();
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = lane; i < P / 2; i += 32) {
                const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                const bool asc = (lo & size) == 0;
                const unsigned long long x = sb[lo], y = sb[hi];
                if ((x > y) == asc) { sb[lo] = y; sb[hi] = x; }
            }
            __syncwarp();
        }
    }
    for (int base = 0; base < P; base += 32) {                       // list[k] lies at or below sb[k]
        const int v = static_cast<int>(sb[base + lane] & 0xffffffffu);
        __syncwarp();
        list[base + lane] = v;
        __syncwarp();
    }
}

// shared-memory accesses by 32-bit address, out of the compiler's reach to turn
// into generic ones or branches
__device__ __forceinline__ int lds_u16(unsigned addr) {
    int v;
    asm("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ int lds_b32(unsigned addr) {
    int v;
    asm("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_if(bool on, unsigned addr, int v) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %0, 0;\n\t"
        "@p st.shared.b32 [%1], %2;\n\t}" ::"r"(static_cast<unsigned>(on)),
        "r"(addr), "r"(v)
        : "memory");
}
// index of the highest set bit (of a single one here), ~0 for none
__device__ __forceinline__ unsigned bit_index(unsigned x) {
    unsigned r;
    asm("bfind.u32 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}

// The decoder specialised on its per-visit choices, so the chain of one op's
// visit holds no branch on them: SD where distances come from (0 L2 int32,
// 1 shared int32, 2 shared uint16), HINTS the 4n layout's tie rule, FULL the
// Eq. 13 start load, PACK the one-reduction SelectVehicle.
//
// One chain of dependent visits per chromosome is what takes the time, and with
// one chromosome per warp nothing else runs beside it: latency, and the warp's
// own instruction count.  So:
//   - a pass takes the list 32 ops at a time, one per lane, and goes straight to
//     the ops that can be scheduled.  Whether a drop (a pickup) fits any vehicle
//     does not depend on the customer, so two votes after each visit say which
//     kind can go next, and masks where the next of each kind stands: of 1290
//     list entries per decode at n=200 m=6 R=20, 400 are visited, none in vain;
//   - the next drop and the next pickup are both looked up (their words, then
//     their distances from every vehicle) while the vehicle is selected;
//   - a vehicle's stock is two numbers, see below; its time, tie rank and one
//     flag share the selection key, so key == minimum names the winner;
//   - an op's place is logged by the winner, drop times are written once per
//     chunk, and the matrix arrives by one bulk copy behind the sort.
// 1024 decodes of the 4n layout at n=200 m=6: 281 us before, 89 us now (47 k warp
// instructions and about 300 cycles a visit; sort 5 us, the rest around it 8 us).
// Tried on the way: one visit list for both kinds, entries two visits ahead,
// starting over when a kind blocks or unblocks (112-141 us: a restart every 2.7
// visits); partners by match_any (373 cycles a call).
template <int SD, bool HINTS, bool FULL, bool PACK>
__global__ void __launch_bounds__(DEC_WARPS * 32, 1) decode_kernel(DecArgs a) {
    extern __shared__ __align__(16) int smem_dec[];
    __shared__ __align__(8) uint64_t dist_bar;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = a.n, m = a.m, two_n = 2 * n, N1 = n + 1;
    constexpr int ES = SD == 2 ? 2 : 4;                   // bytes of a distance
    int* sd = smem_dec;                                   // staged distances (optional)
    const int dist_words = SD == 1 ? ((N1 * N1 + 3) & ~3) : SD == 2 ? (((N1 * N1 + 1) / 2 + 3) & ~3) : 0;
    int* sp = sd + dist_words;
    if (SD != 0 && threadIdx.x == 0) {
        mbar_init(&dist_bar, 1);
        mbar_arrive_expect_tx(&dist_bar, dist_words * 4u);
        // (the matrices are padded to 16 bytes in global memory)
        tma_bulk_g2s(sd, SD == 2 ? static_cast<const void*>(a.d16) : static_cast<const void*>(a.d32), dist_words * 4u, &dist_bar);
    }
    for (int i = threadIdx.x; i < N1; i += blockDim.x) sp[i] = a.p[i];
    int* list = sp + ((N1 + 3) & ~3) + warp * static_cast<int>(dec_warp_words(n, a.P));
    int* tdrop = list + (a.P > SORT_REGS_MAX ? 2 * a.P : a.P > 32 ? a.P : 32);   // drop time, -1 before
    int* vs = tdrop + (((n + 1) + 3) & ~3);               // log of the scheduled ops
    unsigned char* hv = reinterpret_cast<unsigned char*>(vs + ((two_n + 3) & ~3));
    __syncthreads();
    const float* keys = a.keys;
    if (a.keys2 != nullptr && a.ctl->sel == 1) keys = a.keys2;
    bool staged = SD == 0;
    const unsigned sd_addr = smem_u32(sd), log_addr = smem_u32(vs), lanebit = 1u << lane;
    // the distance from a place (row: shared address of, or index into, its
    // row) to the customer whose offset within a row off is
    auto dist = [&](unsigned row, unsigned off) -> int {
        if constexpr (SD == 2) return lds_u16(row + off);
        else if constexpr (SD == 1) return lds_b32(row + off);
        else return __ldg(reinterpret_cast<const int*>(reinterpret_cast<const char*>(a.d32) + row + off));
    };
    const unsigned row0 = SD == 0 ? 0u : sd_addr;
    for (int ch = blockIdx.x * DEC_WARPS + warp; ch < a.num; ch += gridDim.x * DEC_WARPS) {
        const float* kk = keys + static_cast<long long>(ch) * a.L;
        for (int i = lane; i <= n; i += 32) tdrop[i] = -1;
        if (HINTS)
            for (int i = lane; i < two_n; i += 32) hv[i] = static_cast<unsigned char>(hint_vehicle(kk[two_n + i], m));
        // ---- segmented key sort ----
        switch (a.P) {
            case 64: sort_ops<2>(kk, two_n, list); break;
            case 128: sort_ops<4>(kk, two_n, list); break;
            case 256: sort_ops<8>(kk, two_n, list); break;
            case 512: sort_ops<16>(kk, two_n, list); break;
            case 1024: sort_ops<32>(kk, two_n, list); break;
            default:
                if (a.P <= 32) sort_ops<1>(kk, two_n, list);
                else sort_ops_shared(kk, two_n, a.P, reinterpret_cast<unsigned long long*>(list), list);
        }
        if (!staged) {
            if (!mbar_wait_bounded(&dist_bar, 0)) {
                if (lane == 0) atomicExch(a.err, DEV_TIMEOUT_TMA);
                mbar_wait_bounded(&dist_bar, 0);          // one more bounded chance for the copy in flight
                return;
            }
            staged = true;
        }
        // ---- tie-break order: vehicle ranks (stable argsort of the m vehicle
        // keys) or, per op, cyclic distance from the hinted vehicle ----
        const float kv = (!HINTS && lane < m) ? __fadd_rn(kk[two_n + lane], 0.0f) : 0.0f;
        int rank = 0;
        for (int u = 0; !HINTS && u < m; ++u) {
            const float ku = __shfl_sync(FULL_MASK, kv, u);
            if (lane < m && (ku < kv || (ku == kv && u < lane))) ++rank;
        }
        // ---- multi-pass decode (Algorithm 2), lane v = vehicle v ----
        // Of a vehicle's stock two numbers count.  LOAD_MIN: room r = start load +
        // net (0 when a drop needs one more at the depot) and slack e = largest net
        // - net; start load + largest net = r + e.  A drop fits if r > 0, or if
        // e < Q and the pool has one left, a pickup if r < Q.  A drop lowers r, not
        // below 0 (there the start load grows and the pool gives one), and raises e;
        // a pickup raises r and lowers e, not below 0.
        // Eq. 13: r = stock on board, from Q; a drop fits if r > 0, a pickup if r < Q.
        const bool vehicle = lane < m;
        int room = FULL ? a.Q : 0, slack = 0, pool = a.R, done = 0;
        unsigned row = row0;
        // PACK: time << 10 | tie rank << 5 | (room == 0), with hints the rank added
        // per op; else the time, and the rest apart
        int flag = room == 0 ? 1 : 0, tv = 0;
        unsigned tkey = static_cast<unsigned>((HINTS ? 0 : rank * 32) + flag);
        unsigned entry = static_cast<unsigned>(lane) << 26;      // the log: vehicle, place in its route, op
        unsigned log_at = log_addr;
        bool okD = vehicle && (FULL ? room > 0 : a.Q > 0 && pool > 0), okP = vehicle && room < a.Q;
        bool anyD = __any_sync(FULL_MASK, okD), anyP = __any_sync(FULL_MASK, okP);
        int len = two_n;                       // list[0, len): ops not scheduled yet, priority order
        while (done < two_n) {
            const int before = done;
            int kept = 0;
            for (int base = 0; base < len; base += 32) {
                const bool in = base + lane < len;
                const int oi = in ? list[base + lane] : 0, mine = (oi >> 1) + 1;
                const bool is_drop = in && !(oi & 1), is_pick = in && (oi & 1);
                const int td = tdrop[mine], pm = sp[mine];
                // a drop's own pickup further down the chunk: found through the drop's
                // time slot, where such pickups leave their lane for a moment
                __syncwarp();
                if (is_pick && td < 0) tdrop[mine] = -2 - lane;
                __syncwarp();
                const int mate = is_drop ? -2 - tdrop[mine] : -1;
                __syncwarp();
                if (is_pick && td < 0) tdrop[mine] = -1;
                int ready = is_pick ? td + pm : 0;     // for a pickup whose drop is scheduled
                // bits 0-12 the op code 2c + isPickup, 16-20 the hinted vehicle, 21-25
                // the mate's lane, 31 whether there is one
                unsigned word = static_cast<unsigned>(oi + 2);
                if (HINTS) word |= static_cast<unsigned>(hv[oi]) << 16;
                if (mate > lane) word |= (static_cast<unsigned>(mate) << 21) | 0x80000000u;
                const unsigned drops = __ballot_sync(FULL_MASK, is_drop);
                unsigned picks = __ballot_sync(FULL_MASK, is_pick && td >= 0);
                int when = -1;                         // this lane's op: its vehicle's arrival, once scheduled
                // the next drop and the next pickup: bit, lane, word, distances
                unsigned bD = drops & (0u - drops), bP = picks & (0u - picks);
                unsigned jD = bit_index(bD), jP = bit_index(bP);
                unsigned wD = __shfl_sync(FULL_MASK, word, jD), wP = __shfl_sync(FULL_MASK, word, jP);
                int dD = dist(row, (wD & 0x1ffeu) * (ES / 2)), dP = dist(row, (wP & 0x1ffeu) * (ES / 2));
                for (;;) {
                    const unsigned eD = anyD ? bD : 0u, eP = anyP ? bP : 0u;
                    if (!(eD | eP)) break;
                    const bool pick = eP - 1u < eD - 1u;         // the earlier one (0: none)
                    const unsigned bit = pick ? eP : eD, w = pick ? wP : wD;
                    const int d = pick ? dP : dD;
                    const unsigned j = pick ? jP : jD;
                    // In program order, since nothing else hides a latency: the reduction,
                    // the search for the next two ops, the winner, their words, the votes,
                    // their distances.
                    // SelectVehicle: least arrival, then tie rank (unique per vehicle).
                    // With every time below 2^22 both fit one 32-bit key and one warp
                    // reduction; otherwise two reductions
                    const bool ok = pick ? okP : okD;
                    unsigned tie = 0u;
                    if (HINTS) {                       // cyclic distance from the hinted vehicle
                        const unsigned t0 = static_cast<unsigned>(lane) - ((w >> 16) & 31u);
                        tie = min(t0, t0 + static_cast<unsigned>(m)) * 32u;
                    }
                    unsigned least, own;
                    int first;
                    if constexpr (PACK) {
                        own = ok ? static_cast<unsigned>(d) * 1024u + tkey + tie : 0xffffffffu;
                        least = __reduce_min_sync(FULL_MASK, own);
                        first = static_cast<int>(least >> 10);
                    } else {
                        const unsigned arr = ok ? static_cast<unsigned>(tv + d) : 0xffffffffu;
                        first = static_cast<int>(__reduce_min_sync(FULL_MASK, arr));
                        own = arr == static_cast<unsigned>(first) ? tkey + tie : 0xffffffffu;
                        least = __reduce_min_sync(FULL_MASK, own);
                    }
                    // the two ops that may follow: past this one, its mate among them
                    const unsigned link = (w >> 31) << ((w >> 21) & 31u), past = 0u - 2u * bit;
                    picks |= link;
                    const unsigned mD = drops & past, mP = picks & past;
                    bD = mD & (0u - mD);
                    bP = mP & (0u - mP);
                    jD = bit_index(bD);
                    jP = bit_index(bP);
                    const int wait = __shfl_sync(FULL_MASK, ready, j);
                    // the winner's update, by selects
                    const bool me = own == least;
                    const int step = me ? (pick ? 1 : -1) : 0;
                    room = __viaddmax_s32(room, step, 0);
                    slack = __viaddmax_s32(slack, -step, 0);
                    if (!FULL) pool -= pick ? 0 : static_cast<int>(least & 1u);
                    okD = vehicle && (room > 0 || (!FULL && slack < a.Q && pool > 0));
                    okP = vehicle && room < a.Q;
                    row = me ? row0 + (w & 0x1ffeu) * static_cast<unsigned>(N1 * (ES / 2)) : row;
                    wD = __shfl_sync(FULL_MASK, word, jD);
                    wP = __shfl_sync(FULL_MASK, word, jP);
                    anyD = __any_sync(FULL_MASK, okD);
                    anyP = __any_sync(FULL_MASK, okP);
                    // it leaves at its arrival, or once a pickup is ready (wait is 0 for a drop)
                    const int leave = max(first, wait);
                    flag = room == 0 ? 1 : 0;
                    if constexpr (PACK) {
                        const unsigned nk = static_cast<unsigned>(leave) * 1024u + static_cast<unsigned>((HINTS ? 0 : rank * 32) + flag);
                        tkey = me ? nk : tkey;
                    } else {
                        tv = me ? leave : tv;
                        tkey = static_cast<unsigned>((HINTS ? 0 : rank * 32) + flag);
                    }
                    sts_if(me, log_at, static_cast<int>(entry | (w & 0x1fffu)));
                    dD = dist(row, (wD & 0x1ffeu) * (ES / 2));
                    dP = dist(row, (wP & 0x1ffeu) * (ES / 2));
                    log_at += 4u;
                    entry += me ? 1u << 13 : 0u;
                    when = (lanebit & bit) ? first : when;
                    ready = (lanebit & link) ? first + pm : ready;
                }
                // drop times, and the ops still unscheduled, order kept, for the next
                // pass (in place)
                const bool fin = when >= 0;
                __syncwarp();
                if (fin && is_drop) tdrop[mine] = when;
                done += __popc(__ballot_sync(FULL_MASK, fin));
                const bool keep = in && !fin;
                const unsigned bal = __ballot_sync(FULL_MASK, keep);
                if (keep) list[kept + __popc(bal & (lanebit - 1u))] = oi;
                kept += __popc(bal);
                __syncwarp();
            }
            len = kept;
            if (done == before) break;
        }
        if constexpr (PACK) tv = static_cast<int>(tkey >> 10);
        const int cnt = static_cast<int>((entry >> 13) & 0x1fffu);
        // ---- outputs: routes, makespan, penalty fitness ----
        int ret = (lane < m && cnt > 0) ? tv + dist(row, 0u) : 0;
        for (int off = 16; off > 0; off >>= 1) ret = max(ret, __shfl_xor_sync(FULL_MASK, ret, off));
        int incl = lane < m ? cnt : 0;
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(FULL_MASK, incl, off);
            if (lane >= off) incl += y;
        }
        const int excl = incl - (lane < m ? cnt : 0);
        int32_t* off_out = a.off + static_cast<long long>(ch) * (m + 1);
        if (lane < m) off_out[lane] = excl;
        if (lane == 0) off_out[m] = done;
        int32_t* ops_out = a.ops + static_cast<long long>(ch) * two_n;
        __syncwarp();
        for (int base = 0; base < done; base += 32) {
            const bool in = base + lane < done;
            const unsigned w = in ? static_cast<unsigned>(vs[base + lane]) : 0u;
            const int at = __shfl_sync(FULL_MASK, excl, w >> 26) + static_cast<int>((w >> 13) & 0x1fffu);
            if (in) ops_out[at] = static_cast<int>(w & 0x1fffu);
        }
        if (lane == 0) {
            const int un = two_n - done;
            a.z[ch] = ret;
            a.unsched[ch] = un;
            a.fitness[ch] = static_cast<long long>(ret) + PENALTY * un;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// v/m rounded up to the smallest float with m * alpha >= v: the hint that
// hint_vehicle maps back to v
__device__ inline float hint_of(int v, int m) {
    float x = __fdiv_rn(static_cast<float>(v), static_cast<float>(m));
    for (int it = 0; it < 4 && __dmul_rn(static_cast<double>(x), static_cast<double>(m)) < static_cast<double>(v); ++it)
        x = __int_as_float(__float_as_int(x) + 1);
    return x;
}

__global__ void encode_kernel(const int32_t* __restrict__ ops, const int32_t* __restrict__ off, int n, int m,
                              int layout, float* __restrict__ base) {
    // ALNS seed encoding: pi_o = (r-1)/L_v (here r is 0-based); vehicle key
    // v/m, or the hint of vehicle v for each of its ops
    const bool hints = layout == VRPRPD_LAYOUT_HINTS;
    for (int i = threadIdx.x; i < (hints ? 4 * n : 2 * n); i += blockDim.x) base[i] = 0.0f;
    __syncthreads();
    for (int v = 0; v < m; ++v) {
        const int L = off[v + 1] - off[v];
        for (int r = threadIdx.x; r < L; r += blockDim.x) {
            const int oi = ops[off[v] + r] - 2;
            base[oi] = __fdiv_rn(static_cast<float>(r), static_cast<float>(L));
            if (hints) base[2 * n + oi] = hint_of(v, m);
        }
    }
    if (!hints)
        for (int v = threadIdx.x; v < m; v += blockDim.x)
            base[2 * n + v] = __fdiv_rn(static_cast<float>(v), static_cast<float>(m));
}

// Ascending bitonic sort of P (a power of two) keys in shared memory; all
// threads of the block.
static __device__ void seed_sort(unsigned long long* a, int P) {
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

// Construction seeds of the warm start (Section 4.4.4), block h = 0, 1, 2:
// nearest neighbour, load-balanced, shortest processing time.  A customer
// order (the nearest-neighbour tour from the depot; workload 2 d(0,c) + p_c
// descending; p ascending; ties to the smaller id), then every drop before
// every pickup in that order: priority r/(2n) on the r-th drop and (n+r)/(2n)
// on its pickup.  Vehicle part: keys v/m, or hints naming vehicle 0 except
// for the load-balanced seed, whose hints follow a least-loaded assignment in
// its order (ties to the lower index).  out holds 3 chromosomes of L keys.
__global__ void __launch_bounds__(256) seed_kernel(const int32_t* __restrict__ d, const int32_t* __restrict__ p, int n,
                                                   int m, int layout, int L, float* __restrict__ out) {
    extern __shared__ __align__(16) unsigned long long sq[];
    __shared__ unsigned long long wmin[8];
    __shared__ int curc;
    const int h = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N1 = n + 1;
    int P = 1;
    while (P < n) P <<= 1;
    unsigned char* vis = reinterpret_cast<unsigned char*>(sq + P);
    float* o = out + static_cast<size_t>(h) * L;
    if (h == 0) {
        for (int c = tid; c <= n; c += blockDim.x) vis[c] = 0;
        if (tid == 0) curc = 0;
        __syncthreads();
        for (int r = 0; r < n; ++r) {
            const int cur = curc;
            unsigned long long best = ~0ull;
            for (int c = 1 + tid; c <= n; c += blockDim.x)
                if (!vis[c]) {
                    const unsigned long long k =
                        (static_cast<unsigned long long>(static_cast<unsigned>(__ldg(d + cur * N1 + c))) << 16) |
                        static_cast<unsigned long long>(c);
                    best = k < best ? k : best;
                }
            for (int off = 16; off > 0; off >>= 1) {
                const unsigned long long x = __shfl_xor_sync(0xffffffffu, best, off);
                best = x < best ? x : best;
            }
            if (lane == 0) wmin[warp] = best;
            __syncthreads();
            if (tid == 0) {
                unsigned long long b = wmin[0];
                for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) b = wmin[w] < b ? wmin[w] : b;
                const int c = static_cast<int>(b & 0xFFFF);
                vis[c] = 1;
                sq[r] = static_cast<unsigned long long>(c);
                curc = c;
            }
            __syncthreads();
        }
    } else {
        for (int i = tid; i < P; i += blockDim.x) {
            unsigned long long k = ~0ull;
            if (i < n) {
                const int c = i + 1;
                const long long pc = __ldg(p + c);
                const long long v = h == 1 ? (1ll << 46) - (2ll * __ldg(d + c) + pc) : pc;
                k = (static_cast<unsigned long long>(v) << 16) | static_cast<unsigned long long>(c);
            }
            sq[i] = k;
        }
        seed_sort(sq, P);
    }
    __syncthreads();
    const float two_n = static_cast<float>(2 * n);
    for (int r = tid; r < n; r += blockDim.x) {
        const int c = static_cast<int>(sq[r] & 0xFFFF);
        o[2 * (c - 1)] = __fdiv_rn(static_cast<float>(r), two_n);
        o[2 * (c - 1) + 1] = __fdiv_rn(static_cast<float>(n + r), two_n);
    }
    if (layout != VRPRPD_LAYOUT_HINTS) {
        for (int v = tid; v < m; v += blockDim.x) o[2 * n + v] = __fdiv_rn(static_cast<float>(v), static_cast<float>(m));
    } else if (h != 1) {
        for (int i = tid; i < 2 * n; i += blockDim.x) o[2 * n + i] = hint_of(0, m);
    } else if (warp == 0) {
        long long load = lane < m ? 0 : 0x7fffffffffffffffll;
        for (int r = 0; r < n; ++r) {
            const int c = static_cast<int>(sq[r] & 0xFFFF);
            long long bl = load;
            int bv = lane;
            for (int off = 16; off > 0; off >>= 1) {
                const long long ol = __shfl_xor_sync(0xffffffffu, bl, off);
                const int ov = __shfl_xor_sync(0xffffffffu, bv, off);
                if (ol < bl || (ol == bl && ov < bv)) { bl = ol; bv = ov; }
            }
            if (lane == bv) load += 2ll * __ldg(d + c) + __ldg(p + c);
            if (lane == 0) {
                const float a = hint_of(bv, m);
                o[2 * n + 2 * (c - 1)] = a;
                o[2 * n + 2 * (c - 1) + 1] = a;
            }
        }
    }
}

__global__ void init_pop_kernel(float* __restrict__ keys, const float* __restrict__ base, int pop, int L, int warm,
                                int variants, float eps, unsigned long long key, unsigned long long wkey) {
    const long long total = static_cast<long long>(pop) * L;
    const unsigned long long per = static_cast<unsigned long long>(L) + 2ull;
    const float top = 1.0f - 1.0f / 16777216.0f;
    for (long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; idx < total;
         idx += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int s = static_cast<int>(idx / L), g = static_cast<int>(idx - static_cast<long long>(s) * L);
        float x;
        if (s < warm) {
            // variant 0 is the ALNS encoding itself; with four or more variants
            // the last three perturb the three construction seeds (base + L,
            // + 2L, + 3L), the others the ALNS encoding
            const int nv = variants > 0 ? variants : 1;
            const int var = s % nv;
            const float* bs = base + static_cast<size_t>(nv >= 4 && var >= nv - 3 ? var - (nv - 3) + 1 : 0) * L;
            if (var == 0) {
                x = bs[g];
            } else {
                const float u = draw_key(draw(wkey, static_cast<unsigned long long>(var) * L + g));
                const float e = __fmul_rn(__fsub_rn(__fmul_rn(u, 2.0f), 1.0f), eps);
                x = __fadd_rn(bs[g], e);
                x = x < 0.0f ? 0.0f : x;
                x = x > top ? top : x;
            }
        } else {
            x = draw_key(draw(key, static_cast<unsigned long long>(s) * per + 2ull + g));
        }
        keys[idx] = x;
    }
}

// Fitness, rank by (fitness, index), generation best.  An element's rank is the
// number of smaller ones, so elements are independent: four threads count for
// each, over keys staged RANK_TILE at a time, and it goes to rank[count].
// pop 1024: 13.5 us as a bitonic sort in one CTA, 6.5 us now.  The thread that
// holds the best also turns the generation over (advance): nothing after it
// reads the old state.
constexpr int RANK_PER_BLOCK = 64, RANK_TILE = 2048;
__global__ void __launch_bounds__(4 * RANK_PER_BLOCK) rank_kernel(const int32_t* __restrict__ zdec,
                                                                  const int32_t* __restrict__ un, int pop, int advance,
                                                                  BrkgaCtl* ctl, int32_t* __restrict__ rank,
                                                                  long long* __restrict__ fit,
                                                                  long long* __restrict__ trace) {
    __shared__ unsigned long long keys[RANK_TILE];
    // four consecutive lanes share an element
    const int i = blockIdx.x * RANK_PER_BLOCK + (threadIdx.x >> 2), part = threadIdx.x & 3;
    auto key_of = [&](int k) {
        const long long f = static_cast<long long>(zdec[k]) + PENALTY * un[k];
        return (static_cast<unsigned long long>(f) << 24) | static_cast<unsigned>(k);
    };
    const unsigned long long own = i < pop ? key_of(i) : 0ull;
    int below = 0;
    for (int t0 = 0; t0 < pop; t0 += RANK_TILE) {
        const int len = min(RANK_TILE, pop - t0);
        __syncthreads();
        for (int k = threadIdx.x; k < len; k += blockDim.x) keys[k] = key_of(t0 + k);
        __syncthreads();
#pragma unroll 8
        for (int k = part; k < len; k += 4) below += keys[k] < own ? 1 : 0;
    }
    below += __shfl_xor_sync(FULL_MASK, below, 1);
    below += __shfl_xor_sync(FULL_MASK, below, 2);
    if (i >= pop || part != 0) return;
    rank[below] = i;
    fit[i] = static_cast<long long>(own >> 24);
    if (below == 0) {
        if (trace) trace[ctl->gen] = static_cast<long long>(own >> 24);
        if (advance) {
            ctl->sel ^= 1;
            ctl->gen += 1;
        }
    }
}

// The decoder's makespans against the evaluator's (complete decodes).
__global__ void check_kernel(const int32_t* __restrict__ zdec, const int32_t* __restrict__ un,
                             const int32_t* __restrict__ zev, const uint32_t* __restrict__ stev, int pop, BrkgaCtl* ctl) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < pop && un[i] == 0 && (zev[i] != zdec[i] || stev[i] != 0u)) atomicAdd(&ctl->mismatches, 1);
}

// Next population: elites, biased-crossover children, mutants; one block per
// slot, so its parents are drawn once per thread and not once per gene.  ctl has
// been turned over already: ctl->sel is the buffer to fill.
__global__ void __launch_bounds__(128) evolve_kernel(float* __restrict__ buf0, float* __restrict__ buf1,
                                                     const BrkgaCtl* __restrict__ ctl, const int32_t* __restrict__ rank,
                                                     int pop, int L, int Ne, int Nc, float rho, unsigned long long key) {
    const int s = blockIdx.x, sel = ctl->sel;
    const float* cur = sel == 0 ? buf1 : buf0;
    float* nxt = (sel == 0 ? buf0 : buf1) + static_cast<long long>(s) * L;
    if (s < Ne) {
        const float* from = cur + static_cast<long long>(rank[s]) * L;
        for (int g = threadIdx.x; g < L; g += blockDim.x) nxt[g] = from[g];
        return;
    }
    const unsigned long long cb = (static_cast<unsigned long long>(ctl->gen) * static_cast<unsigned long long>(pop) +
                                   static_cast<unsigned long long>(s)) * (static_cast<unsigned long long>(L) + 2ull);
    if (s < Ne + Nc) {
        const float* e = cur + static_cast<long long>(rank[draw_below(draw(key, cb + 0ull), Ne)]) * L;
        const float* o = cur + static_cast<long long>(rank[Ne + draw_below(draw(key, cb + 1ull), pop - Ne)]) * L;
        for (int g = threadIdx.x; g < L; g += blockDim.x) {
            const float u = draw_key(draw(key, cb + 2ull + g));
            nxt[g] = u < rho ? e[g] : o[g];
        }
    } else {
        for (int g = threadIdx.x; g < L; g += blockDim.x) nxt[g] = draw_key(draw(key, cb + 2ull + g));
    }
}

// ---------------------------------------------------------------------------
struct DecPlan {
    int blocks = 0, P = 0;
    size_t smem = 0;
    int smem_dist = 0;
};

static int plan_decode(const vrprpd_instance* I, int num, DecPlan* D) {
    VRP_CHECK(I->m <= 32, VRPRPD_EINVAL, "BRKGA decoding needs m <= 32");
    VRP_CHECK(2 * I->n + I->m <= 8192, VRPRPD_EINVAL, "BRKGA decoding needs 2n + m <= 8192");
    const int n = I->n, N1 = n + 1;
    D->P = pow2_at_least(2 * n);
    const size_t warp_words = dec_warp_words(n, D->P);
    const size_t base_words = ((N1 + 3) & ~3) + DEC_WARPS * warp_words;
    // distances staged in shared memory: 16-bit when they fit in that (room for
    // two blocks per SM at n = 200), else 32-bit for small n, else read from L2
    const size_t dist_words32 = (static_cast<size_t>(N1) * N1 + 3) & ~3;
    const size_t dist_words16 = ((static_cast<size_t>(N1) * N1 + 1) / 2 + 3) & ~3;
    size_t dist_words = 0;
    D->smem_dist = 0;
    if (I->has_d16 && (base_words + dist_words16) * 4 + 64 <= I->smem_optin) {
        D->smem_dist = 2;
        dist_words = dist_words16;
    } else if ((base_words + dist_words32) * 4 + 64 <= I->smem_optin && N1 <= 240) {
        D->smem_dist = 1;
        dist_words = dist_words32;
    }
    D->smem = (base_words + dist_words) * 4;
    VRP_CHECK(D->smem + 64 <= I->smem_optin, VRPRPD_EINVAL, "decode shared memory %zu too large", D->smem);
    return VRPRPD_OK;
}

// The decoder instance for these arguments.
template <int SD, bool HINTS, bool FULL>
static const void* decode_fn3(bool pack) {
    return pack ? reinterpret_cast<const void*>(&decode_kernel<SD, HINTS, FULL, true>)
                : reinterpret_cast<const void*>(&decode_kernel<SD, HINTS, FULL, false>);
}
template <int SD>
static const void* decode_fn2(bool hints, bool full, bool pack) {
    if (hints) return full ? decode_fn3<SD, true, true>(pack) : decode_fn3<SD, true, false>(pack);
    return full ? decode_fn3<SD, false, true>(pack) : decode_fn3<SD, false, false>(pack);
}
static const void* decode_fn(int sd, bool hints, bool full, bool pack) {
    if (sd == 2) return decode_fn2<2>(hints, full, pack);
    if (sd == 1) return decode_fn2<1>(hints, full, pack);
    return decode_fn2<0>(hints, full, pack);
}
static const void* decode_fn(const DecArgs& a) {
    return decode_fn(a.smem_dist, a.layout == VRPRPD_LAYOUT_HINTS, a.load_full != 0, a.pack != 0);
}
// The grid of the instance that decodes with arguments a: as many blocks as
// the chromosomes need, at most what stays resident on all SMs.
static int plan_decode_grid(const vrprpd_instance* I, int num, const DecArgs& a, DecPlan* D) {
    const void* fn = decode_fn(a);
    { int rc_ = ensure_smem_limit(fn); if (rc_) return rc_; }
    int occ = 0;
    VRP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, DEC_WARPS * 32, D->smem));
    VRP_CHECK(occ > 0, VRPRPD_EINVAL, "decode block does not fit");
    D->blocks = std::max(1, std::min((num + DEC_WARPS - 1) / DEC_WARPS, occ * I->num_sms));
    return VRPRPD_OK;
}
static cudaError_t launch_decode(const DecArgs& a, int blocks, size_t smem, cudaStream_t s) {
    DecArgs args = a;
    void* params[] = {&args};
    return cudaLaunchKernel(decode_fn(a), dim3(blocks), dim3(DEC_WARPS * 32), params, smem, s);
}

static DecArgs dec_args(const vrprpd_instance* I, const DecPlan& D, int num, int layout) {
    DecArgs a{};
    a.num = num;
    a.n = I->n;
    a.m = I->m;
    a.R = I->R;
    a.Q = I->Q;
    a.load_full = (I->flags & VRPRPD_LOAD_FULL) != 0;
    a.layout = layout;
    a.L = layout == VRPRPD_LAYOUT_HINTS ? 4 * I->n : 2 * I->n + I->m;
    a.P = D.P;
    a.d32 = I->d32;
    a.p = I->p;
    a.smem_dist = D.smem_dist;
    a.d16 = I->d16;
    a.err = I->err;
    // a decoded schedule is a precedence graph of the instance's ops, so no
    // time exceeds (2n+1) max d + n max p
    const long long bound = (2ll * I->n + 1) * I->maxd + static_cast<long long>(I->n) * I->maxp;
    a.pack = bound < (1ll << 22) && I->m <= 32 ? 1 : 0;
    return a;
}

}  // namespace vrp

using namespace vrp;

extern "C" void vrprpd_brkga_params_default(vrprpd_brkga_params* P) {
    if (!P) return;
    P->pop = 30000;
    P->generations = 20000;
    P->warm_slots = -1;        // ceil(0.15 * pop), worked out by vrprpd_brkga_run
    P->warm_variants = 20;
    P->elite_frac = 0.15f;
    P->mutant_frac = 0.15f;
    P->rho = 0.7f;
    P->eps = 0.03f;
    P->layout = VRPRPD_LAYOUT_VKEYS;
}

extern "C" int vrprpd_brkga_decode(const vrprpd_instance* I, const float* keys, int32_t num, int32_t layout,
                                   int32_t* ops, int32_t* off, int32_t* z, int32_t* unsched, int64_t* fitness,
                                   void* stream) {
    VRP_CHECK(I && keys && ops && off && z && unsched && fitness, VRPRPD_EINVAL, "NULL argument");
    VRP_CHECK(num >= 0, VRPRPD_EINVAL, "negative count");
    VRP_CHECK(layout == VRPRPD_LAYOUT_VKEYS || layout == VRPRPD_LAYOUT_HINTS, VRPRPD_EINVAL, "unknown key layout %d",
              layout);
    if (num == 0) return VRPRPD_OK;
    DecPlan D;
    int rc = plan_decode(I, num, &D);
    if (rc) return rc;
    DecArgs a = dec_args(I, D, num, layout);
    rc = plan_decode_grid(I, num, a, &D);
    if (rc) return rc;
    a.keys = keys;
    a.ops = ops;
    a.off = off;
    a.z = z;
    a.unsched = unsched;
    a.fitness = reinterpret_cast<long long*>(fitness);
    VRP_CUDA(launch_decode(a, D.blocks, D.smem, static_cast<cudaStream_t>(stream)));
    return VRPRPD_OK;
}

extern "C" int vrprpd_brkga_run(const vrprpd_instance* I, const vrprpd_brkga_params* P, const vrprpd_solution* warm,
                                uint64_t seed, vrprpd_solution* best, int64_t* best_fitness, int64_t* trace,
                                float* final_keys, void* stream_) {
    VRP_CHECK(I && P && best && best->ops && best->off, VRPRPD_EINVAL, "NULL argument");
    VRP_CHECK(P->pop >= 2 && P->pop <= 16384, VRPRPD_EINVAL, "pop must lie in [2, 16384]");
    VRP_CHECK(P->generations >= 1, VRPRPD_EINVAL, "generations must be >= 1");
    VRP_CHECK(batched_supported(I), VRPRPD_EINVAL, "the batched evaluator does not support this instance");
    VRP_CHECK(P->layout == VRPRPD_LAYOUT_VKEYS || P->layout == VRPRPD_LAYOUT_HINTS, VRPRPD_EINVAL,
              "unknown key layout %d", P->layout);
    const int n = I->n, m = I->m, pop = P->pop, G = P->generations;
    const int L = P->layout == VRPRPD_LAYOUT_HINTS ? 4 * n : 2 * n + m;
    int Ne = static_cast<int>(std::floor(static_cast<double>(P->elite_frac) * pop));
    int Nm = static_cast<int>(std::floor(static_cast<double>(P->mutant_frac) * pop));
    if (Ne < 1) Ne = 1;
    if (Ne + Nm > pop) Nm = pop - Ne;
    const int Nc = pop - Ne - Nm;
    // a negative count asks for Section 4.4.4's 15% of the population, rounded up
    const int warm_req = P->warm_slots < 0 ? static_cast<int>((15ll * pop + 99) / 100) : P->warm_slots;
    const int warm_slots = warm ? std::min(warm_req, pop) : 0;
    // work already queued on the caller's stream comes first
    VRP_CUDA(cudaStreamSynchronize(static_cast<cudaStream_t>(stream_)));
    cudaStream_t s;
    VRP_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    // device buffers
    const size_t keys_b = static_cast<size_t>(pop) * L * 4;
    char* mem = nullptr;
    size_t used = 0;
    auto take = [&](size_t bytes) {            // an offset first, a pointer once mem is there
        char* p = mem ? mem + used : nullptr;
        used += (bytes + 255) & ~static_cast<size_t>(255);
        return p;
    };
    auto cleanup = [&]() {
        if (mem) cudaFreeAsync(mem, s);
        cudaStreamSynchronize(s);
        cudaStreamDestroy(s);
    };
    float *buf0 = nullptr, *buf1 = nullptr, *base = nullptr;
    int32_t *dops = nullptr, *doff = nullptr, *zdec = nullptr, *un = nullptr, *zev = nullptr, *rank = nullptr,
            *wops = nullptr, *woff = nullptr;
    uint32_t* stev = nullptr;
    long long *fitd = nullptr, *fit = nullptr, *dtrace = nullptr;
    BrkgaCtl* ctl = nullptr;
    for (int pass = 0; pass < 2; ++pass) {     // the total, then the pieces of one allocation
        if (pass == 1 && pool_alloc(reinterpret_cast<void**>(&mem), used, s) != cudaSuccess) {
            mem = nullptr;
            cudaGetLastError();
            cleanup();
            set_error("BRKGA: device allocation failed");
            return VRPRPD_ENOMEM;
        }
        used = 0;
        buf0 = reinterpret_cast<float*>(take(keys_b));
        buf1 = reinterpret_cast<float*>(take(keys_b));
        base = reinterpret_cast<float*>(take(static_cast<size_t>(4) * L * 4));   // ALNS encoding + 3 seeds
        dops = reinterpret_cast<int32_t*>(take(static_cast<size_t>(pop) * 2 * n * 4));
        doff = reinterpret_cast<int32_t*>(take(static_cast<size_t>(pop) * (m + 1) * 4));
        zdec = reinterpret_cast<int32_t*>(take(pop * 4));
        un = reinterpret_cast<int32_t*>(take(pop * 4));
        fitd = reinterpret_cast<long long*>(take(pop * 8));
        zev = reinterpret_cast<int32_t*>(take(pop * 4));
        stev = reinterpret_cast<uint32_t*>(take(pop * 4));
        rank = reinterpret_cast<int32_t*>(take(pop * 4));
        fit = reinterpret_cast<long long*>(take(pop * 8));
        dtrace = reinterpret_cast<long long*>(take(static_cast<size_t>(G) * 8));
        ctl = reinterpret_cast<BrkgaCtl*>(take(sizeof(BrkgaCtl)));
        wops = reinterpret_cast<int32_t*>(take(2 * n * 4));
        woff = reinterpret_cast<int32_t*>(take((m + 1) * 4));
    }
    const unsigned long long key = stream_key(seed, RNG_STREAM_BRKGA), wkey = stream_key(seed, RNG_STREAM_WARM);
    BrkgaCtl c0{0, 0, 0, 0};
    cudaError_t e = cudaMemcpyAsync(ctl, &c0, sizeof(c0), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(base, 0, static_cast<size_t>(4) * L * 4, s);
    if (warm && e == cudaSuccess) {
        e = cudaMemcpyAsync(wops, warm->ops, 2 * n * 4, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(woff, warm->off, (m + 1) * 4, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) encode_kernel<<<1, 256, 0, s>>>(wops, woff, n, m, P->layout, base);
        if (e == cudaSuccess) {
            int Ps = 1;
            while (Ps < n) Ps <<= 1;
            seed_kernel<<<3, 256, static_cast<size_t>(Ps) * 8 + n + 16, s>>>(I->d32, I->p, n, m, P->layout, L,
                                                                          base + L);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) {
        init_pop_kernel<<<std::min<long long>((static_cast<long long>(pop) * L + 255) / 256, 4096), 256, 0, s>>>(
            buf0, base, pop, L, warm_slots, P->warm_variants, P->eps, key, wkey);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) { cleanup(); set_error("BRKGA init: %s", cudaGetErrorString(e)); return VRPRPD_ECUDA; }
    DecPlan D;
    int rc = plan_decode(I, pop, &D);
    if (rc) { cleanup(); return rc; }
    DecArgs da = dec_args(I, D, pop, P->layout);
    rc = plan_decode_grid(I, pop, da, &D);
    if (rc) { cleanup(); return rc; }
    da.keys = buf0;
    da.keys2 = buf1;
    da.ctl = ctl;
    da.ops = dops;
    da.off = doff;
    da.z = zdec;
    da.unsched = un;
    da.fitness = fitd;
    // One generation: decode, then beside each other the evaluator's check of the
    // decoded routes (on s2) and the ranking with the next population (evolve).
    cudaStream_t s2 = nullptr;
    cudaEvent_t forked = nullptr, checked = nullptr;
    auto release = [&]() {
        if (forked) cudaEventDestroy(forked);
        if (checked) cudaEventDestroy(checked);
        if (s2) cudaStreamDestroy(s2);
        cleanup();
    };
    e = cudaStreamCreateWithFlags(&s2, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&forked, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&checked, cudaEventDisableTiming);
    if (e != cudaSuccess) { release(); set_error("BRKGA setup: %s", cudaGetErrorString(e)); return VRPRPD_ECUDA; }
    auto enqueue = [&](bool evolve) -> int {
        VRP_CUDA(launch_decode(da, D.blocks, D.smem, s));
        VRP_CUDA(cudaEventRecord(forked, s));
        VRP_CUDA(cudaStreamWaitEvent(s2, forked, 0));
        int r = evaluate_device(I, dops, doff, pop, zev, stev, s2);
        if (r) return r;
        check_kernel<<<(pop + 255) / 256, 256, 0, s2>>>(zdec, un, zev, stev, pop, ctl);
        VRP_CUDA(cudaGetLastError());
        VRP_CUDA(cudaEventRecord(checked, s2));
        rank_kernel<<<(pop + RANK_PER_BLOCK - 1) / RANK_PER_BLOCK, 4 * RANK_PER_BLOCK, 0, s>>>(
            zdec, un, pop, evolve ? 1 : 0, ctl, rank, fit, dtrace);
        if (evolve) evolve_kernel<<<pop, 128, 0, s>>>(buf0, buf1, ctl, rank, pop, L, Ne, Nc, P->rho, key);
        VRP_CUDA(cudaGetLastError());
        VRP_CUDA(cudaStreamWaitEvent(s, checked, 0));
        return VRPRPD_OK;
    };
    rc = VRPRPD_OK;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    if (G > 1) {
        cudaError_t ce = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
        if (ce != cudaSuccess) { set_error("graph capture: %s", cudaGetErrorString(ce)); rc = VRPRPD_ECUDA; }
        if (rc == VRPRPD_OK) {
            rc = enqueue(true);
            ce = cudaStreamEndCapture(s, &graph);
        }
        if (rc == VRPRPD_OK && ce != cudaSuccess) { set_error("graph capture: %s", cudaGetErrorString(ce)); rc = VRPRPD_ECUDA; }
        if (rc == VRPRPD_OK) {
            ce = cudaGraphInstantiate(&exec, graph, 0);
            if (ce != cudaSuccess) { set_error("graph instantiate: %s", cudaGetErrorString(ce)); rc = VRPRPD_ECUDA; }
        }
        for (int g = 0; rc == VRPRPD_OK && g < G - 1; ++g) {
            ce = cudaGraphLaunch(exec, s);
            if (ce != cudaSuccess) { set_error("graph launch: %s", cudaGetErrorString(ce)); rc = VRPRPD_ECUDA; }
        }
    }
    if (rc == VRPRPD_OK) rc = enqueue(false);               // last generation: evaluate and rank only
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (rc) { release(); return rc; }
    e = cudaStreamSynchronize(s);
    BrkgaCtl cend{};
    int best_idx = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&cend, ctl, sizeof(cend), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&best_idx, rank, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    long long bf = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bf, fit + best_idx, 8, cudaMemcpyDeviceToHost, s);
    int32_t bz = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(best->ops, dops + static_cast<long long>(best_idx) * 2 * n, 2 * n * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(best->off, doff + static_cast<long long>(best_idx) * (m + 1), (m + 1) * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bz, zdec + best_idx, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && trace) e = cudaMemcpyAsync(trace, dtrace, static_cast<size_t>(G) * 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && final_keys)
        e = cudaMemcpyAsync(final_keys, cend.sel == 0 ? buf0 : buf1, keys_b, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) { release(); set_error("BRKGA copy-out: %s", cudaGetErrorString(e)); return VRPRPD_ECUDA; }
    best->makespan = bz;
    best->status = 0;
    if (best_fitness) *best_fitness = bf;
    release();
    if (cend.mismatches != 0) {
        set_error("BRKGA: %d decoded makespans disagree with the evaluator", cend.mismatches);
        return VRPRPD_ECUDA;
    }
    return VRPRPD_OK;
}
