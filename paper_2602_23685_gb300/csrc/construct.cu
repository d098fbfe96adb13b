// The paper's three-phase initial solution (Section 4.2.5), one CTA:
//   1. sweep: customers by exact angle around the depot (half plane, then
//      the integer cross product, then id; by id without coordinates), a
//      bitonic sort with that comparison; cut into m' = min(m, R) sectors of
//      equal count (customer k of the order in sector floor(k m' / n));
//   2. load balancing on w_c = 2 d(0,c) + p_c (one warp): while the spread
//      of the sector workloads is 10% of their mean or more, the heaviest
//      sector (lowest index on ties) hands its boundary customer to its
//      lighter neighbour (lower index on ties), unless that would leave the
//      neighbour at least as heavy as the heaviest was; at most 4n moves;
//   3. nearest-neighbour routes (one warp per vehicle): vehicle v serves
//      its sector alone from the depot at time 0 with b = min(Q, floor(R/m'))
//      resources, each step taking the feasible op that completes first (a
//      drop while a resource is left: its arrival; a pickup of a dropped
//      customer: max(arrival, T_drop + p)), ties by travel, then drop before
//      pickup, then op code.
// The steps of 2 and 3 depend on each other, so their latency is what counts:
// workloads and states in shared memory, a sector per lane in 2 (three
// reductions and two exchanges a move), a customer per lane in 3 (two reductions
// a step).  With the instance's limits (schedule times below 2^27, d below 2^17)
// every sum and key fits 32 bits.  One thread for 2 and one per vehicle for 3
// made the whole start (constructor, evaluation and the calls around them) 656 us
// at n=200 m=6 and 1789 us at n=1000 m=20; now 179 and 240 us.
// Vehicle v's ops start at 2 * (first customer index of its sector), so the
// route offsets follow from the sector bounds.  The refinement rounds that
// follow run in the ALNS kernel's local search.
#include <algorithm>

#include "device_common.cuh"
#include "internal.h"

namespace vrp {
namespace {

__device__ __forceinline__ bool angle_before(const int32_t* xy, int a, int b) {
    const long long ax = xy[2 * a] - xy[0], ay = xy[2 * a + 1] - xy[1];
    const long long bx = xy[2 * b] - xy[0], by = xy[2 * b + 1] - xy[1];
    const int ha = (ay < 0 || (ay == 0 && ax < 0)) ? 1 : 0, hb = (by < 0 || (by == 0 && bx < 0)) ? 1 : 0;
    if (ha != hb) return ha < hb;
    const long long cr = ax * by - ay * bx;
    if (cr != 0) return cr > 0;
    return a < b;
}

__global__ void __launch_bounds__(1024) construct_kernel(const int32_t* __restrict__ xy, const int32_t* __restrict__ d,
                                                         const int32_t* __restrict__ p, int n, int m, int R, int Q,
                                                         int32_t* __restrict__ ops, int32_t* __restrict__ off) {
    extern __shared__ __align__(16) int csm[];
    __shared__ int start[33];
    __shared__ int Wl[32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, N1 = n + 1;
    int P = 1;
    while (P < n) P <<= 1;
    int* rdy = csm;                            // [n+1] pickup-ready times; first the workloads
    int* ord = rdy + N1;                       // [P]
    unsigned char* state = reinterpret_cast<unsigned char*>(ord + P);   // [n+1]
    const int mp = m < R ? m : R;
    const int b = min(Q, R / mp);
    // 1. sweep order (entries past n sort last)
    for (int i = tid; i < P; i += blockDim.x) ord[i] = i < n ? i + 1 : 0x7fffffff;
    for (int c = tid; c <= n; c += blockDim.x) {
        state[c] = 0;
        rdy[c] = c ? 2 * __ldg(d + c) + __ldg(p + c) : 0;
    }
    if (tid < 32) Wl[tid] = 0;
    __syncthreads();
    if (xy) {
        for (int size = 2; size <= P; size <<= 1) {
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int i = tid; i < P / 2; i += blockDim.x) {
                    const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                    const bool asc = (lo & size) == 0;
                    const int x = ord[lo], y = ord[hi];
                    const bool y_first = y != 0x7fffffff && (x == 0x7fffffff || angle_before(xy, y, x));
                    if (y_first == asc) { ord[lo] = y; ord[hi] = x; }
                }
                __syncthreads();
            }
        }
    }
    // 2. sectors and load balancing
    for (int k = tid; k < n; k += blockDim.x)
        atomicAdd(&Wl[static_cast<int>((static_cast<long long>(k) * mp) / n)], rdy[ord[k]]);
    if (tid <= mp) start[tid] = static_cast<int>((static_cast<long long>(tid) * n + mp - 1) / mp);
    __syncthreads();
    if (warp == 0) {
        const bool sector = lane < mp;
        int W = sector ? Wl[lane] : 0, lo = sector ? start[lane] : 0, hi = sector ? start[lane + 1] : 0;
        const long long tot = __reduce_add_sync(FULL_MASK, static_cast<unsigned>(W));     // below 2^27
        for (int mv = 0; mv < 4 * n && mp > 1; ++mv) {
            // the heaviest sector (lowest index) and the least load
            const unsigned top = __reduce_max_sync(FULL_MASK, sector ? (static_cast<unsigned>(W) << 5) | (31u - lane) : 0u);
            const int h = 31 - static_cast<int>(top & 31u), Wh = static_cast<int>(top >> 5);
            const int least = __reduce_min_sync(FULL_MASK, sector ? W : 0x7fffffff);
            if (10ll * mp * (Wh - least) < tot) break;
            const int Wp = __shfl_sync(FULL_MASK, W, (h - 1) & 31), Wn = __shfl_sync(FULL_MASK, W, (h + 1) & 31);
            const int g = h > 0 && (h + 1 >= mp || Wp <= Wn) ? h - 1 : h + 1;
            const int hlo = __shfl_sync(FULL_MASK, lo, h), hhi = __shfl_sync(FULL_MASK, hi, h);
            if (hlo == hhi) break;
            const int wc = rdy[ord[g < h ? hlo : hhi - 1]];
            if ((g < h ? Wp : Wn) + wc >= Wh) break;
            if (lane == g) {
                W += wc;
                if (g < h) ++hi; else --lo;
            }
            if (lane == h) {
                W -= wc;
                if (g < h) ++lo; else --hi;
            }
        }
        if (sector) {
            start[lane] = lo;
            if (lane == mp - 1) start[mp] = hi;
        }
    }
    __syncthreads();
    for (int c = tid; c <= n; c += blockDim.x) rdy[c] = 0;
    __syncthreads();
    // 3. nearest-neighbour routes
    for (int v = warp; v < mp; v += static_cast<int>(blockDim.x >> 5)) {
        const int k0 = start[v], k1 = start[v + 1];
        int t = 0, loc = 0, out = 0, w = 2 * k0;
        for (int step = 0; step < 2 * (k1 - k0); ++step) {
            // completion time first, then travel (below 2^17), drop before pickup, op code
            unsigned fin = 0xffffffffu, rest = 0xffffffffu;
            for (int k = k0 + lane; k < k1; k += 32) {
                const int c = ord[k], st = state[c];
                if (st == 2 || (st == 0 && out >= b)) continue;
                const int dl = __ldg(d + loc * N1 + c);
                const unsigned f = static_cast<unsigned>(st == 1 ? max(t + dl, rdy[c]) : t + dl);
                const unsigned q = (static_cast<unsigned>(dl) << 13) | (static_cast<unsigned>(st) << 12) | static_cast<unsigned>(2 * c + st);
                if (f < fin || (f == fin && q < rest)) { fin = f; rest = q; }
            }
            const unsigned best = __reduce_min_sync(FULL_MASK, fin);
            const unsigned pick = __reduce_min_sync(FULL_MASK, fin == best ? rest : 0xffffffffu);
            const int o = static_cast<int>(pick & 0xfffu), c = o >> 1;
            __syncwarp();
            if (lane == 0) {
                state[c] = (o & 1) ? 2 : 1;
                if (!(o & 1)) rdy[c] = static_cast<int>(best) + __ldg(p + c);
                ops[w] = o;
            }
            out += (o & 1) ? -1 : 1;
            t = static_cast<int>(best);
            loc = c;
            ++w;
            __syncwarp();
        }
    }
    for (int v = tid; v <= m; v += blockDim.x) off[v] = v <= mp ? 2 * start[v] : 2 * n;
}

}  // namespace

// Launch the constructor into device buffers ops (2n) and off (m+1).
int construct_paper_device(const vrprpd_instance* I, int32_t* ops, int32_t* off, cudaStream_t stream) {
    VRP_CHECK(I->R >= 1 && I->Q >= 1, VRPRPD_EINVAL, "initial solution needs R >= 1 and Q >= 1");
    VRP_CHECK(I->m <= 32, VRPRPD_EINVAL, "the three-phase constructor needs m <= 32");
    const int n = I->n;
    int P = 1;
    while (P < n) P <<= 1;
    const size_t smem = static_cast<size_t>(n + 1) * 4 + static_cast<size_t>(P) * 4 + n + 1 + 16;
    VRP_CHECK(smem <= I->smem_optin, VRPRPD_EINVAL, "n=%d too large for the constructor", n);
    { int rc_ = ensure_smem_limit(reinterpret_cast<const void*>(&construct_kernel)); if (rc_) return rc_; }
    construct_kernel<<<1, 1024, smem, stream>>>(I->has_coords ? I->coords : nullptr, I->d32, I->p, n, I->m, I->R,
                                               I->Q, ops, off);
    VRP_CUDA(cudaGetLastError());
    return VRPRPD_OK;
}

}  // namespace vrp
