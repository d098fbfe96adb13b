// Instance construction: validation, device residency and the EUC_2D
// distance kernel (Section 5.1: TSPLIB edge weights as travel times).
#include <algorithm>
#include <cstdarg>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <set>
#include <utility>

#include "device_common.cuh"
#include "internal.h"

namespace vrp {

static thread_local char g_err[512] = "";

void set_error(const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

// d(i,j) for all pairs; one thread per entry; also tracks max(d).
__global__ void euc2d_kernel(const int32_t* __restrict__ coords, int N, int32_t* __restrict__ d32,
                             int* __restrict__ maxd) {
    long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    long long total = static_cast<long long>(N) * N;
    int local_max = 0;
    for (; idx < total; idx += static_cast<long long>(gridDim.x) * blockDim.x) {
        int i = static_cast<int>(idx / N), j = static_cast<int>(idx - static_cast<long long>(i) * N);
        int v = euc2d_exact(coords[2 * i], coords[2 * i + 1], coords[2 * j], coords[2 * j + 1]);
        d32[idx] = v;
        local_max = v > local_max ? v : local_max;
    }
    for (int o = 16; o > 0; o >>= 1) local_max = max(local_max, __shfl_xor_sync(FULL_MASK, local_max, o));
    if ((threadIdx.x & 31) == 0) atomicMax(maxd, local_max);
}

__global__ void narrow16_kernel(const int32_t* __restrict__ d32, uint16_t* __restrict__ d16, long long total) {
    for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        d16[i] = static_cast<uint16_t>(d32[i]);
}

int ensure_smem_limit(const void* kernel) {
    static std::mutex mu;
    static std::set<std::pair<const void*, int>> done;
    int dev = 0;
    VRP_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({kernel, dev})) return VRPRPD_OK;
    cudaFuncAttributes fa{};
    VRP_CUDA(cudaFuncGetAttributes(&fa, kernel));
    int optin = 0;
    VRP_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    VRP_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  optin - static_cast<int>(fa.sharedSizeBytes)));
    done.insert({kernel, dev});
    return VRPRPD_OK;
}

// ---------------------------------------------------------------------------
// Scratch pool.  A search call allocates up to tens of megabytes and frees them
// when it returns; the device's default pool hands such memory back to the
// system at the next synchronisation, and each call then maps it anew.  The
// library's own pool keeps up to POOL_KEEP bytes between calls, as long as an
// instance or a server is alive.  Allocation is stream-ordered, so calls on any
// threads and streams share it.  A served request's instance lives there too: a
// cudaFree waits for every kernel on the device, other requests' searches among
// them.  Measured: a one-generation BRKGA run at n=200 683 us before, 430 us now;
// eight requests of 50 to 300 customers on four slots 63.5 ms before, 39.9 ms now.
// ---------------------------------------------------------------------------
constexpr unsigned long long POOL_KEEP = 256ull << 20;
constexpr int POOL_DEVICES = 64;
static std::mutex g_pool_mu;
static cudaMemPool_t g_pool[POOL_DEVICES] = {};
static int g_pool_holds = 0;

cudaError_t pool_alloc(void** ptr, size_t bytes, cudaStream_t stream) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaMemPool_t pool = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_pool_mu);
        if (dev < POOL_DEVICES && !g_pool[dev]) {
            cudaMemPoolProps props{};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            unsigned long long keep = POOL_KEEP;
            e = cudaMemPoolCreate(&g_pool[dev], &props);
            if (e == cudaSuccess) e = cudaMemPoolSetAttribute(g_pool[dev], cudaMemPoolAttrReleaseThreshold, &keep);
            if (e != cudaSuccess) return e;
        }
        if (dev < POOL_DEVICES) pool = g_pool[dev];
    }
    return pool ? cudaMallocFromPoolAsync(ptr, bytes, pool, stream) : cudaMallocAsync(ptr, bytes, stream);
}

void pool_hold() {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    ++g_pool_holds;
}

void pool_release() {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    if (--g_pool_holds > 0) return;
    for (cudaMemPool_t& pool : g_pool) {
        if (pool) cudaMemPoolDestroy(pool);    // made again by the next call
        pool = nullptr;
    }
}

// Device memory of an instance: its own for the public calls, else the pool's.
static cudaError_t inst_alloc(vrprpd_instance* I, void** ptr, size_t bytes) {
    return I->pooled ? pool_alloc(ptr, bytes, I->stream) : cudaMalloc(ptr, bytes);
}
template <class T>
static cudaError_t inst_alloc(vrprpd_instance* I, T** ptr, size_t bytes) {
    return inst_alloc(I, reinterpret_cast<void**>(ptr), bytes);
}
static void inst_free(vrprpd_instance* I, void* ptr) {
    if (!ptr) return;
    if (I->pooled) cudaFreeAsync(ptr, I->stream);
    else cudaFree(ptr);
}
// host <-> device, done when it returns
static cudaError_t inst_copy(vrprpd_instance* I, void* dst, const void* src, size_t bytes, cudaMemcpyKind kind) {
    if (!I->pooled) return cudaMemcpy(dst, src, bytes, kind);
    const cudaError_t e = cudaMemcpyAsync(dst, src, bytes, kind, I->stream);
    return e == cudaSuccess ? cudaStreamSynchronize(I->stream) : e;
}

static size_t pad16(size_t bytes) { return (bytes + 15) & ~static_cast<size_t>(15); }

static int finish_create(vrprpd_instance* I, vrprpd_instance** out) {
    const int N = I->n + 1;
    const long long NN = static_cast<long long>(N) * N;
    // schedule-time bound: a path enters each op by a route edge or a pickup
    // edge once and ends with a return leg
    long long bound = (2ll * I->n + 1) * I->maxd + static_cast<long long>(I->n) * I->maxp;
    if (bound > 2147483646ll) {
        set_error("instance too large for int32 schedule times: (2n+1)*max(d) + n*max(p) = %lld", bound);
        return VRPRPD_EINVAL;
    }
    if (I->maxd < 65536) {
        VRP_CUDA(inst_alloc(I, &I->d16, pad16(NN * sizeof(uint16_t))));
        narrow16_kernel<<<256, 256, 0, I->stream>>>(I->d32, I->d16, NN);
        VRP_CUDA(cudaGetLastError());
        I->has_d16 = true;
    }
    VRP_CUDA(inst_alloc(I, &I->err, 16));
    VRP_CUDA(cudaMemsetAsync(I->err, 0, 16, I->stream));
    VRP_CUDA(cudaStreamSynchronize(I->stream));   // this creation's own work only
    *out = I;
    return VRPRPD_OK;
}

static int common_init(vrprpd_instance* I, const int32_t* p, int32_t n, int32_t m, int32_t R, int32_t Q,
                       uint32_t flags) {
    VRP_CHECK(n >= 1 && n <= (1 << 20), VRPRPD_EINVAL, "n=%d out of range [1, 2^20]", n);
    VRP_CHECK(m >= 1 && m <= 4096, VRPRPD_EINVAL, "m=%d out of range [1, 4096]", m);
    VRP_CHECK(R >= 0 && Q >= 1, VRPRPD_EINVAL, "need R >= 0 and Q >= 1 (R=%d Q=%d)", R, Q);
    VRP_CHECK(flags == VRPRPD_LOAD_MIN || flags == VRPRPD_LOAD_FULL, VRPRPD_EINVAL, "bad flags %u", flags);
    VRP_CHECK(p != nullptr, VRPRPD_EINVAL, "p is NULL");
    I->n = n;
    I->m = m;
    I->R = R;
    I->Q = Q;
    I->flags = flags;
    I->h_p.assign(n + 1, 0);
    for (int c = 1; c <= n; ++c) {
        VRP_CHECK(p[c - 1] >= 0, VRPRPD_EINVAL, "p[%d] = %d is negative", c - 1, p[c - 1]);
        I->h_p[c] = p[c - 1];
        I->maxp = I->h_p[c] > I->maxp ? I->h_p[c] : I->maxp;
    }
    VRP_CUDA(cudaGetDevice(&I->device));
    VRP_CUDA(cudaDeviceGetAttribute(&I->num_sms, cudaDevAttrMultiProcessorCount, I->device));
    int optin = 0;
    VRP_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, I->device));
    I->smem_optin = static_cast<size_t>(optin);
    // p, then the evaluator's ready-row template: -(p_c + 1) per customer, the
    // "already picked up" word in the depot's slot and past the last customer
    I->row_words = (n + 2 + 3) & ~3;
    const size_t p_words = (n + 1 + 63) & ~static_cast<size_t>(63);
    std::vector<int32_t> h(p_words + I->row_words, INT32_MIN);
    for (int c = 0; c <= n; ++c) h[c] = I->h_p[c];
    for (int c = 1; c <= n; ++c) h[p_words + c] = -1 - I->h_p[c];
    VRP_CUDA(inst_alloc(I, &I->p, h.size() * sizeof(int32_t)));
    I->rowt = I->p + p_words;
    VRP_CUDA(inst_copy(I, I->p, h.data(), h.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
    return VRPRPD_OK;
}

}  // namespace vrp

using namespace vrp;

static int create_from_coords(const int32_t* coords, const int32_t* p, int32_t n, int32_t m, int32_t R, int32_t Q,
                              uint32_t flags, bool pooled, cudaStream_t stream, vrprpd_instance** out) {
    VRP_CHECK(out != nullptr && coords != nullptr, VRPRPD_EINVAL, "coords/out is NULL");
    *out = nullptr;
    vrprpd_instance* I = new vrprpd_instance();
    pool_hold();
    I->pooled = pooled;
    I->stream = stream;
    int rc = common_init(I, p, n, m, R, Q, flags);
    if (rc != VRPRPD_OK) { vrprpd_instance_destroy(I); return rc; }
    const int N = n + 1;
    for (int i = 0; i < 2 * N; ++i)
        if (coords[i] > (1 << 20) || coords[i] < -(1 << 20)) {
            set_error("coordinate %d out of range [-2^20, 2^20]", coords[i]);
            vrprpd_instance_destroy(I);
            return VRPRPD_EINVAL;
        }
    I->h_coords.assign(coords, coords + 2 * N);
    I->has_coords = true;
    const long long NN = static_cast<long long>(N) * N;
    // the box of the points bounds every squared leg
    int lo[2] = {coords[0], coords[1]}, hi[2] = {coords[0], coords[1]};
    for (int i = 0; i < 2 * N; ++i) {
        lo[i & 1] = std::min(lo[i & 1], coords[i]);
        hi[i & 1] = std::max(hi[i & 1], coords[i]);
    }
    const long long dx = hi[0] - lo[0], dy = hi[1] - lo[1];
    I->coords24 = dx * dx + dy * dy < (1ll << 24);
    const bool half = dx * dx + dy * dy < EUC2D_HALF2_LIMIT;
    // one point past the last customer's, the depot's again: where the evaluator
    // puts a code out of range (no leg is longer than the instance's own)
    const size_t c_words = (2 * N + 2 + 63) & ~static_cast<size_t>(63);
    std::vector<int32_t> h(c_words + (half ? I->row_words : 0), 0);
    std::copy(coords, coords + 2 * N, h.begin());
    std::copy(coords, coords + 2, h.begin() + 2 * N);
    for (int i = 0; half && i <= N; ++i) {
        const __half2 v = __floats2half2_rn(static_cast<float>(h[2 * i] - lo[0]),
                                            static_cast<float>(h[2 * i + 1] - lo[1]));
        std::memcpy(&h[c_words + i], &v, 4);
    }
    int* dmax = nullptr;
    cudaError_t e = inst_alloc(I, &I->coords, h.size() * sizeof(int32_t));
    if (e == cudaSuccess && half) I->xy = reinterpret_cast<uint32_t*>(I->coords) + c_words;
    if (e == cudaSuccess) e = inst_alloc(I, &I->d32, pad16(NN * sizeof(int32_t)));
    if (e == cudaSuccess) e = inst_alloc(I, &dmax, sizeof(int));
    if (e == cudaSuccess) e = inst_copy(I, I->coords, h.data(), h.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemsetAsync(dmax, 0, sizeof(int), stream);
    if (e == cudaSuccess) {
        int blocks = static_cast<int>((NN + 255) / 256);
        blocks = blocks > 4096 ? 4096 : blocks;
        euc2d_kernel<<<blocks, 256, 0, stream>>>(I->coords, N, I->d32, dmax);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = inst_copy(I, &I->maxd, dmax, sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) {
        I->h_d.resize(NN);
        e = inst_copy(I, I->h_d.data(), I->d32, NN * sizeof(int32_t), cudaMemcpyDeviceToHost);
    }
    inst_free(I, dmax);
    if (e != cudaSuccess) {
        set_error("instance_create: %s", cudaGetErrorString(e));
        vrprpd_instance_destroy(I);
        return VRPRPD_ECUDA;
    }
    rc = finish_create(I, out);
    if (rc != VRPRPD_OK) vrprpd_instance_destroy(I);
    return rc;
}

extern "C" int vrprpd_instance_create(const int32_t* coords, const int32_t* p, int32_t n, int32_t m,
                                      int32_t R, int32_t Q, uint32_t flags, vrprpd_instance** out) {
    return create_from_coords(coords, p, n, m, R, Q, flags, false, nullptr, out);
}

int vrp::instance_create_on(const int32_t* coords, const int32_t* p, int32_t n, int32_t m, int32_t R, int32_t Q,
                            uint32_t flags, cudaStream_t stream, vrprpd_instance** out) {
    return create_from_coords(coords, p, n, m, R, Q, flags, true, stream, out);
}

extern "C" int vrprpd_instance_create_dist(const int32_t* d, const int32_t* p, int32_t n, int32_t m,
                                           int32_t R, int32_t Q, uint32_t flags, vrprpd_instance** out) {
    VRP_CHECK(out != nullptr && d != nullptr, VRPRPD_EINVAL, "d/out is NULL");
    *out = nullptr;
    vrprpd_instance* I = new vrprpd_instance();
    pool_hold();
    int rc = common_init(I, p, n, m, R, Q, flags);
    if (rc != VRPRPD_OK) { vrprpd_instance_destroy(I); return rc; }
    const long long NN = static_cast<long long>(n + 1) * (n + 1);
    for (long long i = 0; i < NN; ++i) {
        if (d[i] < 0) {
            set_error("d[%lld] = %d is negative", i, d[i]);
            vrprpd_instance_destroy(I);
            return VRPRPD_EINVAL;
        }
        I->maxd = d[i] > I->maxd ? d[i] : I->maxd;
    }
    I->h_d.assign(d, d + NN);
    cudaError_t e = cudaMalloc(&I->d32, pad16(NN * sizeof(int32_t)));
    if (e == cudaSuccess) e = cudaMemcpy(I->d32, d, NN * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        set_error("instance_create_dist: %s", cudaGetErrorString(e));
        vrprpd_instance_destroy(I);
        return VRPRPD_ECUDA;
    }
    rc = finish_create(I, out);
    if (rc != VRPRPD_OK) vrprpd_instance_destroy(I);
    return rc;
}

extern "C" void vrprpd_instance_destroy(vrprpd_instance* I) {
    if (!I) return;
    inst_free(I, I->d32);
    inst_free(I, I->d16);
    inst_free(I, I->coords);
    inst_free(I, I->p);
    inst_free(I, I->err);
    if (I->plain_scratch) cudaFree(I->plain_scratch);
    if (I->stage) cudaFree(I->stage);
    delete I;
    pool_release();
}

extern "C" int vrprpd_instance_get_dist(const vrprpd_instance* I, int32_t* d_host) {
    VRP_CHECK(I && d_host, VRPRPD_EINVAL, "NULL argument");
    std::memcpy(d_host, I->h_d.data(), I->h_d.size() * sizeof(int32_t));
    return VRPRPD_OK;
}

extern "C" int vrprpd_sync(const vrprpd_instance* I, void* stream) {
    VRP_CHECK(I, VRPRPD_EINVAL, "NULL instance");
    VRP_CUDA(cudaStreamSynchronize(static_cast<cudaStream_t>(stream)));
    int err = 0;
    VRP_CUDA(cudaMemcpy(&err, I->err, sizeof(int), cudaMemcpyDeviceToHost));
    if (err != DEV_OK) {
        VRP_CUDA(cudaMemset(I->err, 0, sizeof(int)));
        set_error("device-side error %d (bounded wait gave up)", err);
        return VRPRPD_ETIMEOUT;
    }
    return VRPRPD_OK;
}

extern "C" const char* vrprpd_last_error(void) { return g_err; }
