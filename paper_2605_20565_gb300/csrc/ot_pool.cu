// ot_pool.cu -- device memory of octrees and of the temporaries of their builds, from one
// stream-ordered pool per device; launch shapes looked up once.
//
// A re-adaptation frees an octree and builds the next one of about the same size.  From the
// default pool, which gives its memory back at every synchronisation (a build has some 25: the
// sizes of each level), and from cudaMalloc, mapping memory took more than half as long as the
// build's kernels (17.3M leaves, a re-adaptation 8.68 -> 6.74 ms).  This pool keeps up to
// POOL_KEEP bytes while octrees live on the device and gives them back when the last one is
// destroyed (one pool per device and context).  Memory pools are safe to use from several threads and streams: a block is handed
// out again only after the work before its release, in stream order.
#include <cuda.h>  // driver types only: the two driver calls below are reached through the runtime

#include <map>
#include <mutex>
#include <new>
#include <tuple>
#include <utility>

#include "ot_internal.h"

namespace ot {

namespace {

constexpr uint64_t POOL_KEEP = 4ULL << 30;
constexpr int MAX_DEVICES = 64;

struct Pool {
    cudaMemPool_t pool = nullptr;
    int octrees = 0;
    // a small cudaMalloc block that stays: without one the driver maps and unmaps memory for every small
    // block (a wait's, a batch's counters: creating a batch on 8 leaves 46 us with it, 151 without)
    void* neighbour = nullptr;
};
std::mutex g_pool_mu;
// by device and context: a pool dies with the context that it was made in, and the octrees that
// were left in it no longer count.  Never destroyed: an octree may be, by a static object of the
// caller's, after this library's own statics.
std::map<std::pair<int, unsigned long long>, Pool>& pools() {
    static auto* all = new std::map<std::pair<int, unsigned long long>, Pool>();
    return *all;
}

cudaError_t create_pool(int dev, cudaMemPool_t* out) {
    cudaMemPoolProps p{};
    p.allocType = cudaMemAllocationTypePinned;  // device memory that stays in place
    p.location.type = cudaMemLocationTypeDevice;
    p.location.id = dev;
    cudaError_t e = cudaMemPoolCreate(out, &p);
    if (e != cudaSuccess) return e;
    uint64_t keep = POOL_KEEP;
    return cudaMemPoolSetAttribute(*out, cudaMemPoolAttrReleaseThreshold, &keep);
}

// The current context's identity, made first if there is none yet.
unsigned long long made_context() {
    unsigned long long id = current_context_id();
    if (id == 0) {
        cudaFree(nullptr);
        id = current_context_id();
    }
    return id;
}

} // namespace

// Identity of the current CUDA context (0 when the driver does not say).  A context that was
// destroyed and created again -- cudaDeviceReset, for instance -- has a new identity; what the
// library keeps per device (memory pools, the address of its device array) belongs to one.
unsigned long long current_context_id() {
    using GetCurrent = CUresult (*)(CUcontext*);
    using GetId = CUresult (*)(CUcontext, unsigned long long*);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<GetCurrent>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetId>(f);
    });
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (get_current && get_id && get_current(&ctx) == CUDA_SUCCESS && ctx && get_id(ctx, &id) == CUDA_SUCCESS)
        return id;
    return 0;
}

cudaError_t pool_malloc(void** p, size_t bytes, cudaStream_t s) {
    *p = nullptr;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long context = made_context();
    cudaMemPool_t pool;
    try {
        std::lock_guard<std::mutex> lock(g_pool_mu);
        Pool& q = pools()[{dev, context}];
        if (!q.pool && (e = create_pool(dev, &q.pool)) != cudaSuccess) {
            q.pool = nullptr;
            return e;
        }
        pool = q.pool;
    } catch (const std::bad_alloc&) {
        return cudaErrorMemoryAllocation;
    }
    e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e != cudaSuccess) cudaGetLastError();  // returned here; the next call's launches do not report it again
    return e;
}

unsigned long long pool_octree_made(int dev) {
    const unsigned long long context = made_context();
    try {
        std::lock_guard<std::mutex> lock(g_pool_mu);
        Pool& q = pools()[{dev, context}];
        ++q.octrees;
        if (!q.neighbour && cudaMalloc(&q.neighbour, 64) != cudaSuccess) q.neighbour = nullptr, cudaGetLastError();
    } catch (const std::bad_alloc&) {  // not counted: the pool is given back with the others
    }
    return context;
}

void pool_octree_left(int dev, unsigned long long context) {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    Pool* q = nullptr;
    try {
        const auto it = pools().find({dev, context});
        if (it != pools().end()) q = &it->second;
    } catch (const std::bad_alloc&) {
    }
    if (!q || --q->octrees > 0 || !q->pool) return;
    int cur = dev;
    cudaGetDevice(&cur);
    if (cur != dev) cudaSetDevice(dev);
    // (a pool of another context than the device's may no longer exist)
    if (current_context_id() == context) cudaMemPoolTrimTo(q->pool, 0);
    if (cur != dev) cudaSetDevice(cur);
}

// Whether what was made in this context of the device is still there.  (After cudaDeviceReset it is not,
// and its addresses and handles may be those of something newer.)
bool context_lives(int dev, unsigned long long context) {
    if (context == 0) return true;
    int cur = dev;
    cudaGetDevice(&cur);
    if (cur != dev) cudaSetDevice(dev);
    const bool same = made_context() == context;
    if (cur != dev) cudaSetDevice(cur);
    return same;
}

// Until the work that the device has is done.  By cudaFree, which waits for every stream: unlike
// cudaDeviceSynchronize it is allowed while another thread captures a stream in its own mode or the
// relaxed one (that call is refused then and ends the capture).  (cudaFree of pool memory does not wait.)
// false when it could not be waited for.
bool wait_device(int dev) {
    int cur = dev;
    cudaGetDevice(&cur);
    if (cur != dev) cudaSetDevice(dev);
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, 64);
    e = e == cudaSuccess ? cudaFree(p) : cudaDeviceSynchronize();
    if (e != cudaSuccess || !p) cudaGetLastError();
    if (cur != dev) cudaSetDevice(cur);
    return e == cudaSuccess;
}

int num_sms() {
    static std::mutex mu;
    static int sms[MAX_DEVICES] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return 1;
    std::lock_guard<std::mutex> lock(mu);
    if (sms[dev] == 0) {
        cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
        if (sms[dev] < 1) return sms[dev] = 0, 1;
    }
    return sms[dev];
}

// Resident blocks per SM of a kernel (at least 1): a property of its code and the device, asked for
// once (the query takes longer than a launch).
int blocks_per_sm(const void* fn, int block, size_t smem) {
    static std::mutex mu;
    using Known = std::map<std::tuple<const void*, int, size_t, int>, int>;
    static auto* known = new (std::nothrow) Known();  // (never destroyed, as above)
    int dev = 0;
    cudaGetDevice(&dev);
    const auto key = std::make_tuple(fn, block, smem, dev);
    if (known) {
        std::lock_guard<std::mutex> lock(mu);
        const auto it = known->find(key);
        if (it != known->end()) return it->second;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, smem) != cudaSuccess || per_sm < 1) return 1;
    try {
        std::lock_guard<std::mutex> lock(mu);
        if (known) (*known)[key] = per_sm;
    } catch (...) {  // no memory to keep it: asked for again
    }
    return per_sm;
}

} // namespace ot
