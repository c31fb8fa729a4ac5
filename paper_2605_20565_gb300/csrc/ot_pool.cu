// ot_pool.cu -- device memory of octrees and of the temporaries of their builds, from one
// stream-ordered pool per device; launch shapes looked up once.
//
// A re-adaptation frees an octree and builds the next one of about the same size.  From the
// default pool, which gives its memory back at every synchronisation (a build has some 25: the
// sizes of each level), and from cudaMalloc, mapping memory took more than half as long as the
// build's kernels (17.3M leaves, a re-adaptation 8.68 -> 6.74 ms).  This pool keeps up to
// POOL_KEEP bytes while octrees live on the device and gives everything back when the last one is
// destroyed.  Memory pools are safe to use from several threads and streams: a block is handed
// out again only after the work before its release, in stream order.
#include <map>
#include <mutex>
#include <tuple>

#include "ot_internal.h"

namespace ot {

namespace {

constexpr uint64_t POOL_KEEP = 4ULL << 30;
constexpr int MAX_DEVICES = 64;

struct Pool {
    cudaMemPool_t pool = nullptr;
    int octrees = 0;
};
std::mutex g_pool_mu;
Pool g_pools[MAX_DEVICES];

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

} // namespace

cudaError_t pool_malloc(void** p, size_t bytes, cudaStream_t s) {
    *p = nullptr;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaMallocAsync(p, bytes, s);
    cudaMemPool_t pool;
    {
        std::lock_guard<std::mutex> lock(g_pool_mu);
        if (!g_pools[dev].pool && (e = create_pool(dev, &g_pools[dev].pool)) != cudaSuccess) {
            g_pools[dev].pool = nullptr;
            return e;
        }
        pool = g_pools[dev].pool;
    }
    e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e != cudaSuccess) cudaGetLastError();  // returned here; the next call's launches do not report it again
    return e;
}

void pool_octree(int dev, int change) {
    if (dev < 0 || dev >= MAX_DEVICES) return;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    Pool& q = g_pools[dev];
    q.octrees += change;
    if (change < 0 && q.octrees == 0 && q.pool) cudaMemPoolTrimTo(q.pool, 0);
}

void wait_device(int dev) {
    int cur = dev;
    cudaGetDevice(&cur);
    if (cur != dev) cudaSetDevice(dev);
    cudaDeviceSynchronize();
    if (cur != dev) cudaSetDevice(cur);
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
    static std::map<std::tuple<const void*, int, size_t, int>, int> known;
    int dev = 0;
    cudaGetDevice(&dev);
    const auto key = std::make_tuple(fn, block, smem, dev);
    {
        std::lock_guard<std::mutex> lock(mu);
        const auto it = known.find(key);
        if (it != known.end()) return it->second;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, smem) != cudaSuccess || per_sm < 1) return 1;
    try {
        std::lock_guard<std::mutex> lock(mu);
        known[key] = per_sm;
    } catch (...) {  // no memory to keep it: asked for again
    }
    return per_sm;
}

} // namespace ot
