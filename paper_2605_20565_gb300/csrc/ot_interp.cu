// ot_interp.cu -- single-op kernels: locate, trilinear and delta-kernel interpolation.
// Persistent grid-stride launches (a few blocks per SM).
#include <algorithm>
#include <type_traits>

#include "ot_internal.h"
#include "ot_points.cuh"
#include "ot_queue.cuh"

namespace ot {

namespace {

template <bool LEARNED>
__global__ void __launch_bounds__(256) k_locate(TreeView t, const double* __restrict__ x,
                                                const double* __restrict__ y, const double* __restrict__ z, int64_t n,
                                                int32_t* __restrict__ host, unsigned long long* n_miss) {
    // the learned search inlined with the root network in shared memory: 10M points 268 -> 245 us
    __shared__ RootModel s_root;
    if (LEARNED) stage_root<LEARNED>(t, s_root);
    unsigned miss = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t X[3];
        int h = -1;
        if (fixpoint3(x[i], y[i], z[i], X)) {
            const uint64_t q = morton3((uint32_t)(X[0] >> 32), (uint32_t)(X[1] >> 32), (uint32_t)(X[2] >> 32));
            if (LEARNED) {
                const uint32_t c = map_cell(t, q);
                const int ca = (int)t.lmap[c], ce = map_end(t, c);
                h = ce - ca <= 1 ? ca
                                 : learned_in_cell_inline(t.key, &s_root, t.mids, t.models, t.n, t.n_leaf, ca, ce, q,
                                                          t.fallbacks, t.err);
            } else {
                h = search_plain(t, q);
            }
        } else {
            ++miss;
        }
        host[i] = h;
    }
    if (miss) {
        atomicOr(t.err, (unsigned)OT_DEV_OUTSIDE);
        if (n_miss) atomicAdd(n_miss, (unsigned long long)miss);
    }
}

template <typename T, bool LEARNED, bool MATES>
__global__ void __launch_bounds__(256) k_trilinear(TreeView t, const double* __restrict__ x,
                                                   const double* __restrict__ y, const double* __restrict__ z,
                                                   int64_t n, const int32_t* __restrict__ host_in,
                                                   const T* __restrict__ field, const T* __restrict__ pyr,
                                                   T* __restrict__ u, int32_t* __restrict__ host_out) {
    // warp-aligned iteration: every lane of a warp runs the same trip count (the trilinear
    // routine is warp-cooperative)
    using Q = typename std::conditional<MATES, HostQueue, WarpQueue>::type;
    __shared__ Q s_queue[256 / 32];
    __shared__ RootModel s_root;
    Q& wq = s_queue[threadIdx.x >> 5];
    stage_root<LEARNED>(t, s_root);
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = warp0 * 32; base < n; base += nwarps * 32) {
        const int64_t i = base + lane;
        const bool inr = i < n;
        T o[3];
        int hin = -1;
        bool active = inr;
        if (inr && host_in) {
            hin = host_in[i];
            if (hin < 0 || hin >= t.n) {
                // no host (outside the cube) or an index that is not a leaf: no value
                if (hin >= t.n) atomicOr(t.err, (unsigned)OT_DEV_OUTSIDE);
                active = false;
            }
        }
        const double xi = inr ? x[i] : 0.0, yi = inr ? y[i] : 0.0, zi = inr ? z[i] : 0.0;
        int h;
        if constexpr (MATES)
            h = trilinear_mates<T, LEARNED>(t, s_root, field, pyr, wq, active, xi, yi, zi, hin, o);
        else
            h = trilinear_queued<T, LEARNED>(t, s_root, field, pyr, wq, active, xi, yi, zi, hin, o);
        if (inr) {
            u[i] = o[0];
            u[n + i] = o[1];
            u[2 * n + i] = o[2];
            if (host_out) host_out[i] = h;
        }
    }
}

// Flags the cell means that the points' level-mates take (need: one byte per mean).
__global__ void __launch_bounds__(256) k_mark_means(TreeView t, const double* __restrict__ x,
                                                    const double* __restrict__ y, const double* __restrict__ z,
                                                    int64_t n, const int32_t* __restrict__ host_in,
                                                    uint8_t* __restrict__ need) {
    __shared__ WarpQueue s_queue[256 / 32];
    __shared__ RootModel s_root;  // (not read: the plain search finds the same leaves)
    WarpQueue& wq = s_queue[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = warp0 * 32; base < n; base += nwarps * 32) {
        const int64_t i = base + lane;
        uint64_t X[3] = {0, 0, 0};
        int hin = -1;
        bool ok = i < n;
        if (ok && host_in) {
            hin = host_in[i];
            ok = hin >= 0 && hin < t.n;
        }
        ok = ok && fixpoint3(x[i], y[i], z[i], X);
        TriCorners<float> c8;
        tri_corners<float, false>(t, s_root, wq, ok, X, ok ? hin : -1, c8);
        if (ok)
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (c8.lvl[k] > c8.l) need[c8.mean(t, k)] = 1;
    }
}

template <typename T, int K, bool LEARNED>
__global__ void __launch_bounds__(256) k_delta(TreeView t, const double* __restrict__ x,
                                               const double* __restrict__ y, const double* __restrict__ z, int64_t n,
                                               const T* __restrict__ field, T* __restrict__ u,
                                               int32_t* __restrict__ host_out) {
    __shared__ DeltaStage<T> s_stage[256 / 32];
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // markers per warp at a time: 32, fewer (4 at least) when there are not that many for every warp
    const int64_t per = min((int64_t)32, max((int64_t)4, (n + nwarps - 1) / nwarps));
    for (int64_t base = per * warp; base < n; base += per * nwarps)
        delta_markers<T, K, LEARNED>(t, field, s_stage[threadIdx.x >> 5], x, y, z, n, base, base + per, u, host_out);
}

size_t mean_flags_at(const ot_octree* t, size_t elem) { return (pyramid_bytes(t, elem) + 255) & ~(size_t)255; }

template <typename Kern>
unsigned persistent_grid(Kern k, int block, size_t smem, int64_t n) {
    const int per_sm = blocks_per_sm((const void*)k, block, smem);
    int64_t need = (n + block - 1) / block;
    int64_t g = std::min<int64_t>((int64_t)num_sms() * per_sm, need);
    return (unsigned)std::max<int64_t>(g, 1);
}

template <typename Kern>
ot_status prep_smem(Kern k, size_t smem) {
    if (smem > 48 * 1024) OT_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return OT_OK;
}

} // namespace

ot_status launch_locate(const ot_octree* t, const double* x, const double* y, const double* z, int64_t n, int search,
                        int32_t* host, unsigned long long* n_miss, cudaStream_t s) {
    if (n == 0) return OT_OK;
    const bool learned = search == OT_LEARNED;
    TreeView v = tree_view(t);
    const size_t smem = 0;
    const int block = 256;
    if (learned) {
        auto k = k_locate<true>;
        ot_status st = prep_smem(k, smem);
        if (st != OT_OK) return st;
        k<<<persistent_grid(k, block, smem, n), block, smem, s>>>(v, x, y, z, n, host, n_miss);
    } else {
        auto k = k_locate<false>;
        ot_status st = prep_smem(k, smem);
        if (st != OT_OK) return st;
        k<<<persistent_grid(k, block, smem, n), block, smem, s>>>(v, x, y, z, n, host, n_miss);
    }
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

template <typename T>
ot_status launch_interp(const ot_octree* t, int kernel, const double* x, const double* y, const double* z, int64_t n,
                        const int32_t* host_in, int search, const T* field, T* u, int32_t* host_out, void* ws,
                        size_t ws_bytes, cudaStream_t s) {
    if (n == 0) return OT_OK;
    if (kernel == OT_TRILINEAR && (ws_bytes < interp_ws_bytes(t, kernel, sizeof(T)) || !ws || ((uintptr_t)ws & 15)))
        return OT_ERR_ARG;
    const bool learned = search == OT_LEARNED;
    TreeView v = tree_view(t);
    const size_t smem = 0;
    const int block = 256;
    ot_status st = OT_OK;
#define OT_LAUNCH(KERN, ...)                                                               \
    do {                                                                                   \
        auto k_ = KERN;                                                                    \
        if ((st = prep_smem(k_, smem)) != OT_OK) return st;                                \
        k_<<<persistent_grid(k_, block, smem, n * lanes), block, smem, s>>>(__VA_ARGS__);  \
    } while (0)
    const int64_t lanes = kernel == OT_TRILINEAR ? 1 : 8;  // per point
    if (kernel == OT_TRILINEAR) {
        // cell means of the field (refined level-mates), in the caller's workspace: those that the
        // level-mate table reads; without it every one or, when the points are few against the
        // leaves, those that they read, flagged first (flags after the means in the workspace).
        // Flagging costs about what interpolating does (71 ps per point) and 3 ps per leaf, all means 15
        // ps per leaf: on 9.3M leaves, flagged against all, 1,000 points 85 and 172 us, 400,000 139
        // and 214, 860,000 205 and 216 in FP32 (FP64 92 and 222, 186 and 279, 282 and 331)
        T* pyr = static_cast<T*>(ws);
        const uint8_t* need = t->d_need_flags;
        if (!t->d_mates && 8 * n + 2400000 < t->n) {
            uint8_t* flags = static_cast<uint8_t*>(ws) + mean_flags_at(t, sizeof(T));
            OT_CUDA(cudaMemsetAsync(flags, 0, need_flag_bytes(t), s));
            OT_LAUNCH(k_mark_means, v, x, y, z, n, host_in, flags);
            count_launch();
            if ((st = close_need_flags(t, flags, s)) != OT_OK) return st;
            need = flags;
        }
        if ((st = launch_pyramid<T>(t, field, pyr, need, s)) != OT_OK) return st;
        if (t->d_mates && learned)
            OT_LAUNCH((k_trilinear<T, true, true>), v, x, y, z, n, host_in, field, pyr, u, host_out);
        else if (t->d_mates)
            OT_LAUNCH((k_trilinear<T, false, true>), v, x, y, z, n, host_in, field, pyr, u, host_out);
        else if (learned)
            OT_LAUNCH((k_trilinear<T, true, false>), v, x, y, z, n, host_in, field, pyr, u, host_out);
        else
            OT_LAUNCH((k_trilinear<T, false, false>), v, x, y, z, n, host_in, field, pyr, u, host_out);
    } else if (kernel == OT_PESKIN4) {
        if (learned)
            OT_LAUNCH((k_delta<T, OT_PESKIN4, true>), v, x, y, z, n, field, u, host_out);
        else
            OT_LAUNCH((k_delta<T, OT_PESKIN4, false>), v, x, y, z, n, field, u, host_out);
    } else {
        if (learned)
            OT_LAUNCH((k_delta<T, OT_ROMA3, true>), v, x, y, z, n, field, u, host_out);
        else
            OT_LAUNCH((k_delta<T, OT_ROMA3, false>), v, x, y, z, n, field, u, host_out);
    }
#undef OT_LAUNCH
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

template ot_status launch_interp<float>(const ot_octree*, int, const double*, const double*, const double*, int64_t,
                                        const int32_t*, int, const float*, float*, int32_t*, void*, size_t,
                                        cudaStream_t);
template ot_status launch_interp<double>(const ot_octree*, int, const double*, const double*, const double*, int64_t,
                                         const int32_t*, int, const double*, double*, int32_t*, void*, size_t,
                                         cudaStream_t);

// Trilinear workspace: the cell means, then their flags.
size_t interp_ws_bytes(const ot_octree* t, int kernel, size_t elem) {
    return kernel == OT_TRILINEAR ? mean_flags_at(t, elem) + (need_flag_bytes(t) + 15) / 16 * 16 : 0;
}

} // namespace ot
