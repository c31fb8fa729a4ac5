// ot_batch.cu -- persistent launches over every group of points (IBM markers with a delta
// kernel, point particles with trilinear interpolation), replayed from a CUDA graph.
//
// A graph replay first recomputes the pyramid of cell means of the field (refined trilinear
// level-mates read it; a few small launches), then runs the batch kernel: one launch over all
// groups, or, with the octree's level-mate table, a launch for the delta-kernel groups and
// one for the trilinear groups, each at its own occupancy.  Work is cut into tiles of
// 32 * tile points; warps take tiles from a global counter, the expensive marker groups first
// (their tiles come first in the tile space), so uneven groups balance across the SMs without
// a host round trip.  The counters are reset by a memset node captured in the same graph.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "ot_internal.h"
#include "ot_points.cuh"
#include "ot_queue.cuh"

struct ot_batch {
    const ot_octree* tree = nullptr;
    int device = 0;
    unsigned long long context = 0;  // the octree's, that its memory and graph belong to
    int n_groups = 0;
    std::vector<void*> bufs;   // per ordered group: point-order workspace and the ordered copies
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    unsigned* d_counter = nullptr;
    float* d_pyr = nullptr;    // pyramid of cell means, recomputed at every replay
    int kernels = 1;           // kernels in one replay of the graph
    // value records of the hot leaves' grid nodes (trilinear launch with the level-mate table): the
    // cells' entries, the list of the nodes, and per node the 8 values around it, rewritten from
    // the field at every replay
    void* d_cells = nullptr;
    uint2* d_nodes = nullptr;
    float* d_rec = nullptr;
    int64_t n_rec = 0;
};

namespace ot {

constexpr int MAX_GROUPS = 16;
constexpr int TRI_MINB = 4;  // register budget of the trilinear-only launch (level-mate table)

struct GroupDev {
    int kernel;
    const double *x, *y, *z;
    int64_t n;
    float* u;
    int32_t* host;
    int64_t tile0; // first tile of the group
};

struct BatchArgs {
    GroupDev g[MAX_GROUPS];
    int ng;
    int64_t ntiles;
    int pts;  // points per tile
};

// MINB: the register budget (blocks of 256 resident per SM it is compiled for); 3 is the
// default, 2 trades occupancy for no register spills and is picked with blocks_per_sm = 2.
// MATES: trilinear level-mates read from the octree's level-mate table instead of searched.
// KINDS: the group kinds the instance serves -- K_ALL, K_DELTA (delta-kernel groups only) or
// K_TRI (trilinear groups only: with the table it needs far fewer registers than the delta
// path, so it runs as its own launch at a higher occupancy).
enum { K_ALL = 0, K_DELTA = 1, K_TRI = 2 };
template <bool LEARNED, int MINB, bool MATES, int KINDS = K_ALL>
__global__ void __launch_bounds__(256, MINB) k_batch(TreeView t, BatchArgs a, const float* __restrict__ field,
                                               const float* __restrict__ pyr, unsigned* __restrict__ counter) {
    // per warp: the search's task list (with the table 32 host searches) or the delta kernel's stage,
    // whichever the warp's tile needs
    using Q = typename std::conditional<MATES && KINDS == K_TRI, HostQueue, WarpQueue>::type;
    using D = DeltaStage<float>;
    constexpr size_t bytes = KINDS == K_TRI ? sizeof(Q) : KINDS == K_DELTA ? sizeof(D)
                             : sizeof(Q) > sizeof(D) ? sizeof(Q) : sizeof(D);
    __shared__ __align__(16) unsigned char s_mem[256 / 32][(bytes + 15) / 16 * 16];
    __shared__ RootModel s_root;
    Q& wq = *reinterpret_cast<Q*>(s_mem[threadIdx.x >> 5]);
    D& sg = *reinterpret_cast<D*>(s_mem[threadIdx.x >> 5]);
    stage_root<LEARNED>(t, s_root);
    const int lane = threadIdx.x & 31;
    const int64_t tile_pts = a.pts;
    for (;;) {
        unsigned tl = 0;
        if (lane == 0) tl = atomicAdd(counter, 1u);
        tl = __shfl_sync(0xffffffffu, tl, 0);
        if ((int64_t)tl >= a.ntiles) break;
        int g = 0;
        while (g + 1 < a.ng && (int64_t)tl >= a.g[g + 1].tile0) ++g;
        const GroupDev& gr = a.g[g];
        const int64_t base = ((int64_t)tl - gr.tile0) * tile_pts;
        if (KINDS == K_DELTA || (KINDS == K_ALL && gr.kernel != OT_TRILINEAR)) {
            const int64_t end = min(base + tile_pts, gr.n);
            for (int64_t b = base; b < end; b += 32) {  // warp-uniform
                const int64_t e = min(b + 32, end);
                if (gr.kernel == OT_PESKIN4)
                    delta_markers<float, OT_PESKIN4, LEARNED>(t, field, sg, gr.x, gr.y, gr.z, gr.n, b, e, gr.u, gr.host);
                else
                    delta_markers<float, OT_ROMA3, LEARNED>(t, field, sg, gr.x, gr.y, gr.z, gr.n, b, e, gr.u, gr.host);
            }
            continue;
        }
        if constexpr (KINDS != K_DELTA) {
            for (int64_t i = base + lane; i - lane < min(base + tile_pts, gr.n); i += 32) {  // warp-uniform
                const bool active = i < gr.n;
                float o[3];
                const double x = active ? gr.x[i] : 0.0, y = active ? gr.y[i] : 0.0, z = active ? gr.z[i] : 0.0;
                int h;
                if constexpr (MATES)
                    h = trilinear_mates<float, LEARNED>(t, s_root, field, pyr, wq, active, x, y, z, -1, o);
                else
                    h = trilinear_queued<float, LEARNED>(t, s_root, field, pyr, wq, active, x, y, z, -1, o);
                if (active) {
                    gr.u[i] = o[0];
                    gr.u[gr.n + i] = o[1];
                    gr.u[2 * gr.n + i] = o[2];
                    if (gr.host) gr.host[i] = h;
                }
            }
        }
    }
}


// ------------------------------------------------------------------------------------------
// Value records of the hot leaves.  A leaf is hot when its level is at most the hot level (a level
// whose leaves receive several points per launch) and so at most the map level.  The 8
// level-mates of a point in a leaf of level l are the 8 level-l cells around one node of the
// level-l grid, the corner of the leaf in the point's octant, and the value a cell takes (its own,
// the coarser leaf's that covers it, its mean when refined) does not depend on which of the 8 is
// the host; neither does a cell past a face, which takes the value of the one before it.  So the
// record -- 24 floats by position, copied from a level-mate row at every replay -- is kept per node
// at the node's place in the level's (2^l + 1)^3 grid: the hot leaves of 50M uniform points on
// the many-bubble tree (154k leaves) have 0.2M nodes, 19 MB that stay in L2, where a record per
// (leaf, octant) took 118 MB that did not.  A point reads its cell's entry (leaf and level), computes
// the node from its coordinates and reads the 96-byte record (three 32-byte loads); values and
// sums are those of the level-mate row, so the results are bit-identical.
// What bounds the launch on random points is the traffic from L2 to the SMs (79% of its sector rate
// on 64 bubbles; DRAM 45%), so the records' smaller set gains where neighbouring points share
// lines: 20M particles in Morton order 315 -> 307 us, refreshing the records 78 -> 35 us; 50M in
// random order 1217 -> 1157 us, the refresh 40 -> 18 us.  Looking cells up first in a coarser
// table that stays in L1 gained 3% there and lost 5% on the others; loading the next row's
// positions ahead lost 2 to 10%.
// ------------------------------------------------------------------------------------------
// Packed entry of a cell: level << 28 | leaf, all ones where no hot leaf covers the cell.  Trees of
// 2^28 leaves or more keep leaf and level in two words.
template <bool WIDE> struct Cell;
template <> struct Cell<false> {
    using type = uint32_t;
    static __host__ __device__ uint32_t none() { return 0xFFFFFFFFu; }
    static __device__ uint32_t make(uint32_t leaf, int lv) { return ((uint32_t)lv << 28) | leaf; }
    static __device__ bool hot(uint32_t e) { return e != 0xFFFFFFFFu; }
    static __device__ int level(uint32_t e) { return (int)(e >> 28); }
    static __device__ int leaf(uint32_t e) { return (int)(e & 0xFFFFFFFu); }
};
template <> struct Cell<true> {
    using type = uint2;
    static __device__ uint2 none() { return make_uint2(0u, 0xFFFFFFFFu); }
    static __device__ uint2 make(uint32_t leaf, int lv) { return make_uint2(leaf, (uint32_t)lv); }
    static __device__ bool hot(uint2 e) { return e.y != 0xFFFFFFFFu; }
    static __device__ int level(uint2 e) { return (int)e.y; }
    static __device__ int leaf(uint2 e) { return (int)e.x; }
};
constexpr int REC_FLOATS = 24;
constexpr int MAX_HOT = 8;  // map levels are at most 8

// First node of every level's grid, from the tree's coarsest level on.
struct NodeGrid {
    uint32_t off[MAX_HOT + 2];
};
NodeGrid node_grid(int lmin, int hot_l) {
    NodeGrid g{};
    for (int l = lmin; l <= hot_l; ++l) {
        const uint32_t s = (1u << l) + 1u;
        g.off[l + 1] = g.off[l] + s * s * s;
    }
    return g;
}

// Entries of the level-map cells.
template <bool WIDE>
__global__ void k_cells(TreeView t, int hot_l, typename Cell<WIDE>::type* __restrict__ cells) {
    using C = Cell<WIDE>;
    const int64_t ncell = (int64_t)1 << (3 * t.lmap_level);
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x) {
        const uint4 d = t.desc[c];
        const int lv = (int)((d.z >> 16) & 0xFFu);
        cells[c] = (d.z & DESC_COVERED) && lv <= hot_l ? C::make(d.w, lv) : C::none();
    }
}

// The nodes of the hot leaves, each once (seen: one bit per node): the leaf whose row gives the
// record, and node | octant << 28 (at most 2^25 nodes).  nodes null: counts them only.
__global__ void k_hot_nodes(TreeView t, int hot_l, NodeGrid g, uint32_t* __restrict__ seen,
                            uint2* __restrict__ nodes, uint32_t* __restrict__ count) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < t.n; i += (int64_t)gridDim.x * blockDim.x) {
        const int l = t.level[i];
        if (l > hot_l) continue;
        uint32_t c[3];
        demorton3(t.key[i] >> (3 * (MAXLEVEL - l)), c[0], c[1], c[2]);
        const uint32_t s = (1u << l) + 1u;
        for (uint32_t o = 0; o < 8; ++o) {
            const uint32_t node = g.off[l] + (c[0] + (o & 1)) + s * ((c[1] + ((o >> 1) & 1)) + s * (c[2] + (o >> 2)));
            const uint32_t bit = 1u << (node & 31);
            if (atomicOr(seen + (node >> 5), bit) & bit) continue;
            const uint32_t at = atomicAdd(count, 1u);
            if (nodes) nodes[at] = make_uint2((uint32_t)i, node | (o << 28));
        }
    }
}

// One record per listed node, rewritten from the field and the cell means.
__global__ void __launch_bounds__(256) k_hot_records(TreeView t, const uint2* __restrict__ nodes, int64_t n_rec,
                                                     const float* __restrict__ field, const float* __restrict__ pyr,
                                                     float* __restrict__ rec) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_rec; r += (int64_t)gridDim.x * blockDim.x) {
        const uint2 nd = nodes[r];
        const uint4* row = t.mates + 2 * (8 * (long long)nd.x + (nd.y >> 28));
        const uint4 r0 = __ldg(row), r1 = __ldg(row + 1);
        const uint32_t sl[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
        float v[REC_FLOATS];
#pragma unroll
        for (int corner = 0; corner < 8; ++corner) {
            const uint32_t sv = sl[corner];
            const float4 f = Vec4<float>::load((sv >> 31) ? pyr : field, (long long)(sv & 0x7FFFFFFFu));
            v[3 * corner] = f.x, v[3 * corner + 1] = f.y, v[3 * corner + 2] = f.z;
        }
        float4* dst = reinterpret_cast<float4*>(rec + REC_FLOATS * (size_t)(nd.y & 0xFFFFFFFu));
#pragma unroll
        for (int k = 0; k < REC_FLOATS / 4; ++k) dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    }
}

// The default L2 priority, as the hint that a 32-byte load takes.
__device__ __forceinline__ uint64_t policy_normal() {
    uint64_t pol;
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// 32 bytes from global memory in one load (sm_100 and later), read-only path, L2 policy pol.
__device__ __forceinline__ void ld_nc_v8(const float* p, float* r, uint64_t pol) {
    asm("ld.global.nc.L2::cache_hint.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
        : "l"(p), "l"(pol));
}

// The trilinear launch with value records.  Per 32-point row: quantise, read the level of the
// level-map cell; a point in a hot cell takes its node's record and is done; the others (cold:
// deeper leaves, uncovered cells) are queued per warp and, whenever 32 are queued (and at the
// end), interpolated together by the level-mate-table routine with every lane busy.
template <bool LEARNED, bool WIDE>
__global__ void __launch_bounds__(256, TRI_MINB) k_tri_rec(TreeView t, BatchArgs a, const float* __restrict__ field,
                                                          const float* __restrict__ pyr,
                                                          unsigned* __restrict__ counter,
                                                          const typename Cell<WIDE>::type* __restrict__ cells,
                                                          const float* __restrict__ rec, NodeGrid grid) {
    // per warp of the block: its host task list and its queue of cold points (dynamic shared
    // memory sized by the block's warps: what the block does not use is left to the L1 cache)
    extern __shared__ __align__(16) unsigned char tri_smem[];
    HostQueue* s_queue = reinterpret_cast<HostQueue*>(tri_smem);
    long long (*s_cold)[64] = reinterpret_cast<long long (*)[64]>(tri_smem + sizeof(HostQueue) * (blockDim.x >> 5));
    __shared__ RootModel s_root;
    // Morton spreading of 8-bit cell coordinates (bit b -> bit 3b): the level-map cell of a point
    // is spread[cx] | spread[cy] << 1 | spread[cz] << 2 (map levels are at most 8)
    __shared__ uint32_t s_spread[256];
    for (int v = threadIdx.x; v < 256; v += blockDim.x) s_spread[v] = (uint32_t)part1by2((uint32_t)v);
    __shared__ uint32_t s_off[MAX_HOT + 2];
    if (threadIdx.x < MAX_HOT + 2) s_off[threadIdx.x] = grid.off[threadIdx.x];
    const int wid = threadIdx.x >> 5;
    HostQueue& wq = s_queue[wid];
    long long* cq = s_cold[wid];
    stage_root<LEARNED>(t, s_root);
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int cell_shift = MAXLEVEL - t.lmap_level;  // of the 21-bit coordinates
    const int64_t tile_pts = a.pts;
    // the positions and results stream through once: evict-first (.cs), so that they push out
    // neither the cells' entries nor the records
    const uint64_t normal = policy_normal();
    using C = Cell<WIDE>;
    int qn = 0;  // queued cold points (warp-uniform)
    // the first cnt queued points, one per lane (warp-wide)
    auto drain = [&](int cnt) {
        const bool act = lane < cnt;
        const long long it = act ? cq[lane] : 0;
        const GroupDev& gq = a.g[(int)(it >> 40)];
        const int64_t i = it & ((1LL << 40) - 1);
        const double x = act ? gq.x[i] : 0.0, y = act ? gq.y[i] : 0.0, z = act ? gq.z[i] : 0.0;
        float o[3];
        const int h = trilinear_mates<float, LEARNED>(t, s_root, field, pyr, wq, act, x, y, z, -1, o);
        if (act) {
            gq.u[i] = o[0];
            gq.u[gq.n + i] = o[1];
            gq.u[2 * gq.n + i] = o[2];
            if (gq.host) gq.host[i] = h;
        }
    };
    for (;;) {
        unsigned tl = 0;
        if (lane == 0) tl = atomicAdd(counter, 1u);
        tl = __shfl_sync(0xffffffffu, tl, 0);
        if ((int64_t)tl >= a.ntiles) break;
        int g = 0;
        while (g + 1 < a.ng && (int64_t)tl >= a.g[g + 1].tile0) ++g;
        const GroupDev& gr = a.g[g];
        const int64_t base = ((int64_t)tl - gr.tile0) * tile_pts;
        for (int64_t i = base + lane; i - lane < min(base + tile_pts, gr.n); i += 32) {  // warp-uniform
            const bool active = i < gr.n;
            const double x = active ? __ldcs(gr.x + i) : 0.0, y = active ? __ldcs(gr.y + i) : 0.0,
                         z = active ? __ldcs(gr.z + i) : 0.0;
            uint64_t X[3];
            const bool ok = active && fixpoint3(x, y, z, X);
            typename C::type e = C::none();
            if (ok)
                e = __ldg(cells + (s_spread[(uint32_t)(X[0] >> 32) >> cell_shift] |
                                   (s_spread[(uint32_t)(X[1] >> 32) >> cell_shift] << 1) |
                                   (s_spread[(uint32_t)(X[2] >> 32) >> cell_shift] << 2)));
            const bool hot = C::hot(e);
            if (hot) {
                const int l = C::level(e);
                const uint32_t s = (1u << l) + 1u;
                uint32_t nd[3];  // the node: the cell index rounded up in the upper half
#pragma unroll
                for (int d = 0; d < 3; ++d) nd[d] = ((uint32_t)(X[d] >> (52 - l)) + 1u) >> 1;
                const float* rp = rec + REC_FLOATS * (size_t)(s_off[l] + nd[0] + s * (nd[1] + s * nd[2]));
                float f[3][2];
                tri_octant<float>(X, l, f);
                float vv[REC_FLOATS];
                ld_nc_v8(rp, vv, normal);
                ld_nc_v8(rp + 8, vv + 8, normal);
                ld_nc_v8(rp + 16, vv + 16, normal);
                float v[8][3];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k][0] = vv[3 * k], v[k][1] = vv[3 * k + 1], v[k][2] = vv[3 * k + 2];
                float o[3];
                tri_sum<float>(f, v, o);
                __stcs(gr.u + i, o[0]);
                __stcs(gr.u + gr.n + i, o[1]);
                __stcs(gr.u + 2 * gr.n + i, o[2]);
                if (gr.host) __stcs(gr.host + i, C::leaf(e));
            } else if (active && !ok) {  // outside the cube: no host, no value
                atomicOr(t.err, (unsigned)OT_DEV_OUTSIDE);
                const float nan = qnan<float>();
                gr.u[i] = nan;
                gr.u[gr.n + i] = nan;
                gr.u[2 * gr.n + i] = nan;
                if (gr.host) gr.host[i] = -1;
            }
            const bool cold = ok && !hot;
            const unsigned m = __ballot_sync(0xffffffffu, cold);
            if (cold) cq[qn + __popc(m & lt)] = ((long long)g << 40) | i;
            qn += __popc(m);
            __syncwarp();
            if (qn >= 32) {
                drain(32);
                __syncwarp();
                qn -= 32;
                if (lane < qn) cq[lane] = cq[32 + lane];
                __syncwarp();
            }
        }
    }
    if (qn > 0) drain(qn);
}

// Ordered copies of a group's positions: the i-th ordered point is point (pairs[i] & mask).
__global__ void __launch_bounds__(256) k_gather_points(const uint64_t* __restrict__ pairs, int64_t n, uint64_t mask,
                                                       const double* __restrict__ x, const double* __restrict__ y,
                                                       const double* __restrict__ z, double* __restrict__ xs,
                                                       double* __restrict__ ys, double* __restrict__ zs) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = (int64_t)(pairs[i] & mask);
        xs[i] = x[j];
        ys[i] = y[j];
        zs[i] = z[j];
    }
}

// Results back to the caller's order.
__global__ void __launch_bounds__(256) k_scatter_results(const uint64_t* __restrict__ pairs, int64_t n, uint64_t mask,
                                                         const float* __restrict__ us, const int32_t* __restrict__ hs,
                                                         float* __restrict__ u, int32_t* __restrict__ host) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = (int64_t)(pairs[i] & mask);
        u[j] = us[i];
        u[n + j] = us[n + i];
        u[2 * n + j] = us[2 * n + i];
        if (host) host[j] = hs[i];
    }
}

unsigned grid_b(int64_t n) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 8));
}

bool wide_cells(const ot_octree* t) { return t->n >= (int64_t)1 << 28; }

// Cells' entries, node list and record buffer of a batch (synchronises the legacy stream; batch
// creation is not stream-ordered work).  Leaves b->n_rec = 0, without an error, when no leaf is hot
// or one of them (the records' grids: up to 1.9 GB at hot level 8) finds no memory: the rows serve then.
ot_status build_hot_records(const ot_octree* t, int hot_l, const NodeGrid& grid, ot_batch* b) {
    const size_t n_node = grid.off[hot_l + 1], seen_bytes = ((n_node + 31) / 32) * 4;
    uint32_t* seen = nullptr;  // the bits, then the count
    auto done = [&](cudaError_t e) {
        if (seen) cudaFree(seen);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            if (b->d_rec) cudaFree(b->d_rec);
            if (b->d_nodes) cudaFree(b->d_nodes);
            b->d_rec = nullptr, b->d_nodes = nullptr;
            return OT_OK;
        }
        return e == cudaSuccess ? OT_OK : cuda_status(e);
    };
    cudaStream_t s = nullptr;
    cudaError_t e;
    TreeView v = tree_view(t);
    uint32_t count = 0;
    if ((e = cudaMalloc(&seen, seen_bytes + 4)) != cudaSuccess) return done(e);
    uint32_t* d_count = seen + seen_bytes / 4;
    for (int pass = 0; pass < 2; ++pass) {  // count, then list
        if ((e = cudaMemsetAsync(seen, 0, seen_bytes + 4, s)) != cudaSuccess) return done(e);
        k_hot_nodes<<<grid_b(t->n), 256, 0, s>>>(v, hot_l, grid, seen, b->d_nodes, d_count);
        count_launch();
        if (pass == 1) break;
        if ((e = cudaMemcpy(&count, d_count, sizeof(count), cudaMemcpyDeviceToHost)) != cudaSuccess) return done(e);
        if (count == 0) return done(cudaSuccess);
        if ((e = cudaMalloc(&b->d_rec, sizeof(float) * REC_FLOATS * n_node)) != cudaSuccess) return done(e);
        if ((e = cudaMalloc(&b->d_nodes, sizeof(uint2) * (size_t)count)) != cudaSuccess) return done(e);
    }
    const bool wide = wide_cells(t);
    const int64_t ncell = (int64_t)1 << (3 * t->lmap_level);
    if ((e = cudaMalloc(&b->d_cells, (size_t)ncell * (wide ? 8 : 4))) != cudaSuccess) return done(e);
    if (wide)
        k_cells<true><<<grid_b(ncell), 256, 0, s>>>(v, hot_l, static_cast<uint2*>(b->d_cells));
    else
        k_cells<false><<<grid_b(ncell), 256, 0, s>>>(v, hot_l, static_cast<uint32_t*>(b->d_cells));
    count_launch();
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) b->n_rec = count;
    return done(e);
}

} // namespace ot

using namespace ot;

extern "C" ot_status ot_batch_create(const ot_octree* t, const ot_group* groups, int n_groups, const float* d_field,
                                     int search, const ot_launch* launch, void* stream, ot_batch** out) {
    if (!t || !groups || !out || !d_field || n_groups < 1 || n_groups > MAX_GROUPS) return OT_ERR_ARG;
    if (search != OT_BINARY && search != OT_LEARNED) return OT_ERR_ARG;
    if (search == OT_LEARNED && !t->has_index) return OT_ERR_NO_INDEX;
    *out = nullptr;
    const int block = (launch && launch->block) ? launch->block : 256;
    const int tile = (launch && launch->tile) ? launch->tile : 4;
    const int order_level = launch ? launch->order_level : 0;
    const int tri_tile = (launch && launch->tri_tile) ? launch->tri_tile : tile;
    const int tri_per_sm = (launch && launch->tri_blocks_per_sm) ? launch->tri_blocks_per_sm : 2;
    const int tri_records = launch ? launch->tri_records : 0;
    if (tri_records < -1 || tri_records > MAXLEVEL) return OT_ERR_ARG;
    if (block < 64 || block > 256 || block % 32 || tile < 1 || tile > 64) return OT_ERR_ARG;
    if (tri_tile < 1 || tri_tile > 64 || tri_per_sm < 1 || (launch && launch->blocks_per_sm < 0)) return OT_ERR_ARG;
    if (order_level < 0 || order_level > MAXLEVEL) return OT_ERR_ARG;
    BatchArgs a{};
    a.ng = n_groups;
    a.pts = 32 * tile;
    // delta-kernel groups first: the longest work is taken first
    std::vector<int> order;
    for (int pass = 0; pass < 2; ++pass)
        for (int g = 0; g < n_groups; ++g)
            if ((groups[g].kernel != OT_TRILINEAR) == (pass == 0)) order.push_back(g);
    int64_t tile0 = 0;
    for (int k = 0; k < n_groups; ++k) {
        const ot_group& gi = groups[order[k]];
        if (gi.kernel != OT_TRILINEAR && gi.kernel != OT_PESKIN4 && gi.kernel != OT_ROMA3) return OT_ERR_ARG;
        if (gi.n < 0 || (gi.n > 0 && (!gi.d_x || !gi.d_y || !gi.d_z || !gi.d_u))) return OT_ERR_ARG;
        if (gi.kernel != OT_TRILINEAR && t->lmax < 1) return OT_ERR_ARG;
        GroupDev& d = a.g[k];
        d = GroupDev{gi.kernel, gi.d_x, gi.d_y, gi.d_z, gi.n, gi.d_u, gi.d_host, tile0};
        tile0 += (gi.n + 32 * (int64_t)tile - 1) / (32 * (int64_t)tile);
    }
    a.ntiles = tile0;
    if (a.ntiles >= (1LL << 32)) return OT_ERR_LIMIT;

    ot_batch* b = new ot_batch();
    b->tree = t;
    b->device = t->device;
    b->context = t->context;
    b->n_groups = n_groups;
    // trilinear groups processed in Morton order of their points' level-order_level cells:
    // per group, the sort workspace and ordered copies of positions and results
    struct Ordered {
        int k;                 // slot in a.g
        GroupDev user;         // the caller's arrays
        uint64_t* pairs;
        double *xs, *ys, *zs;
        float* us;
        int32_t* hs;
    };
    std::vector<Ordered> ordered;
    cudaStream_t cs = nullptr;
    auto fail = [&](cudaError_t e) {
        if (cs) cudaStreamDestroy(cs);
        ot_batch_destroy(b);
        return cuda_status(e);
    };
    cudaError_t e;
    if ((e = cudaMalloc(&b->d_counter, sizeof(unsigned))) != cudaSuccess) return fail(e);
    for (int k = 0; order_level > 0 && k < n_groups; ++k) {
        GroupDev& d = a.g[k];
        if (d.kernel != OT_TRILINEAR || d.n < 64 || !order_fits(d.n, order_level)) continue;
        Ordered o{k, d, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
        // the pieces from `base`, each on 256 bytes; the bytes they take (base null: only that)
        auto carve = [&](char* base) {
            size_t at = 0;
            auto take = [&](size_t sz) {
                char* r = base ? base + at : nullptr;
                at += (sz + 255) & ~(size_t)255;
                return r;
            };
            o.pairs = reinterpret_cast<uint64_t*>(take(order_ws_bytes(d.n)));
            o.xs = reinterpret_cast<double*>(take(sizeof(double) * d.n));
            o.ys = reinterpret_cast<double*>(take(sizeof(double) * d.n));
            o.zs = reinterpret_cast<double*>(take(sizeof(double) * d.n));
            o.us = reinterpret_cast<float*>(take(3 * sizeof(float) * d.n));
            if (d.host) o.hs = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * d.n));
            return at;
        };
        void* p = nullptr;
        if ((e = cudaMalloc(&p, carve(nullptr))) != cudaSuccess) return fail(e);
        b->bufs.push_back(p);
        carve(static_cast<char*>(p));
        d.x = o.xs, d.y = o.ys, d.z = o.zs, d.u = o.us, d.host = o.hs;
        ordered.push_back(o);
    }
    bool has_tri = false;
    for (int k = 0; k < n_groups; ++k) has_tri = has_tri || groups[k].kernel == OT_TRILINEAR;
    if (has_tri && (e = cudaMalloc(&b->d_pyr, pyramid_bytes(t, sizeof(float)))) != cudaSuccess) return fail(e);
    TreeView v = tree_view(t);
    const size_t smem = 0;
    const bool two = launch && launch->blocks_per_sm == 2;
    const bool learned = search == OT_LEARNED;
    // The launches of one replay: without the level-mate table, one kernel over every group;
    // with it, the delta-kernel groups and the trilinear groups as two launches (the trilinear
    // one at its own, higher, occupancy), each over its own tile range and counter.
    struct Launch {
        void* fn;
        BatchArgs args;
        unsigned grid;
        bool records;  // k_tri_rec: three more arguments
        size_t dsmem;  // dynamic shared memory per block
    };
    std::vector<Launch> launches;
    NodeGrid grid{};
    // min_pts: while there are fewer tiles than warps, the tiles are halved down to this many points
    // (11,000 points in tiles of 128 would keep 86 of thousands of warps busy), to a multiple of it: the
    // trilinear kernels take rows of 32 and would read an odd half row's points into the next tile's
    auto add_launch = [&](void* fn, BatchArgs args, int cap, int min_pts, size_t dsmem = 0) -> cudaError_t {
        int per_sm = 0;
        cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, dsmem);
        if (err != cudaSuccess) return err;
        if (cap > 0) per_sm = std::min(per_sm, cap);
        per_sm = std::max(per_sm, 1);
        const int64_t warps = (int64_t)num_sms() * per_sm * (block / 32);
        while (args.ntiles < warps && args.pts / 2 >= min_pts) {
            args.pts = args.pts / 2 / min_pts * min_pts;
            args.ntiles = 0;
            for (int k = 0; k < args.ng; ++k) {
                args.g[k].tile0 = args.ntiles;
                args.ntiles += (args.g[k].n + args.pts - 1) / args.pts;
            }
        }
        launches.push_back(Launch{fn, args, (unsigned)(num_sms() * per_sm), false, dsmem});
        return cudaSuccess;
    };
    // every warp takes one tile number past the last tile before it stops: the 32-bit tile
    // counter must hold ntiles plus one per warp of the launch without wrapping
    auto counter_fits = [&]() {
        for (const Launch& l : launches)
            if ((uint64_t)l.args.ntiles + (uint64_t)l.grid * (uint64_t)(block / 32) >= (1ULL << 32)) return false;
        return true;
    };
    if (!t->d_mates) {
        void* fn = learned ? (two ? (void*)k_batch<true, 2, false> : (void*)k_batch<true, 3, false>)
                           : (two ? (void*)k_batch<false, 2, false> : (void*)k_batch<false, 3, false>);
        if ((e = add_launch(fn, a, launch ? launch->blocks_per_sm : 0, 32)) != cudaSuccess) return fail(e);
    } else {
        BatchArgs part[2] = {};
        for (int k = 0; k < a.ng; ++k) {
            BatchArgs& p = part[a.g[k].kernel == OT_TRILINEAR ? 1 : 0];
            GroupDev d = a.g[k];
            d.tile0 = p.ntiles;
            p.pts = 32 * (a.g[k].kernel == OT_TRILINEAR ? tri_tile : tile);
            p.g[p.ng++] = d;
            p.ntiles += (d.n + p.pts - 1) / p.pts;
        }
        if (part[1].ntiles >= (1LL << 32)) {
            ot_batch_destroy(b);
            return OT_ERR_LIMIT;
        }
        if (part[0].ng > 0) {
            void* fn = learned ? (two ? (void*)k_batch<true, 2, true, K_DELTA> : (void*)k_batch<true, 3, true, K_DELTA>)
                               : (two ? (void*)k_batch<false, 2, true, K_DELTA> : (void*)k_batch<false, 3, true, K_DELTA>);
            if ((e = add_launch(fn, part[0], launch ? launch->blocks_per_sm : 0, 4)) != cudaSuccess) return fail(e);
        }
        if (part[1].ng > 0) {
            // value records of the hot leaves: leaves of level <= min(map level, hot level), where
            // the hot level is the deepest whose leaves would receive at least 4 of the trilinear
            // points if these were spread evenly over the cube (n 8^-l >= 4)
            int64_t n_tri = 0;
            for (int k = 0; k < part[1].ng; ++k) n_tri += part[1].g[k].n;
            int hot_l = 0;
            while (hot_l < MAXLEVEL && (n_tri >> (3 * (hot_l + 1))) >= 4) ++hot_l;
            hot_l = std::min(hot_l, t->lmap_level);
            if (tri_records > 0) hot_l = std::min(hot_l, tri_records);
            if (tri_records >= 0 && t->d_lmap && hot_l >= t->lmin) {
                grid = node_grid(t->lmin, hot_l);
                ot_status st = build_hot_records(t, hot_l, grid, b);
                if (st != OT_OK) {
                    ot_batch_destroy(b);
                    return st;
                }
            }
            const bool rec = b->n_rec > 0;
            const bool wide = wide_cells(t);
            void* fn = rec ? (learned ? (wide ? (void*)k_tri_rec<true, true> : (void*)k_tri_rec<true, false>)
                                      : (wide ? (void*)k_tri_rec<false, true> : (void*)k_tri_rec<false, false>))
                           : (learned ? (void*)k_batch<true, TRI_MINB, true, K_TRI>
                                      : (void*)k_batch<false, TRI_MINB, true, K_TRI>);
            const size_t dsmem = rec ? (sizeof(HostQueue) + 64 * sizeof(long long)) * (size_t)(block / 32) : 0;
            if ((e = add_launch(fn, part[1], tri_per_sm, 32, dsmem)) != cudaSuccess) return fail(e);
            launches.back().records = rec;
        }
    }
    if (!counter_fits()) {
        ot_batch_destroy(b);
        return OT_ERR_LIMIT;
    }
    if (launches.size() > 1) {
        cudaFree(b->d_counter);
        b->d_counter = nullptr;
        if ((e = cudaMalloc(&b->d_counter, sizeof(unsigned) * launches.size())) != cudaSuccess) return fail(e);
    }

    if ((e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking)) != cudaSuccess) return fail(e);
    // the kernels captured below run at every replay: count them once here, as the replay's
    const uint64_t launches0 = g_launches.load();
    if ((e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) return fail(e);
    cudaMemsetAsync(b->d_counter, 0, sizeof(unsigned) * launches.size(), cs);
    bool cap_ok = true;
    std::vector<int> ibs;
    for (Ordered& o : ordered) {
        int ib = 0;
        cap_ok = cap_ok && launch_point_sort(o.user.x, o.user.y, o.user.z, o.user.n, order_level, o.pairs, &ib,
                                             &o.pairs, cs) == OT_OK;
        ibs.push_back(ib);
        k_gather_points<<<grid_b(o.user.n), 256, 0, cs>>>(o.pairs, o.user.n, (1ULL << ib) - 1, o.user.x, o.user.y,
                                                          o.user.z, o.xs, o.ys, o.zs);
        count_launch();
    }
    if (cap_ok && has_tri) cap_ok = launch_pyramid<float>(t, d_field, b->d_pyr, t->d_need_flags, cs) == OT_OK;
    if (cap_ok && b->n_rec > 0) {
        k_hot_records<<<grid_b(b->n_rec), 256, 0, cs>>>(v, b->d_nodes, b->n_rec, d_field, b->d_pyr, b->d_rec);
        count_launch();
    }
    for (size_t i = 0; cap_ok && i < launches.size(); ++i) {
        unsigned* ctr = b->d_counter + i;
        void* args[] = {&v, &launches[i].args, (void*)&d_field, (void*)&b->d_pyr, &ctr, (void*)&b->d_cells,
                        (void*)&b->d_rec, &grid};
        cap_ok = cudaLaunchKernel(launches[i].fn, dim3(launches[i].grid), dim3(block), args, launches[i].dsmem, cs) ==
                 cudaSuccess;
        count_launch();
    }
    for (size_t i = 0; cap_ok && i < ordered.size(); ++i) {
        const Ordered& o = ordered[i];
        k_scatter_results<<<grid_b(o.user.n), 256, 0, cs>>>(o.pairs, o.user.n, (1ULL << ibs[i]) - 1, o.us, o.hs,
                                                            o.user.u, o.user.host);
        count_launch();
    }
    b->kernels = (int)(g_launches.load() - launches0);
    g_launches.fetch_sub((uint64_t)b->kernels);
    if (!cap_ok) {
        cudaGraph_t g = nullptr;
        cudaStreamEndCapture(cs, &g);
        if (g) cudaGraphDestroy(g);
        return fail(cudaErrorUnknown);
    }
    e = cudaStreamEndCapture(cs, &b->graph);
    if (e != cudaSuccess) return fail(e);
    if ((e = cudaGraphInstantiate(&b->exec, b->graph, 0)) != cudaSuccess) return fail(e);
    cudaStreamDestroy(cs);
    *out = b;
    return OT_OK;
}

extern "C" ot_status ot_batch_run(ot_batch* b, void* stream) {
    if (!b || !b->exec) return OT_ERR_ARG;
    cudaError_t e = cudaGraphLaunch(b->exec, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_status(e);
    count_launch((uint64_t)b->kernels);
    return OT_OK;
}

extern "C" ot_status ot_batch_destroy(ot_batch* b) {
    if (!b) return OT_OK;
    if (!context_lives(b->device, b->context)) {
        delete b;
        return OT_OK;
    }
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    if (b->d_counter) cudaFree(b->d_counter);
    if (b->d_pyr) cudaFree(b->d_pyr);
    if (b->d_cells) cudaFree(b->d_cells);
    if (b->d_nodes) cudaFree(b->d_nodes);
    if (b->d_rec) cudaFree(b->d_rec);
    for (void* p : b->bufs) cudaFree(p);
    delete b;
    return OT_OK;
}
