// ot_pyramid.cu -- means of the field over refined cells: the value a refined trilinear
// level-mate takes, the volume-weighted mean of the leaves inside it (the coalescence average
// of Sec. 2.1.1), in one load whatever its level.
//   Node means, levels Lc+1 .. lmax-1 (Lc = min(lmax, 7)): one array of N entries per level,
//   indexed by the refined cell's first leaf (the leaf holding its anchor, which the level-mate
//   search finds).  The refined cells of each level are listed once per octree; every
//   recomputation takes each listed cell as the mean of its 8 children, deepest level first, a
//   child being a leaf or a refined cell of the next level whose leaf count (kept in the 4th
//   component, as integer bits) gives the start of the next child.
//   Dense pyramid, levels 0 .. Lc: level Lc holds each cell's mean (the covering leaf's value,
//   or the mean of its 8 children as above); every coarser level the mean of its 8 children.
// Recomputed whenever the field changes (every replay of a batch graph).
#include <algorithm>
#include <vector>

#include "ot_internal.h"
#include "ot_points.cuh"
#include "ot_select.cuh"

namespace ot {

namespace {

// bit-exact integer count in the 4th component
__device__ __forceinline__ float count_bits(int c, float) { return __int_as_float(c); }
__device__ __forceinline__ double count_bits(int c, double) { return __longlong_as_double((long long)c); }
__device__ __forceinline__ int bits_count(float v) { return __float_as_int(v); }
__device__ __forceinline__ int bits_count(double v) { return (int)__double_as_longlong(v); }

// Mean of the 8 children of the refined cell of level l whose first leaf is a, written to p with the
// cell's leaf count.  child: node means of level l + 1 (not read when l + 1 == lmax: every child is a
// leaf, the 8 from a on, loaded together).  Otherwise from child to child by their leaf counts
// (searching the 8 children side by side measured 10% slower: more to read).
template <typename T>
__device__ __forceinline__ void children_mean(const TreeView& t, int l, const T* __restrict__ field,
                                              const T* __restrict__ child, int a, T* __restrict__ p) {
    using V = Vec4<T>;
    T s0 = T(0), s1 = T(0), s2 = T(0);
    int pos = a;
    if (l + 1 == t.lmax) {
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
            const auto f = V::load(field, a + ch);
            s0 += f.x;
            s1 += f.y;
            s2 += f.z;
        }
        pos += 8;
    } else {
        for (int ch = 0; ch < 8; ++ch) {
            typename V::type f;
            int step = 1;
            if ((int)t.level[pos] == l + 1) {
                f = V::load(field, pos);
            } else {
                f = V::load(child, pos);
                step = bits_count(f.w);
            }
            s0 += f.x;
            s1 += f.y;
            s2 += f.z;
            pos += step;
        }
    }
    p[0] = s0 * T(0.125), p[1] = s1 * T(0.125), p[2] = s2 * T(0.125), p[3] = count_bits(pos - a, T(0));
}

// Level Lc of the pyramid: the covering leaf's value, or the mean of the 8 children.
template <typename T>
__device__ __forceinline__ void base_mean(const TreeView& t, int Lc, const T* __restrict__ field,
                                          const T* __restrict__ child, int64_t c, T* __restrict__ out) {
    using V = Vec4<T>;
    const uint64_t anchor = (uint64_t)c * key_span(Lc);
    int lv;
    const int a = search_plain(t, anchor, lv);
    T* p = out + 4 * c;
    if (lv <= Lc) {
        const auto f = V::load(field, a);
        p[0] = f.x, p[1] = f.y, p[2] = f.z, p[3] = T(0);
    } else {
        children_mean<T>(t, Lc, field, child, a, p);
    }
}

// need (nullable): only the cells flagged there
template <typename T>
__global__ void __launch_bounds__(256) k_pyr_base(TreeView t, int Lc, const T* __restrict__ field,
                                                  const T* __restrict__ child, T* __restrict__ out,
                                                  const uint8_t* __restrict__ need) {
    const int64_t ncell = (int64_t)1 << (3 * Lc);
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x)
        if (!need || need[c]) base_mean<T>(t, Lc, field, child, c, out);
}

// Refined cells of level l listed in nodes[0, cnt): their means, at index first leaf (need,
// nullable: only the cells flagged there, by first leaf).
template <typename T>
__global__ void __launch_bounds__(256) k_node_means(TreeView t, const int* __restrict__ nodes, int64_t cnt, int l,
                                                    const T* __restrict__ field, const T* __restrict__ child,
                                                    T* __restrict__ out, const uint8_t* __restrict__ need) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x) {
        const int a = nodes[i];
        if (!need || need[a]) children_mean<T>(t, l, field, child, a, out + 4 * (int64_t)a);
    }
}

template <typename T>
__device__ __forceinline__ void up_mean(const T* __restrict__ fine, T* __restrict__ coarse, int64_t c) {
    using V = Vec4<T>;
    T s0 = T(0), s1 = T(0), s2 = T(0);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const auto f = V::load(fine, 8 * c + k);
        s0 += f.x;
        s1 += f.y;
        s2 += f.z;
    }
    T* p = coarse + 4 * c;
    p[0] = s0 * T(0.125), p[1] = s1 * T(0.125), p[2] = s2 * T(0.125), p[3] = T(0);
}

template <typename T>
__global__ void __launch_bounds__(256) k_pyr_up(const T* __restrict__ fine, T* __restrict__ coarse, int64_t ncell,
                                                const uint8_t* __restrict__ need) {
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x)
        if (!need || need[c]) up_mean<T>(fine, coarse, c);
}

// The levels from TOP_LEVEL (512 cells) up in one block and one launch: they take less than a launch each.
constexpr int TOP_LEVEL = 3;
template <typename T>
__global__ void __launch_bounds__(1024) k_pyr_top(T* pyr, int top, const uint8_t* __restrict__ need) {
    for (int l = top; l >= 0; --l) {
        const long long o = pyr_offset(l), fine = pyr_offset(l + 1);
        for (int c = threadIdx.x; c < 1 << (3 * l); c += blockDim.x) {
            if (need && !need[o + c]) continue;
            // (plain loads: the level below was written by this block)
            const T* f = pyr + 4 * (fine + 8 * (long long)c);
            T s[3] = {T(0), T(0), T(0)};
#pragma unroll
            for (int k = 0; k < 8; ++k)
#pragma unroll
                for (int d = 0; d < 3; ++d) s[d] += f[4 * k + d];
            T* p = pyr + 4 * (o + c);
            p[0] = s[0] * T(0.125), p[1] = s[1] * T(0.125), p[2] = s[2] * T(0.125), p[3] = T(0);
        }
        __syncthreads();
    }
}

// ---- the cell means the level-mate table reads, closed under "a mean needs its children's" ----

// needed dense cell c of level l -> its 8 children of level l + 1
__global__ void k_close_dense(const uint8_t* __restrict__ need, int64_t ncell, uint8_t* __restrict__ child_need) {
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x)
        if (need[c])
#pragma unroll
            for (int k = 0; k < 8; ++k) child_need[8 * c + k] = 1;
}

// The refined children of the refined cell of level l with the given anchor key, flagged by their
// first leaves (a search per child).
__device__ __forceinline__ void mark_refined_children(const TreeView& t, uint64_t anchor, int l,
                                                      uint8_t* __restrict__ child_need) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        int lv;
        const int f = search_plain(t, anchor + (uint64_t)k * key_span(l + 1), lv);
        if (lv > l + 1) child_need[f] = 1;
    }
}

// needed base cells (level Lc) that are refined -> their refined children (node level 0)
__global__ void k_close_base(TreeView t, const uint8_t* __restrict__ need, int Lc, uint8_t* __restrict__ child_need) {
    const int64_t ncell = (int64_t)1 << (3 * Lc);
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x) {
        if (!need[c]) continue;
        const uint64_t anchor = (uint64_t)c * key_span(Lc);
        int lv;
        search_plain(t, anchor, lv);
        if (lv > Lc) mark_refined_children(t, anchor, Lc, child_need);
    }
}

// needed refined cells of level l (by first leaf) -> their refined children (level l + 1)
__global__ void k_close_node(TreeView t, const uint8_t* __restrict__ need, int l, uint8_t* __restrict__ child_need) {
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < t.n; a += (int64_t)gridDim.x * blockDim.x)
        if (need[a]) mark_refined_children(t, t.key[a] & ~(key_span(l) - 1), l, child_need);
}

// The leaves that start a refined cell of level l: level > l and key aligned to level l.
struct StartsCell {
    const uint64_t* key;
    const uint8_t* level;
    int l;
    __device__ bool operator()(int64_t i) const {
        return (int)__ldg(level + i) > l && (ldg_key(key + i) & (key_span(l) - 1)) == 0;
    }
};
struct ListLeaf {
    int* out;
    __device__ void operator()(int64_t i, uint32_t at) const { out[at] = (int)i; }
};

unsigned grid_n(int64_t n, int b) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + b - 1) / b, (int64_t)num_sms() * 16));
}

} // namespace

int64_t pyramid_offset(int l) { return ((int64_t)1 << (3 * l)) / 7; }  // sum_{k<l} 8^k = (8^l - 1)/7

int node_levels(const ot_octree* t) { return std::max(0, t->lmax - 1 - t->pyr_level); }

size_t pyramid_bytes(const ot_octree* t, size_t elem) {
    return elem * 4 * ((size_t)pyramid_offset(t->pyr_level + 1) + (size_t)node_levels(t) * (size_t)t->n) + 256;
}

// Lists, once per octree, the refined cells of every node level (by first leaf, in key order).
ot_status build_node_lists(ot_octree* t, cudaStream_t s) {
    const int nl = node_levels(t);
    if (t->d_nodes) cudaFree(t->d_nodes);
    t->d_nodes = nullptr;
    if (nl == 0 || t->n == 0) return OT_OK;
    // counts of all levels first, then one allocation
    const int64_t nt = select_tiles(t->n);
    uint32_t* cnt = nullptr;
    OT_CUDA(pool_malloc((void**)&cnt, sizeof(uint32_t) * (size_t)(nl * (nt + 1)), s));
    uint32_t* tot = cnt + nl * nt;
    ot_status st = OT_OK;
    for (int k = 0; k < nl && st == OT_OK; ++k)
        st = select_count(StartsCell{t->d_key, t->d_level, t->pyr_level + 1 + k}, t->n, cnt + k * nt, tot + k, s);
    std::vector<uint32_t> h(nl);
    if (st == OT_OK) {
        OT_CUDA(cudaMemcpyAsync(h.data(), tot, sizeof(uint32_t) * nl, cudaMemcpyDeviceToHost, s));
        OT_CUDA(cudaStreamSynchronize(s));
        int64_t total = 0;
        for (int k = 0; k < nl; ++k) {
            t->node_off[k] = total;
            t->node_cnt[k] = h[k];
            total += h[k];
        }
        OT_CUDA(pool_malloc((void**)&t->d_nodes, sizeof(int) * std::max<int64_t>(total, 1), s));
    }
    for (int k = 0; k < nl && st == OT_OK; ++k)
        st = select_emit(StartsCell{t->d_key, t->d_level, t->pyr_level + 1 + k}, ListLeaf{t->d_nodes + t->node_off[k]},
                         t->n, cnt + k * nt, s);
    cudaFreeAsync(cnt, s);
    if (st != OT_OK) return st;
    OT_CUDA(cudaStreamSynchronize(s));
    return OT_OK;
}

size_t need_flag_bytes(const ot_octree* t) {
    return (size_t)pyramid_offset(t->pyr_level + 1) + (size_t)node_levels(t) * (size_t)t->n;
}

// Closes the flags of the means the level-mate table reads (need: one byte per entry of the
// means array, dense pyramid then node levels, set by the table builder) under "a mean needs
// its children's"; the octree keeps them, and every later pyramid computes the flagged means
// only.
ot_status close_need_flags(const ot_octree* t, uint8_t* need, cudaStream_t s) {
    const int Lc = t->pyr_level;
    const int nl = node_levels(t);
    const int n = (int)t->n;
    const TreeView v = tree_view(t);
    for (int l = 0; l < Lc; ++l) {
        const int64_t nc = (int64_t)1 << (3 * l);
        k_close_dense<<<grid_n(nc, 256), 256, 0, s>>>(need + pyramid_offset(l), nc, need + pyramid_offset(l + 1));
        count_launch();
    }
    uint8_t* node_need = need + pyramid_offset(Lc + 1);
    if (nl > 0) {
        const int64_t nc = (int64_t)1 << (3 * Lc);
        k_close_base<<<grid_n(nc, 256), 256, 0, s>>>(v, need + pyramid_offset(Lc), Lc, node_need);
        count_launch();
    }
    for (int k = 0; k + 1 < nl; ++k) {
        k_close_node<<<grid_n(n, 256), 256, 0, s>>>(v, node_need + (int64_t)k * n, Lc + 1 + k,
                                                     node_need + (int64_t)(k + 1) * n);
        count_launch();
    }
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

template <typename T>
ot_status launch_pyramid(const ot_octree* t, const T* field, T* pyr, const uint8_t* need, cudaStream_t s) {
    const int Lc = t->pyr_level;
    const int nl = node_levels(t);
    const TreeView v = tree_view(t);
    T* nodes = pyr + 4 * pyramid_offset(Lc + 1);
    // node means, deepest level first (each reads the next level's)
    for (int k = nl - 1; k >= 0; --k) {
        T* out = nodes + 4 * (int64_t)k * t->n;
        const T* child = k + 1 < nl ? out + 4 * (int64_t)t->n : nullptr;
        if (t->node_cnt[k] > 0) {
            const uint8_t* nk = need ? need + pyramid_offset(Lc + 1) + (int64_t)k * t->n : nullptr;
            k_node_means<T><<<grid_n(t->node_cnt[k], 256), 256, 0, s>>>(v, t->d_nodes + t->node_off[k], t->node_cnt[k],
                                                                       Lc + 1 + k, field, child, out, nk);
            count_launch();
        }
    }
    const int64_t ncell = (int64_t)1 << (3 * Lc);
    k_pyr_base<T><<<grid_n(ncell, 256), 256, 0, s>>>(v, Lc, field, nl > 0 ? nodes : nullptr,
                                                    pyr + 4 * pyramid_offset(Lc),
                                                    need ? need + pyramid_offset(Lc) : nullptr);
    count_launch();
    int l = Lc - 1;
    for (; l > TOP_LEVEL; --l) {
        const int64_t nc = (int64_t)1 << (3 * l);
        k_pyr_up<T><<<grid_n(nc, 256), 256, 0, s>>>(pyr + 4 * pyramid_offset(l + 1), pyr + 4 * pyramid_offset(l), nc,
                                                    need ? need + pyramid_offset(l) : nullptr);
        count_launch();
    }
    if (l >= 0) {
        k_pyr_top<T><<<1, 1024, 0, s>>>(pyr, l, need);
        count_launch();
    }
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

template ot_status launch_pyramid<float>(const ot_octree*, const float*, float*, const uint8_t*, cudaStream_t);
template ot_status launch_pyramid<double>(const ot_octree*, const double*, double*, const uint8_t*, cudaStream_t);

} // namespace ot
