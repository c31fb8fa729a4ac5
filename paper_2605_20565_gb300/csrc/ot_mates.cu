// ot_mates.cu -- the level-mate table: the trilinear level-mate rule (Sec. 2.3.2 reading:
// host cell c of level l, level-mates c + {0, s_d}) resolved once per octree instead of at
// every query.  For leaf h and octant o of its cell (bit d of o: the upper half on axis d, so
// s_d = +1), row 8h + o holds the 8 value slots of the level-mates by position (bit d of the
// corner: the upper of the two cells on axis d), 32 bytes:
//   slot < 2^31: a leaf index -- a leaf of level l, or the coarser leaf covering the level-mate;
//   slot >= 2^31: (slot - 2^31) indexes the array of cell means of a refined level-mate (the
//   dense pyramid for l <= pyr_level, else the node means of level l by first leaf).
// Out-of-cube neighbours take the host's index on that axis, or wrap when the cube is periodic.
// A query then needs its host leaf, one 32-byte row and the 8 values: the values are those the
// per-query search finds, so results are bit-identical either way.
// 256 bytes per leaf; the table depends on the leaves and the periodic setting only.
//
// Built with it, the parent-block table of the delta kernels (Sec. 2.2 stencils on the finest
// level): for every parent block -- a cell of level lmax-1 whose 8 children are leaves of
// level lmax, identified by its first child's index a0 (a0 >> 3 is unique per block) -- row
// a0 >> 3 holds the first child of each of the 27 blocks (b + {-1, 0, 1}^3, entry
// sum (delta_d + 1) 3^d), or -1 for a block outside the cube (wrapped when periodic) or not
// refined to the finest level; 32 entries per row (128 bytes).  A delta stencil's 2-3 blocks
// per axis all lie within one block's neighbourhood, so a marker needs one lookup and one row
// instead of one lookup per block (visit_parents).
#include <algorithm>

#include "ot_internal.h"
#include "ot_points.cuh"

namespace ot {

namespace {

// The level-l cell at dilated (Morton-interleaved) coordinates v, one axis: v + 1 and v - 1 on the
// axis's bits M, wrapping around the cube.
__device__ __forceinline__ uint64_t dil_inc(uint64_t v, uint64_t M) { return ((v | ~M) + (M & (0ULL - M))) & M; }
__device__ __forceinline__ uint64_t dil_dec(uint64_t v, uint64_t M) { return (v - (M & (0ULL - M))) & M; }

// Value slot of the level-l cell with Morton index kk (and its leaf and level): the leaf that covers it,
// or its mean, whose flag is set, when it is refined.
__device__ __forceinline__ uint32_t value_slot(const TreeView& t, uint64_t kk, int l, uint8_t* __restrict__ need,
                                               int& leaf, int& lvl) {
    const uint64_t q = kk << (3 * (MAXLEVEL - l));
    leaf = search_plain(t, q, lvl);
    if (lvl <= l) return (uint32_t)leaf;
    const int Lp = t.pyr_level;
    const long long ri = l <= Lp ? pyr_offset(l) + (long long)kk
                                 : pyr_offset(Lp + 1) + (long long)(l - Lp - 1) * t.n + leaf;
    need[ri] = 1;  // a mean the table reads
    return 0x80000000u | (uint32_t)ri;
}

// A warp takes 32 consecutive leaves.  Most leaves come in families, the 8 children of one cell, all
// leaves: their level-mates are the 4x4x4 cells around (and of) the family, looked up once for the
// 8 of them -- 56 searches instead of 208 -- into shared memory, from which the warp writes the
// family's 2 KB of rows contiguously, and its row of the parent-block table when it is of the finest
// level (the first leaves of the 26 blocks around are those of their cells next to the family).
// The other leaves are done one by one: 26 searches by lanes 0..26, direction sum (delta_d + 1) 3^d.
// Bound by the instructions of the searches before (214 per leaf): 17.3M leaves 4.36 + 0.82 ms (rows,
// blocks), now 1.68 together for 4.7 GB written.
constexpr int MATES_T = 256;
__global__ void __launch_bounds__(MATES_T) k_mates(TreeView t, uint4* __restrict__ out, int* __restrict__ pnbr,
                                                   uint8_t* __restrict__ need) {
    constexpr unsigned FULLM = 0xffffffffu;
    __shared__ uint32_t s_slot[MATES_T / 32][64];
    __shared__ int s_blk[MATES_T / 32][64];
    const int lane = threadIdx.x & 31;
    uint32_t* slot = s_slot[threadIdx.x >> 5];
    int* blk = s_blk[threadIdx.x >> 5];
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // family rows: this lane's octant and z corner in rows of leaves 2 it + (lane >> 4)
    const int ox = (lane >> 1) & 1, oy = (lane >> 2) & 1, oz = (lane >> 3) & 1;
    const int from0 = ((lane >> 4) + ox) + 4 * oy + 16 * (oz + (lane & 1));
    // single rows: the sources of this lane's corners 2 (lane & 3), + 1 of octant lane >> 2
    int src[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int corner = 2 * (lane & 3) + k;
        src[k] = 0;
#pragma unroll
        for (int d = 0, p3 = 1; d < 3; ++d, p3 *= 3) src[k] += (((corner >> d) & 1) + (((lane >> 2) >> d) & 1)) * p3;
    }
    for (int64_t base = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 32; base < t.n;
         base += nwarps * 32) {
        const int64_t i = base + lane;
        uint64_t key = 0;
        int lv = 0, child = 0;
        bool fam = false;
        if (i < t.n) {
            key = ldg_key(t.key + i);
            lv = t.level[i];
            if (lv > 0) {
                child = (int)(key >> (3 * (MAXLEVEL - lv))) & 7;
                const int64_t h = i - child;
                const uint64_t first = key & ~(key_span(lv - 1) - 1);
                // 8 leaves from the parent's anchor to its last child's: the children themselves
                fam = h >= 0 && h + 7 < t.n && ldg_key(t.key + h) == first &&
                      ldg_key(t.key + h + 7) == first + 7 * key_span(lv) && t.level[h] == lv && t.level[h + 7] == lv;
            }
        }
        for (unsigned heads = __ballot_sync(FULLM, fam && child == 0); heads; heads &= heads - 1u) {
            const int from = __ffs(heads) - 1;
            const int64_t leaf0 = base + from;
            const int l = __shfl_sync(FULLM, lv, from);
            const uint64_t kk = __shfl_sync(FULLM, key, from) >> (3 * (MAXLEVEL - l));  // child 0
            const uint64_t M0 = 0x1249249249249249ULL & ((1ULL << (3 * l)) - 1ULL);
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int pos[3] = {lane & 3, (lane >> 2) & 3, (lane >> 4) + 2 * r};  // 1, 2: the family's cells
                uint64_t cell = 0;
                int own = 0;
                bool ours = true, inside = true;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const uint64_t M = M0 << d, b = kk & M;  // child bit 0 on this axis
                    int p = pos[d];
                    uint64_t v = p == 0 ? dil_dec(b, M) : b | ((uint64_t)(p >> 1) << d);
                    if (p == 3) v = dil_inc(v, M);
                    if (!t.periodic && ((p == 0 && b == 0) || (p == 3 && v == 0))) {
                        // past a face: the cell before it, on this axis
                        inside = false;
                        p = p == 0 ? 1 : 2;
                        v = b | ((uint64_t)(p >> 1) << d);
                    }
                    ours = ours && (p == 1 || p == 2);
                    own |= (p >> 1) << d;
                    cell |= v;
                }
                int leaf = (int)leaf0 + own, lvl = l;
                uint32_t sl = (uint32_t)leaf;
                if (!ours) sl = value_slot(t, cell, l, need, leaf, lvl);
                slot[lane + 32 * r] = sl;
                blk[lane + 32 * r] = inside && lvl == l ? leaf : -1;
            }
            __syncwarp();
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const uint32_t* sp = slot + from0 + 4 * (it & 1) + 16 * (it >> 1);
                out[16 * leaf0 + 32 * it + lane] = make_uint4(sp[0], sp[1], sp[4], sp[5]);
            }
            if (l == t.lmax && pnbr) {
                int v = -1;
                if (lane < 27) {
                    int at = 0, ch = 0;
#pragma unroll
                    for (int d = 0, p3 = 1; d < 3; ++d, p3 *= 3) {
                        const int dir = (lane / p3) % 3;  // 0: the block below, whose upper cells touch the family
                        at += (dir == 0 ? 0 : dir == 1 ? 1 : 3) << (2 * d);
                        ch |= (dir == 0 ? 1 : 0) << d;
                    }
                    v = blk[at];
                    if (v >= 0) v -= ch;
                }
                pnbr[32 * (leaf0 >> 3) + lane] = v;
            }
        }
        for (unsigned rest = __ballot_sync(FULLM, i < t.n && !fam); rest; rest &= rest - 1u) {
            const int from = __ffs(rest) - 1;
            const int64_t leaf0 = base + from;
            const int l = __shfl_sync(FULLM, lv, from);
            const uint64_t kk = __shfl_sync(FULLM, key, from) >> (3 * (MAXLEVEL - l));
            const uint64_t M0 = 0x1249249249249249ULL & ((1ULL << (3 * l)) - 1ULL);
            uint32_t sl = (uint32_t)leaf0;
            if (lane < 27) {
                uint64_t cell = 0;
#pragma unroll
                for (int d = 0, p3 = 1; d < 3; ++d, p3 *= 3) {
                    const int dir = (lane / p3) % 3;
                    const uint64_t M = M0 << d, b = kk & M;
                    uint64_t v = dir == 0 ? dil_dec(b, M) : dir == 2 ? dil_inc(b, M) : b;
                    if (!t.periodic && ((dir == 0 && b == 0) || (dir == 2 && v == 0))) v = b;
                    cell |= v;
                }
                int leaf, lvl;
                if (cell != kk) sl = value_slot(t, cell, l, need, leaf, lvl);
            }
            const uint32_t p0 = __shfl_sync(FULLM, sl, src[0]), p1 = __shfl_sync(FULLM, sl, src[1]);
            reinterpret_cast<uint2*>(out)[32 * leaf0 + lane] = make_uint2(p0, p1);
        }
    }
}

} // namespace

size_t pnbr_slots(const ot_octree* t) { return t->lmax >= 1 ? (size_t)(t->n / 8 + 1) : 0; }

// level-mate table, then the parent-block table
size_t mates_bytes(const ot_octree* t) { return (size_t)256 * (size_t)t->n + 128 * pnbr_slots(t); }

// Every slot must fit in 31 bits.
bool mates_fit(const ot_octree* t) {
    const int64_t means = pyramid_offset(t->pyr_level + 1) + (int64_t)node_levels(t) * t->n;
    return means < ((int64_t)1 << 31) && t->n < ((int64_t)1 << 31);
}

// Frees the flags (pool memory, whose release does not wait for work that may still read it).
void drop_need_flags(ot_octree* t) {
    if (!t->d_need_flags) return;
    if (wait_device(t->device)) cudaFree(t->d_need_flags);
    t->d_need_flags = nullptr;
}

// Fills the octree's table (t->d_mates, mates_bytes(t) bytes) on stream s.
ot_status build_mates(ot_octree* t, cudaStream_t s) {
    if (!t->d_mates) return OT_ERR_ARG;
    if (!mates_fit(t)) return OT_ERR_LIMIT;
    TreeView v = tree_view(t);
    const int64_t grid = std::min<int64_t>((t->n + MATES_T - 1) / MATES_T,
                                           (int64_t)num_sms() * blocks_per_sm((const void*)k_mates, MATES_T, 0));
    // flags of the cell means the table reads (kept by the octree: later pyramids compute
    // those only)
    const size_t nbytes = std::max<size_t>(need_flag_bytes(t), 1);
    drop_need_flags(t);
    uint8_t* need = nullptr;
    OT_CUDA(pool_malloc((void**)&need, nbytes, s));
    OT_CUDA(cudaMemsetAsync(need, 0, nbytes, s));
    int* pn = pnbr_slots(t) ? reinterpret_cast<int*>(reinterpret_cast<char*>(t->d_mates) + (size_t)256 * t->n) : nullptr;
    k_mates<<<(unsigned)std::max<int64_t>(grid, 1), MATES_T, 0, s>>>(v, reinterpret_cast<uint4*>(t->d_mates), pn, need);
    count_launch();
    OT_CUDA(cudaGetLastError());
    const ot_status st = close_need_flags(t, need, s);
    if (st != OT_OK) {
        cudaFreeAsync(need, s);
        return st;
    }
    t->d_need_flags = need;
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

} // namespace ot

using namespace ot;

namespace {

// Drops the octree's table (freed when the library owns it).
void drop_mates(ot_octree* t) {
    drop_need_flags(t);  // without the table every mean is computed again
    if (t->d_mates && t->mates_owned) cudaFree(t->d_mates);
    t->d_mates = nullptr;
    t->mates_owned = false;
}

} // namespace

extern "C" ot_status ot_octree_build_mates(ot_octree* t, int enable, void* stream) {
    if (!t || (enable != 0 && enable != 1)) return OT_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (!enable) {
        if (t->d_mates) OT_CUDA(cudaStreamSynchronize(s));
        drop_mates(t);
        return OT_OK;
    }
    if (!mates_fit(t)) return OT_ERR_LIMIT;
    if (!t->d_mates) {
        const cudaError_t e = cudaMalloc(&t->d_mates, mates_bytes(t));
        if (e != cudaSuccess) {
            t->d_mates = nullptr;
            return cuda_status(e);
        }
        t->mates_owned = true;
    }
    ot_status st = build_mates(t, s);
    if (st == OT_OK && cudaStreamSynchronize(s) != cudaSuccess) st = OT_ERR_CUDA;
    if (st != OT_OK) drop_mates(t);
    return st;
}

extern "C" ot_status ot_octree_mates_bytes(const ot_octree* t, size_t* bytes) {
    if (!t || !bytes) return OT_ERR_ARG;
    *bytes = mates_bytes(t);
    return OT_OK;
}

extern "C" ot_status ot_octree_build_mates_in(ot_octree* t, void* d_buffer, size_t bytes, void* stream) {
    if (!t || !d_buffer || ((uintptr_t)d_buffer & 15) || bytes < mates_bytes(t)) return OT_ERR_ARG;
    if (!mates_fit(t)) return OT_ERR_LIMIT;
    cudaStream_t s = (cudaStream_t)stream;
    if (t->d_mates) OT_CUDA(cudaStreamSynchronize(s));
    drop_mates(t);
    t->d_mates = static_cast<uint32_t*>(d_buffer);
    ot_status st = build_mates(t, s);
    if (st == OT_OK && cudaStreamSynchronize(s) != cudaSuccess) st = OT_ERR_CUDA;
    if (st != OT_OK) drop_mates(t);
    return st;
}

extern "C" ot_status ot_octree_has_mates(const ot_octree* t, int* has) {
    if (!t || !has) return OT_ERR_ARG;
    *has = t->d_mates != nullptr;
    return OT_OK;
}
