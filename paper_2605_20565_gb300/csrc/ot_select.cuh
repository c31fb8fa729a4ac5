// ot_select.cuh -- order-preserving selection: the items of 0 .. n - 1 that satisfy a predicate are
// counted per tile of 4096, the tile counts scanned by one block, and each selected item handed to
// an emitter with its rank.  The predicate is evaluated twice and nothing is written per item in
// between; with a flag and a scanned position per item (8 bytes written and read, and the scan's
// own passes) the lists of refined cells of 17.3M leaves took 590 us, now 230.
#pragma once

#include "ot_internal.h"

namespace ot {

constexpr int SEL_T = 256, SEL_I = 16, SEL_TILE = SEL_T * SEL_I;

inline int64_t select_tiles(int64_t n) { return (n + SEL_TILE - 1) / SEL_TILE; }

// Warp w of a block owns the tile's items [512 w, 512 w + 512), 32 at a time: (warp, round, lane) order
// is index order.
template <typename Pred>
__global__ void __launch_bounds__(SEL_T) k_select_count(Pred pred, int64_t n, uint32_t* __restrict__ cnt) {
    __shared__ uint32_t s_cnt[SEL_T / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i0 = (int64_t)blockIdx.x * SEL_TILE + warp * (32 * SEL_I) + lane;
    uint32_t c = 0;
#pragma unroll
    for (int r = 0; r < SEL_I; ++r) c += i0 + 32 * r < n && pred(i0 + 32 * r) ? 1u : 0u;
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) s_cnt[warp] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < SEL_T / 32; ++w) t += s_cnt[w];
        cnt[blockIdx.x] = t;
    }
}

template <typename Pred, typename Emit>
__global__ void __launch_bounds__(SEL_T) k_select_emit(Pred pred, Emit emit, int64_t n,
                                                       const uint32_t* __restrict__ offs) {
    __shared__ uint32_t s_cnt[SEL_T / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i0 = (int64_t)blockIdx.x * SEL_TILE + warp * (32 * SEL_I) + lane;
    uint32_t mine = 0;  // bit r: the item of round r is selected
#pragma unroll
    for (int r = 0; r < SEL_I; ++r) mine |= (i0 + 32 * r < n && pred(i0 + 32 * r) ? 1u : 0u) << r;
    const uint32_t total = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(mine));
    if (lane == 0) s_cnt[warp] = total;
    __syncthreads();
    uint32_t at = offs[blockIdx.x];
    for (int w = 0; w < warp; ++w) at += s_cnt[w];
    if (total == 0) return;  // warp-uniform
#pragma unroll
    for (int r = 0; r < SEL_I; ++r) {
        const unsigned m = __ballot_sync(0xffffffffu, (mine >> r) & 1u);
        if ((mine >> r) & 1u) emit(i0 + 32 * r, at + __popc(m & ((1u << lane) - 1u)));
        at += __popc(m);
    }
}

// Tile counts of n items into cnt (select_tiles(n) values, scanned in place) and their total to *total.
template <typename Pred>
ot_status select_count(Pred pred, int64_t n, uint32_t* cnt, uint32_t* total, cudaStream_t s) {
    k_select_count<<<(unsigned)select_tiles(n), SEL_T, 0, s>>>(pred, n, cnt);
    count_launch();
    return scan_row(cnt, (int)select_tiles(n), total, s);
}
template <typename Pred, typename Emit>
ot_status select_emit(Pred pred, Emit emit, int64_t n, const uint32_t* cnt, cudaStream_t s) {
    k_select_emit<<<(unsigned)select_tiles(n), SEL_T, 0, s>>>(pred, emit, n, cnt);
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

} // namespace ot
