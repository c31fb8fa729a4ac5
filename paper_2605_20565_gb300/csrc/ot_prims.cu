// ot_prims.cu -- scan, compaction, unique and a stable LSD radix sort for the octree builder
// and the deterministic spreading.
#include <algorithm>

#include "ot_internal.h"
#include "ot_select.cuh"

namespace ot {

std::atomic<uint64_t> g_launches{0};

ot_status cuda_status(cudaError_t e) {
    if (e == cudaErrorMemoryAllocation) return OT_ERR_OOM;
    return OT_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------
// Exclusive scan (uint32): block-local scans, scan of block totals (recursive), add-back.
// ------------------------------------------------------------------------------------------
constexpr int SCAN_T = 512, SCAN_I = 8, SCAN_TILE = SCAN_T * SCAN_I;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* s_warp, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        uint32_t w = lane < nw ? s_warp[lane] : 0u;
        uint32_t ws = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, ws, o);
            if (lane >= o) ws += y;
        }
        if (lane < nw) s_warp[lane] = ws - w;
        if (lane == nw - 1) s_warp[32] = ws;
    }
    __syncthreads();
    uint32_t r = s_warp[warp] + x - v;
    *total = s_warp[32];
    __syncthreads();
    return r;
}

__global__ void k_scan_tiles(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t n,
                             uint32_t* __restrict__ tile_total) {
    __shared__ uint32_t s_warp[33];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_I;
    uint32_t v[SCAN_I];
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < SCAN_I; ++i) {
        v[i] = (base + i < n) ? in[base + i] : 0u;
        sum += v[i];
    }
    uint32_t tot;
    uint32_t run = block_exclusive_scan(sum, s_warp, &tot);
#pragma unroll
    for (int i = 0; i < SCAN_I; ++i) {
        if (base + i < n) out[base + i] = run;
        run += v[i];
    }
    if (threadIdx.x == 0 && tile_total) tile_total[blockIdx.x] = tot;
}

__global__ void k_scan_add(uint32_t* __restrict__ out, int64_t n, const uint32_t* __restrict__ tile_off) {
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    const uint32_t add = tile_off[blockIdx.x];
    for (int i = threadIdx.x; i < SCAN_TILE; i += blockDim.x)
        if (base + i < n) out[base + i] += add;
}

__global__ void k_total(const uint32_t* in_last, const uint32_t* scan_last, uint32_t* total) {
    *total = *in_last + *scan_last;
}

// Tile totals of every level of the recursive scan of n values.
static int64_t scan_tile_elems(int64_t n) {
    int64_t total = 0;
    for (int64_t m = n; m > SCAN_TILE; m = (m + SCAN_TILE - 1) / SCAN_TILE) total += (m + SCAN_TILE - 1) / SCAN_TILE;
    return total;
}

static size_t scan_ws_bytes(int64_t n) { return (size_t)(scan_tile_elems(n) + 1) * sizeof(uint32_t) + 256; }

// The recursive scan with its tile totals in tmp (scan_tile_elems(n) uint32).
static ot_status scan_levels(const uint32_t* d_in, uint32_t* d_out, int64_t n, uint32_t* tmp, cudaStream_t s) {
    const int64_t nt = (n + SCAN_TILE - 1) / SCAN_TILE;
    if (nt == 1) {
        k_scan_tiles<<<1, SCAN_T, 0, s>>>(d_in, d_out, n, nullptr);
        count_launch();
        return OT_OK;
    }
    k_scan_tiles<<<(unsigned)nt, SCAN_T, 0, s>>>(d_in, d_out, n, tmp);
    count_launch();
    ot_status st = scan_levels(tmp, tmp, nt, tmp + nt, s);
    if (st != OT_OK) return st;
    k_scan_add<<<(unsigned)nt, 256, 0, s>>>(d_out, n, tmp);
    count_launch();
    return OT_OK;
}

static ot_status scan_u32_ws(const uint32_t* d_in, uint32_t* d_out, int64_t n, uint32_t* d_total, void* ws,
                             cudaStream_t s) {
    if (n <= 0) {
        if (d_total) OT_CUDA(cudaMemsetAsync(d_total, 0, sizeof(uint32_t), s));
        return OT_OK;
    }
    // the total needs the last input, which an in-place scan overwrites: keep it first
    uint32_t* last = static_cast<uint32_t*>(ws);
    if (d_total) OT_CUDA(cudaMemcpyAsync(last, d_in + n - 1, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    ot_status st = scan_levels(d_in, d_out, n, last + 1, s);
    if (st != OT_OK) return st;
    if (d_total) {
        k_total<<<1, 1, 0, s>>>(last, d_out + n - 1, d_total);
        count_launch();
    }
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

ot_status scan_u32(const uint32_t* d_in, uint32_t* d_out, int64_t n, uint32_t* d_total, cudaStream_t s) {
    void* ws = nullptr;
    OT_CUDA(pool_malloc((void**)&ws, scan_ws_bytes(n), s));
    ot_status st = scan_u32_ws(d_in, d_out, n, d_total, ws, s);
    cudaFreeAsync(ws, s);
    return st;
}

// ------------------------------------------------------------------------------------------
// Stable LSD radix sort of uint64 keys, digits of up to 8 bits (the bits are split evenly over
// the passes).  A pass is three launches: digit counts per tile, one block per digit scanning
// that digit's row of tile counts, and the scatter.  A tile is RT threads x RI keys; warp w owns
// the tile's keys [w, w + 1) RTILE / RW, 32 at a time, so (warp, round, lane) order is input
// order.
// The scatter is bound by its stores: written straight from the ranking rounds, 256 keys go to
// 256 digits, 8 bytes to a 32-byte sector each, with four block barriers per round.  Instead a
// warp ranks its keys against its own digit counters (no block barrier), the tile is put in
// digit order in shared memory and written out in order: 16 consecutive keys per digit on
// average, 128-byte runs.
// ------------------------------------------------------------------------------------------
constexpr int RT = 256, RI = 16, RTILE = RT * RI, RW = RT / 32;

__global__ void __launch_bounds__(RT) k_radix_hist(const uint64_t* __restrict__ in, int64_t n, int shift,
                                                   uint32_t mask, uint32_t* __restrict__ hist, int ntiles) {
    __shared__ uint32_t cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RTILE;
    if (base + RTILE <= n) {  // a whole tile: every load issued before the first count
        uint32_t d[RI];
#pragma unroll
        for (int r = 0; r < RI; ++r) d[r] = (uint32_t)(__ldg(in + base + r * RT + threadIdx.x) >> shift) & mask;
#pragma unroll
        for (int r = 0; r < RI; ++r) atomicAdd(&cnt[d[r]], 1u);
    } else {
        for (int r = 0; r < RI; ++r) {
            const int64_t i = base + r * RT + threadIdx.x;
            if (i < n) atomicAdd(&cnt[(uint32_t)(in[i] >> shift) & mask], 1u);
        }
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

// Block d: exclusive scan of digit d's row of tile counts in place; its total to totals[d].
constexpr int ROW_T = 512, ROW_I = 4;
__global__ void __launch_bounds__(ROW_T) k_radix_rows(uint32_t* __restrict__ hist, int ntiles,
                                                      uint32_t* __restrict__ totals) {
    __shared__ uint32_t s_warp[33];
    uint32_t* row = hist + (int64_t)blockIdx.x * ntiles;
    uint32_t carry = 0;
    for (int base = 0; base < ntiles; base += ROW_T * ROW_I) {
        const int i0 = base + (int)threadIdx.x * ROW_I;
        uint32_t v[ROW_I], sum = 0;
#pragma unroll
        for (int k = 0; k < ROW_I; ++k) {
            v[k] = i0 + k < ntiles ? row[i0 + k] : 0u;
            sum += v[k];
        }
        uint32_t tot;
        uint32_t run = carry + block_exclusive_scan(sum, s_warp, &tot);
#pragma unroll
        for (int k = 0; k < ROW_I; ++k) {
            if (i0 + k < ntiles) row[i0 + k] = run;
            run += v[k];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

__global__ void __launch_bounds__(RT) k_radix_scatter(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                                      int64_t n, int shift, uint32_t mask,
                                                      const uint32_t* __restrict__ offs, int ntiles,
                                                      const uint32_t* __restrict__ totals) {
    __shared__ uint64_t s_key[RTILE];
    __shared__ uint32_t s_cnt[RW][256];  // per warp: digit counts, then the warp's first place per digit
    // per warp and digit, the lanes of the current round (used before the keys are placed)
    uint32_t (*s_grp)[256] = reinterpret_cast<uint32_t (*)[256]>(s_key);
    __shared__ uint32_t s_base[256];     // digit: its place in out, less its place in the tile
    __shared__ uint32_t s_warp[33];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t base = (int64_t)blockIdx.x * RTILE;
    const int cnt = (int)min((int64_t)RTILE, n - base);
    const int first = warp * (RTILE / RW) + lane;
    uint64_t v[RI];
#pragma unroll
    for (int r = 0; r < RI; ++r) v[r] = first + 32 * r < cnt ? __ldg(in + base + first + 32 * r) : 0ULL;
    const uint32_t toff = offs[(int64_t)tid * ntiles + blockIdx.x], tot = totals[tid];
#pragma unroll
    for (int w = 0; w < RW; ++w) s_cnt[w][tid] = 0, s_grp[w][tid] = 0;
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    uint32_t rank[RI];
#pragma unroll
    for (int r = 0; r < RI; ++r) {
        const bool valid = first + 32 * r < cnt;
        const uint32_t d = (uint32_t)(v[r] >> shift) & mask;
        // the lanes with this lane's digit: all valid ones when the digits agree (coherent
        // input), else gathered by an OR in shared memory
        unsigned grp = __ballot_sync(0xffffffffu, valid);
        const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);  // every lane takes part
        if (__any_sync(0xffffffffu, valid && d != d0)) {      // warp-uniform
            if (valid) atomicOr(&s_grp[warp][d], 1u << lane);
            __syncwarp();
            if (valid) grp = s_grp[warp][d];
        }
        const uint32_t before = __popc(grp & lt);
        uint32_t old = 0;
        if (valid) old = s_cnt[warp][d];
        __syncwarp();
        if (valid && before == 0) s_cnt[warp][d] = old + __popc(grp), s_grp[warp][d] = 0;
        __syncwarp();
        rank[r] = old + before;
    }
    __syncthreads();
    // digit tid: the warps' places within the digit, the digit's place within the tile and in out
    uint32_t run = 0, unused;
#pragma unroll
    for (int w = 0; w < RW; ++w) {
        const uint32_t c = s_cnt[w][tid];
        s_cnt[w][tid] = run;
        run += c;
    }
    const uint32_t start = block_exclusive_scan(run, s_warp, &unused);
    const uint32_t dig = block_exclusive_scan(tot, s_warp, &unused);
#pragma unroll
    for (int w = 0; w < RW; ++w) s_cnt[w][tid] += start;
    s_base[tid] = dig + toff - start;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RI; ++r)
        if (first + 32 * r < cnt) s_key[s_cnt[warp][(uint32_t)(v[r] >> shift) & mask] + rank[r]] = v[r];
    __syncthreads();
    for (int i = tid; i < cnt; i += RT) {
        const uint64_t k = s_key[i];
        out[s_base[(uint32_t)(k >> shift) & mask] + (uint32_t)i] = k;
    }
}

// Tile counts (256 per tile) and the digits' totals.
size_t radix_ws_bytes(int64_t n) {
    const int64_t nt = std::max<int64_t>((n + RTILE - 1) / RTILE, 1);
    return (size_t)(256 * nt + 256) * sizeof(uint32_t) + 256;
}

ot_status radix_sort_u64_ws(uint64_t* d_keys, uint64_t* d_tmp, int64_t n, int bit0, int bit1, void* ws,
                            cudaStream_t s, uint64_t** result) {
    if (result) *result = d_keys;
    if (n <= 1 || bit1 <= bit0) return OT_OK;
    const int nt = (int)((n + RTILE - 1) / RTILE);
    uint32_t* hist = static_cast<uint32_t*>(ws);
    uint32_t* totals = hist + 256 * (int64_t)nt;
    uint64_t* src = d_keys;
    uint64_t* dst = d_tmp;
    for (int sh = bit0, passes = (bit1 - bit0 + 7) / 8; passes > 0; --passes) {
        const int nb = (bit1 - sh + passes - 1) / passes;
        const uint32_t mask = (1u << nb) - 1u;
        k_radix_hist<<<nt, RT, 0, s>>>(src, n, sh, mask, hist, nt);
        k_radix_rows<<<256, ROW_T, 0, s>>>(hist, nt, totals);
        k_radix_scatter<<<nt, RT, 0, s>>>(src, dst, n, sh, mask, hist, nt, totals);
        count_launch(3);
        std::swap(src, dst);
        sh += nb;
    }
    if (result)
        *result = src;  // the caller takes the sorted keys where the last pass left them
    else if (src != d_keys)
        OT_CUDA(cudaMemcpyAsync(d_keys, src, sizeof(uint64_t) * n, cudaMemcpyDeviceToDevice, s));
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

ot_status radix_sort_u64(uint64_t* d_keys, uint64_t* d_tmp, int64_t n, int bit0, int bit1, cudaStream_t s) {
    if (n <= 1 || bit1 <= bit0) return OT_OK;
    void* ws = nullptr;
    OT_CUDA(pool_malloc((void**)&ws, radix_ws_bytes(n), s));
    ot_status st = radix_sort_u64_ws(d_keys, d_tmp, n, bit0, bit1, ws, s);
    cudaFreeAsync(ws, s);
    return st;
}

// ------------------------------------------------------------------------------------------
// Compaction and unique.
// ------------------------------------------------------------------------------------------
namespace {
struct Flagged {
    const uint32_t* flag;
    __device__ bool operator()(int64_t i) const { return __ldg(flag + i) != 0; }
};
struct FirstOfEqual {
    const uint64_t* k;
    __device__ bool operator()(int64_t i) const { return i == 0 || k[i] != k[i - 1]; }
};
struct CopyTo {
    const uint64_t* in;
    uint64_t* out;
    __device__ void operator()(int64_t i, uint32_t at) const { out[at] = in[i]; }
};

template <typename Pred>
ot_status select_u64(Pred pred, const uint64_t* d_in, int64_t n, uint64_t* d_out, int64_t* h_count, cudaStream_t s) {
    uint32_t* cnt = nullptr;
    const int64_t nt = select_tiles(n);
    OT_CUDA(pool_malloc((void**)&cnt, sizeof(uint32_t) * (size_t)(nt + 1), s));
    ot_status st = select_count(pred, n, cnt, cnt + nt, s);
    if (st == OT_OK) st = select_emit(pred, CopyTo{d_in, d_out}, n, cnt, s);
    uint32_t h = 0;
    cudaError_t e = cudaMemcpyAsync(&h, cnt + nt, sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(cnt, s);
    if (st != OT_OK) return st;
    OT_CUDA(e);
    OT_CUDA(cudaStreamSynchronize(s));
    *h_count = h;
    return OT_OK;
}
} // namespace

ot_status scan_row(uint32_t* d_row, int n, uint32_t* d_total, cudaStream_t s) {
    k_radix_rows<<<1, ROW_T, 0, s>>>(d_row, n, d_total);
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

ot_status compact_u64(const uint64_t* d_in, const uint32_t* d_flag, int64_t n, uint64_t* d_out, int64_t* h_count,
                      cudaStream_t s) {
    if (n <= 0) {
        *h_count = 0;
        return OT_OK;
    }
    return select_u64(Flagged{d_flag}, d_in, n, d_out, h_count, s);
}

ot_status unique_u64(const uint64_t* d_keys, int64_t n, uint64_t* d_out, int64_t* h_count, cudaStream_t s) {
    if (n <= 0) {
        *h_count = 0;
        return OT_OK;
    }
    return select_u64(FirstOfEqual{d_keys}, d_keys, n, d_out, h_count, s);
}

} // namespace ot
