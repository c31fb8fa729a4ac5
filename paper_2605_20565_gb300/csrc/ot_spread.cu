// ot_spread.cu -- force spreading, the adjoint of the delta-kernel interpolation (Sec. 2.2):
//   f(cell) += sum_k F_k phi(rx) phi(ry) phi(rz) dV_k / h^3.
// OT_ATOMIC: each marker adds its stencil contributions with float atomics.
// OT_SORTED: the finest level is cut into tiles of 4x4x4 cells.  The markers are sorted (stably)
//   by their home tile, the tile of their stencil's first cell; a stencil reaches at most one
//   tile further per axis, so a tile gathers from the markers of its 8 home tiles T - {0,1}^3,
//   in the order of these and of the markers within, each cell summed in registers and added to
//   f once.  No atomics on f: bit-identical from run to run and for any launch shape.
// Sorting markers instead of one pair per (marker, overlapped 2x2x2 block) leaves 1/16 of the keys
// to sort and one record per marker to write, and a record is read by the 5.4 tiles that its
// stencil overlaps on average instead of by 15.6 blocks.  2M markers of 64 bubbles: spreading
// 1.84 -> 0.65 ms (keys and sort 0.08, records 0.08, tiles 0.49: issue-bound, 58% of the issue slots
// at 17 warps per SM, half of the instructions staging and per-tile set-up).
#include <algorithm>
#include <type_traits>

#include "ot_internal.h"
#include "ot_points.cuh"

namespace ot {

namespace {

template <typename T> __device__ __forceinline__ void add3(T* f, int leaf, T a, T b, T c);
template <> __device__ __forceinline__ void add3<float>(float* f, int leaf, float a, float b, float c) {
    atomicAdd(reinterpret_cast<float4*>(f) + leaf, make_float4(a, b, c, 0.0f));
}
template <> __device__ __forceinline__ void add3<double>(double* f, int leaf, double a, double b, double c) {
    double* p = f + 4 * (size_t)leaf;
    atomicAdd(p, a);
    atomicAdd(p + 1, b);
    atomicAdd(p + 2, c);
}

template <typename T>
__device__ __forceinline__ T marker_volume(const T* __restrict__ dV, int64_t k, int lmax) {
    return dV ? dV[k] * (T)ldexp(1.0, 3 * lmax) : T(1);
}

template <typename T, int K>
__global__ void __launch_bounds__(256) k_spread_atomic(TreeView t, const double* __restrict__ x,
                                                       const double* __restrict__ y, const double* __restrict__ z,
                                                       const T* __restrict__ F, const T* __restrict__ dV, int64_t n,
                                                       T* __restrict__ f) {
    constexpr int W = Stencil<K>::W;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        uint64_t X[3];
        if (!fixpoint3(x[k], y[k], z[k], X)) {
            atomicOr(t.err, (unsigned)OT_DEV_OUTSIDE);
            continue;
        }
        int i0[3];
        T w[3][W];
        stencil_weights<K, T>(t.lmax, X, i0, w);
        const T vol = marker_volume(dV, k, t.lmax);
        const T F0 = F[k] * vol, F1 = F[n + k] * vol, F2 = F[2 * n + k] * vol;
        const bool ok = visit_stencil<K, false>(t, i0, [&](int leaf, int ax, int ay, int az) {
            const T wt = w[0][ax] * w[1][ay] * w[2][az];
            add3<T>(f, leaf, F0 * wt, F1 * wt, F2 * wt);
        });
        if (!ok) atomicOr(t.err, (unsigned)OT_DEV_STENCIL);
    }
}

// ------------------------------------------------------------------------------------------
// Sorted spreading.
// ------------------------------------------------------------------------------------------

// Markers in home-tile order: pairs[i] = (tile key << ib) | marker.  A key of 3 (lmax - 2) bits
// that does not fit beside the marker index (lmax > 14 at most) was sorted in two parts; pairs
// then hold the upper part only and the tile is recomputed from the marker's position.
struct TileOrder {
    const uint64_t* pairs;
    const double *x, *y, *z;
    int64_t n;
    int ib;
    int whole;  // the pairs hold whole keys
    int lmax, periodic;
};

// First stencil cell per axis: in [0, 2^lmax) when periodic, from -2 otherwise.
template <int K>
__device__ __forceinline__ void first_cells(const uint64_t X[3], int lmax, int periodic, int i0[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        i0[d] = Stencil<K>::first((int)fix_cell(X[d], lmax), fix_upper_half(X[d], lmax) ? 1 : 0);
        if (periodic) i0[d] &= (1 << lmax) - 1;
    }
}

// Home tile (Morton key on level lmax - 2) of a marker; a marker outside the cube, which adds
// nothing, goes to tile 0.  Stencils that start outside the cube belong to the tile at the face.
template <int K>
__device__ __forceinline__ uint64_t home_tile(double x, double y, double z, int lmax, int periodic) {
    uint64_t X[3];
    if (!fixpoint3(x, y, z, X)) return 0;
    int i0[3];
    first_cells<K>(X, lmax, periodic, i0);
    return morton3((uint32_t)max(i0[0], 0) >> 2, (uint32_t)max(i0[1], 0) >> 2, (uint32_t)max(i0[2], 0) >> 2);
}

template <int K>
__device__ __forceinline__ uint64_t tile_at(const TileOrder& o, int64_t i) {
    const uint64_t p = __ldg(reinterpret_cast<const unsigned long long*>(o.pairs) + i);
    if (o.whole) return p >> o.ib;
    const int64_t k = (int64_t)(p & ((1ULL << o.ib) - 1));
    return home_tile<K>(o.x[k], o.y[k], o.z[k], o.lmax, o.periodic);
}

// Runs of the markers of one home tile, by tile: open addressing, entry (first << 32) | end (never
// 0: end > first), verified by the tile of its first marker.
struct RunTable {
    unsigned long long* e;
    uint32_t mask;
};
__device__ __forceinline__ uint32_t tile_hash(uint64_t tile) {
    return (uint32_t)((tile * 0x9E3779B97F4A7C15ULL) >> 32);
}

// Keys bits [shift, shift + bits) of the markers in the order of `in` (null: as they are).  Also
// clears the run table and the run count for the passes that follow.
template <int K>
__global__ void __launch_bounds__(256) k_tile_keys(TileOrder o, const uint64_t* in, int shift, int bits,
                                                   uint64_t* out, RunTable rt, uint32_t* __restrict__ n_runs) {
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < o.n; i += step) {
        const int64_t k = in ? (int64_t)(in[i] & ((1ULL << o.ib) - 1)) : i;
        const uint64_t key = home_tile<K>(o.x[k], o.y[k], o.z[k], o.lmax, o.periodic) >> shift;
        out[i] = ((key & ((1ULL << bits) - 1)) << o.ib) | (uint64_t)k;
    }
    for (int64_t i = i0; i <= (int64_t)rt.mask; i += step) rt.e[i] = 0;
    if (i0 == 0) *n_runs = 0;
}

// Up to SMALL_SORT markers: keys and sort in one block and one launch instead of 1 + 3 per digit (a
// launch costs more than a pass over a few thousand keys).  A stable LSD radix sort in shared
// memory, 8-bit digits: warp w ranks its own stretch of the keys against its own counters, as
// the tiles of the radix sort in ot_prims.cu do.
constexpr int SMALL_SORT = 8192, SMALL_T = 512, SMALL_I = SMALL_SORT / SMALL_T;
constexpr size_t SMALL_SMEM = SMALL_SORT * 8 + (SMALL_T / 32) * 256 * 4 * 2;
template <int K>
__global__ void __launch_bounds__(SMALL_T) k_tile_sort_small(TileOrder o, int bits, uint64_t* __restrict__ out,
                                                             RunTable rt, uint32_t* __restrict__ n_runs) {
    constexpr int NW = SMALL_T / 32;
    constexpr unsigned FULLM = 0xffffffffu;
    extern __shared__ uint64_t s_pair[];
    uint32_t (*s_cnt)[256] = reinterpret_cast<uint32_t (*)[256]>(s_pair + SMALL_SORT);  // per warp and digit
    uint32_t (*s_grp)[256] = s_cnt + NW;
    __shared__ uint32_t s_tot[8];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n = (int)o.n;
    const unsigned lt = (1u << lane) - 1u;
    const int rounds = (n + SMALL_T - 1) / SMALL_T;  // keys per thread
    const int first = warp * rounds * 32 + lane;     // the warp's stretch, 32 keys a round
    uint64_t v[SMALL_I];
#pragma unroll
    for (int r = 0; r < SMALL_I; ++r) {
        const int i = first + 32 * r;
        v[r] = r < rounds && i < n
                   ? (home_tile<K>(o.x[i], o.y[i], o.z[i], o.lmax, o.periodic) << o.ib) | (uint64_t)i : 0ULL;
    }
    for (int64_t i = tid; i <= (int64_t)rt.mask; i += SMALL_T) rt.e[i] = 0;
    if (tid == 0) *n_runs = 0;
    for (int sh = o.ib; sh < o.ib + bits; sh += 8) {
        for (int i = tid; i < 2 * NW * 256; i += SMALL_T) s_cnt[0][i] = 0;
        __syncthreads();
        uint32_t rank[SMALL_I];
#pragma unroll
        for (int r = 0; r < SMALL_I; ++r) {
            if (r >= rounds) break;  // block-uniform
            const bool valid = first + 32 * r < n;
            const uint32_t d = (uint32_t)(v[r] >> sh) & 255u;
            if (valid) atomicOr(&s_grp[warp][d], 1u << lane);
            __syncwarp();
            unsigned grp = 0;
            uint32_t old = 0;
            if (valid) grp = s_grp[warp][d], old = s_cnt[warp][d];
            __syncwarp();
            if (valid && !(grp & lt)) s_cnt[warp][d] = old + __popc(grp), s_grp[warp][d] = 0;
            __syncwarp();
            rank[r] = old + __popc(grp & lt);
        }
        __syncthreads();
        // thread d < 256: the warps' places within digit d, then the digit's place
        uint32_t run = 0;
        if (tid < 256) {
            for (int w = 0; w < NW; ++w) {
                const uint32_t c = s_cnt[w][tid];
                s_cnt[w][tid] = run;
                run += c;
            }
            uint32_t x = run;
#pragma unroll
            for (int k = 1; k < 32; k <<= 1) {
                const uint32_t u = __shfl_up_sync(FULLM, x, k);
                if (lane >= k) x += u;
            }
            if (lane == 31) s_tot[warp] = x;
            run = x - run;  // exclusive within the warp
        }
        __syncthreads();
        if (tid < 256) {
            for (int w = 0; w < warp; ++w) run += s_tot[w];
            for (int w = 0; w < NW; ++w) s_cnt[w][tid] += run;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SMALL_I; ++r)
            if (r < rounds && first + 32 * r < n)
                s_pair[s_cnt[warp][(uint32_t)(v[r] >> sh) & 255u] + rank[r]] = v[r];
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SMALL_I; ++r)
            if (r < rounds && first + 32 * r < n) v[r] = s_pair[first + 32 * r];
    }
#pragma unroll
    for (int r = 0; r < SMALL_I; ++r)
        if (r < rounds && first + 32 * r < n) out[first + 32 * r] = v[r];
}

// A marker as the tiles read it: per-axis weights, force times volume, and per axis the first
// stencil cell relative to the home tile, -2 .. 3 (biased by 8, one byte each).
template <typename T>
struct __align__(16) MarkerRec {
    T w[3][4];
    T F[3];
    T off;  // the bytes as the low bits of an integer of T's size
};
__device__ __forceinline__ float bits_to(uint32_t v, float) { return __uint_as_float(v); }
__device__ __forceinline__ double bits_to(uint32_t v, double) { return __longlong_as_double((long long)v); }
__device__ __forceinline__ uint32_t bits_of(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t bits_of(double v) { return (uint32_t)__double_as_longlong(v); }
constexpr uint32_t OFF_NONE = 0x404040u;  // a marker that reaches no tile

// Records in home-tile order (F null: the forces come later), and the runs: a warp takes 32
// consecutive markers, finds the first of each run, its end (for the last one of the warp a 32-ary search over the markers that follow)
// and enters it in the table and the list of runs (whose order does not matter; one atomic
// per block's 256 markers).
constexpr int REC_T = 256;
template <typename T, int K>
__global__ void __launch_bounds__(REC_T) k_tile_records(TileOrder o, const T* __restrict__ F, const T* __restrict__ dV,
                                                        MarkerRec<T>* __restrict__ recs, RunTable rt,
                                                        uint32_t* __restrict__ runs, uint32_t* __restrict__ n_runs,
                                                        unsigned* __restrict__ err) {
    constexpr int W = Stencil<K>::W, NW = REC_T / 32;
    constexpr unsigned FULLM = 0xffffffffu;
    __shared__ uint32_t s_heads[NW], s_slot;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = o.n;
    const int ncell = 1 << o.lmax;
    for (int64_t block0 = blockIdx.x * (int64_t)REC_T; block0 < n; block0 += (int64_t)gridDim.x * REC_T) {
        const int64_t base = block0 + warp * 32, i = base + lane;
        const bool in = i < n;
        uint64_t tile = ~0ULL;
        if (in) {
            tile = tile_at<K>(o, i);
            const int64_t k = (int64_t)(o.pairs[i] & ((1ULL << o.ib) - 1));
            MarkerRec<T> r;
            uint64_t X[3];
            uint32_t off = OFF_NONE;
            if (fixpoint3(o.x[k], o.y[k], o.z[k], X)) {
                int i0[3];
                T w[3][W];
                stencil_weights<K, T>(o.lmax, X, i0, w);
                bool out = false;
                off = 0;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    if (o.periodic) i0[d] &= ncell - 1;
                    out = out || (!o.periodic && (i0[d] < 0 || i0[d] + W > ncell));
                    off |= (uint32_t)(i0[d] - (max(i0[d], 0) & ~3) + 8) << (8 * d);
#pragma unroll
                    for (int a = 0; a < 4; ++a) r.w[d][a] = a < W ? w[d][a] : T(0);
                }
                if (out) atomicOr(err, (unsigned)OT_DEV_STENCIL);
                const T vol = marker_volume(dV, k, o.lmax);
#pragma unroll
                for (int d = 0; d < 3; ++d) r.F[d] = F ? F[d * n + k] * vol : T(0);
            } else {
                atomicOr(err, (unsigned)OT_DEV_OUTSIDE);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    r.F[d] = T(0);
#pragma unroll
                    for (int a = 0; a < 4; ++a) r.w[d][a] = T(0);
                }
            }
            r.off = bits_to(off, T(0));
            recs[i] = r;
        }
        // the runs that start in this warp's markers
        uint64_t prev = __shfl_up_sync(FULLM, tile, 1);
        if (lane == 0 && base > 0 && base < n) prev = tile_at<K>(o, base - 1);
        const bool head = in && (i == 0 || tile != prev);
        const unsigned m = __ballot_sync(FULLM, head);
        if (lane == 0) s_heads[warp] = (uint32_t)__popc(m);
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t c = 0;
            for (int w = 0; w < NW; ++w) c += s_heads[w];
            s_slot = c ? atomicAdd(n_runs, c) : 0u;
        }
        __syncthreads();
        uint32_t slot = s_slot;
        for (int w = 0; w < warp; ++w) slot += s_heads[w];
        if (m) {  // warp-uniform
            // where the last of them ends: lo is in the run, hi past it (or the end of the markers)
            int64_t lo = min(base + 31, n - 1), hi = n;
            const uint64_t last = __shfl_sync(FULLM, tile, 31 - __clz(m));
            for (int64_t step = 1; hi - lo > 1; step = (hi - lo + 31) / 32) {
                const int64_t p = lo + step * (lane + 1);
                const int c = __popc(__ballot_sync(FULLM, p < hi && tile_at<K>(o, min(p, n - 1)) == last));
                if (c < 32) hi = min(hi, lo + step * (c + 1));  // (all 32: only at the first step)
                lo += step * c;
            }
            if (head) {
                const unsigned above = lane < 31 ? m & (FULLM << (lane + 1)) : 0u;
                const int64_t end = above ? base + __ffs(above) - 1 : hi;
                runs[slot + __popc(m & ((1u << lane) - 1u))] = (uint32_t)i;
                const unsigned long long e = ((unsigned long long)i << 32) | (unsigned long long)end;
                uint32_t h = tile_hash(tile) & rt.mask;
                for (uint32_t tries = 0; tries <= rt.mask; ++tries) {  // the table has more places than runs
                    if (atomicCAS(rt.e + h, 0ULL, e) == 0ULL) break;
                    h = (h + 1) & rt.mask;
                }
            }
        }
        __syncthreads();  // s_heads, s_slot
    }
}

// Run of home tile `tile`: (first, end), (0, 0) when no marker has it.
template <int K>
__device__ __forceinline__ uint2 find_run(const TileOrder& o, const RunTable& rt, uint64_t tile) {
    uint32_t h = tile_hash(tile) & rt.mask;
    for (uint32_t tries = 0; tries <= rt.mask; ++tries) {
        const unsigned long long e = __ldg(rt.e + h);
        if (e == 0ULL) break;
        if (tile_at<K>(o, (int64_t)(e >> 32)) == tile) return make_uint2((uint32_t)(e >> 32), (uint32_t)e);
        h = (h + 1) & rt.mask;
    }
    return make_uint2(0u, 0u);
}

// w shifted to the tile's cells: a[c] = w[c - rel] for the cells of the stencil, 0 elsewhere.
template <typename T>
__device__ __forceinline__ void align_weights(const T (&w)[4], int rel, T (&a)[4]) {
    const int s = rel < 0 ? -rel : rel;
    T v[4] = {w[0], w[1], w[2], w[3]}, u[4];
    const bool neg = rel < 0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        u[c] = !(s & 1) ? v[c] : neg ? (c < 3 ? v[(c + 1) & 3] : T(0)) : (c > 0 ? v[(c + 3) & 3] : T(0));
#pragma unroll
    for (int c = 0; c < 4; ++c)
        a[c] = !(s & 2) ? u[c] : neg ? (c < 2 ? u[(c + 2) & 3] : T(0)) : (c > 1 ? u[(c + 2) & 3] : T(0));
}

// What a warp stages of up to 32 markers: the 16 products of the x and y weights at the tile's cells
// (rows padded to 33 so that both the staging lane-per-marker stores and the lane-per-cell loads
// are free of bank conflicts), the z weights in pairs, and the force with the bits of the cells
// that the stencil covers per axis.
template <typename T>
struct __align__(16) TileStage {
    T wxy[16][33];
    T wz[2][33][2];
    T F[32][4];
};
__device__ __forceinline__ void load4(const float* p, float v[4]) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ __forceinline__ void load4(const double* p, double v[4]) {
    const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}
__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store4(double* p, double a, double b, double c, double d) {
    *reinterpret_cast<double2*>(p) = make_double2(a, b);
    *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
}

template <typename T> struct Acc3 {
    T x = T(0), y = T(0), z = T(0);
    __device__ __forceinline__ void add(T w, T a, T b, T c) { x += w * a, y += w * b, z += w * c; }
    __device__ __forceinline__ void add(const Acc3& a) { x += a.x, y += a.y, z += a.z; }
    __device__ __forceinline__ bool zero() const { return x == T(0) && y == T(0) && z == T(0); }
};

// by the exponent bits (no FP64 comparison)
__device__ __forceinline__ bool is_finite(float v) { return (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u; }
__device__ __forceinline__ bool is_finite(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// VEC: f starts on 16 bytes.  It may start at any float, a view into a larger buffer say.
template <bool VEC>
__device__ __forceinline__ void add_leaf(float* f, int leaf, const Acc3<float>& a) {
    float* p = f + 4 * (size_t)leaf;
    if constexpr (VEC) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        *reinterpret_cast<float2*>(p) = make_float2(v.x + a.x, v.y + a.y);
        p[2] = v.z + a.z;
    } else {
        p[0] += a.x, p[1] += a.y, p[2] += a.z;
    }
}
template <bool>
__device__ __forceinline__ void add_leaf(double* f, int leaf, const Acc3<double>& a) {
    double* p = f + 4 * (size_t)leaf;
    p[0] += a.x, p[1] += a.y, p[2] += a.z;
}

// Where a tile's sums go: added to f and, scaled, to u when there is one (multi-direct forcing's
// velocity correction).
template <typename T, bool VEC> struct TileOut {
    T* f;
    T* u;
    T scale;
    __device__ __forceinline__ void add(int leaf, const Acc3<T>& a) const {
        add_leaf<VEC>(f, leaf, a);
        if constexpr (sizeof(T) == 4) {  // (the forcing is FP32)
            if (!u) return;
            Acc3<T> b;
            b.x = scale * a.x, b.y = scale * a.y, b.z = scale * a.z;
            add_leaf<VEC>(u, leaf, b);
        }
    }
};

// A run of home tile H stands for the tiles H + {0,1}^3; each tile is taken by the first of its 8
// home tiles (in the order of their offsets) that has markers.  Its markers are listed run after run
// and summed in segments of SEG list places, each from zero and the segments in order, so that
// the result does not depend on who sums which: one warp per run takes its tiles whole or, when the
// runs are too few to fill the chip, one block per tile deals the segments to its warps.
// Lane: column (x, y) = (lane & 3, lane >> 2 & 3) and the cells z = 2 (lane >> 4), + 1 (in FP64 z = lane
// >> 4, + 2: more than half of the stencils reach only the lower or only the upper two layers of a
// tile, and the products of the other ones, which the FP64 pipe bounds, are left out: 1M 3-point markers
// at 8 to a cell 2,737 -> 2,165 us, Peskin-4 4,058 -> 3,307 us), whose sums it keeps in registers; a marker is staged by one lane and costs the warp 3 shared loads, 2
// products and 6 fused multiply-adds.  A cell whose sums are all zero is left as it is.
// The line of 4096 runs, some 5 blocks of 4 warps on each of 152 SMs, FP32 spreading by warps per run and
// by blocks per tile: 500,000 markers in 750, 3,000, 5,800 and 11,700 runs 670/295, 298/282, 259/334
// and 237/468 us; 100,000 in 740, 2,900 and 5,500 runs 194/130, 125/179 and 125/256 us.  With few
// markers per run the warps are ahead earlier (10,000 in 2,400 runs 85/139 us): the number of
// markers is not in the rule.
constexpr int TILE_T = 128, SEG = 64;
constexpr int64_t WIDE_RUNS = 4096;
template <typename T, int K, bool VEC>
__global__ void __launch_bounds__(TILE_T) k_tile_reduce(TreeView t, TileOrder o, RunTable rt,
                                                        const uint32_t* __restrict__ runs,
                                                        const uint32_t* __restrict__ n_runs,
                                                        const MarkerRec<T>* __restrict__ recs, TileOut<T, VEC> out) {
    constexpr int W = Stencil<K>::W, NW = TILE_T / 32;
    constexpr bool HALVES = sizeof(T) == 8;  // a lane's cells are 2 apart, one in each half of the tile
    constexpr unsigned FULLM = 0xffffffffu;
    __shared__ TileStage<T> s_stage[NW];
    __shared__ T s_part[NW][6][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    TileStage<T>& sg = s_stage[warp];
    const unsigned lt = (1u << lane) - 1u;
    const int64_t nr = *n_runs;
    const bool wide = nr <= WIDE_RUNS;  // a task is a tile and a block's, else a run and a warp's
    const int64_t ntask = wide ? nr * 8 : nr;
    const int64_t task0 = wide ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * NW + warp;
    const int64_t step = wide ? (int64_t)gridDim.x : (int64_t)gridDim.x * NW;
    const int nt = 1 << (t.lmax - 2);  // tiles per axis
    const int shb = MAXLEVEL - (t.lmax - 1);
    const int cx = lane & 3, cy = (lane >> 2) & 3, zh = lane >> 4;
    const uint32_t cells = (1u << cx) | (1u << (4 + cy));
    bool missing = false;
    for (int64_t task = task0; task < ntask; task += step) {
        uint32_t h[3];
        // (wide tasks by tile offset: those of offset 0 are all taken here, the later ones seldom)
        const int own8 = wide ? (int)(task / nr) : 0;
        demorton3(tile_at<K>(o, runs[wide ? task - own8 * nr : task]), h[0], h[1], h[2]);
        // lane < 27: the run of home tile H + {-1, 0, 1}^3
        uint2 run = make_uint2(0u, 0u);
        if (lane < 27) {
            int q[3] = {(int)h[0] + lane % 3 - 1, (int)h[1] + (lane / 3) % 3 - 1, (int)h[2] + lane / 9 - 1};
            bool inside = true;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (t.periodic) q[d] &= nt - 1;
                inside = inside && q[d] >= 0 && q[d] < nt;
            }
            if (inside) run = find_run<K>(o, rt, morton3((uint32_t)q[0], (uint32_t)q[1], (uint32_t)q[2]));
        }
        const unsigned have = __ballot_sync(FULLM, run.y > run.x);
        // lane d < 8: whether tile T = H + d is this task's -- inside, and no home tile T - s with s < d
        // has markers (T - s is neighbour 13 + at(d) - at(s) of H, at(v) = v_x + 3 v_y + 9 v_z)
        const int s = lane & 7;
        const int at_s = (s & 1) + 3 * ((s >> 1) & 1) + 9 * (s >> 2);
        bool mine = !wide || s == own8;
#pragma unroll
        for (int k = 0; k < 3; ++k) mine = mine && (t.periodic || (int)h[k] + ((s >> k) & 1) < nt);
#pragma unroll
        for (int k = 0; k < 7; ++k)
            mine = mine && !(k < s && ((have >> (13 + at_s - ((k & 1) + 3 * ((k >> 1) & 1) + 9 * (k >> 2)))) & 1u));
        for (unsigned todo = __ballot_sync(FULLM, mine) & 0xffu; todo; todo &= todo - 1u) {  // uniform in the task
            const int d8 = __ffs(todo) - 1;
            int tc[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                tc[k] = (int)h[k] + ((d8 >> k) & 1);
                if (t.periodic) tc[k] &= nt - 1;
            }
            // lane s < 8: home tile T - s
            const int from = 13 + (d8 & 1) + 3 * ((d8 >> 1) & 1) + 9 * (d8 >> 2) - at_s;
            const uint32_t st = __shfl_sync(FULLM, run.x, from), en = __shfl_sync(FULLM, run.y, from);
            uint32_t incl = en - st;  // lanes 0..7 (repeated above): scan of the run lengths
#pragma unroll
            for (int k = 1; k < 8; k <<= 1) {
                const uint32_t v = __shfl_up_sync(FULLM, incl, k);
                if (s >= k) incl += v;
            }
            const uint32_t total = __shfl_sync(FULLM, incl, 7);
            const uint32_t first = st - (incl - (en - st));  // record of list place p: first + p
            // the tile's 8 blocks of 8 finest leaves: first leaf, -1 when not refined to the finest
            const int a0 = find_block<false>(t, morton3((uint32_t)(2 * tc[0] + (s & 1)) << shb,
                                                        (uint32_t)(2 * tc[1] + ((s >> 1) & 1)) << shb,
                                                        (uint32_t)(2 * tc[2] + (s >> 2)) << shb));
            const unsigned valid = __ballot_sync(FULLM, a0 >= 0) & 0xffu;
            // this lane's two cells: leaf and the one above it in its block, or (HALVES) leaf and leaf1 of the
            // blocks above one another
            const int mine0 = __shfl_sync(FULLM, a0, (cx >> 1) | ((cy >> 1) << 1) | (HALVES ? 0 : zh << 2));
            const int leaf = mine0 + ((cx & 1) | ((cy & 1) << 1) | (HALVES ? zh << 2 : 0));
            int mine1 = -1, leaf1 = 0;
            if constexpr (HALVES) {
                mine1 = __shfl_sync(FULLM, a0, (cx >> 1) | ((cy >> 1) << 1) | 4);
                leaf1 = mine1 + (leaf - mine0);
                if (mine0 >= 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(out.f + 4 * (size_t)leaf));
                if (mine1 >= 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(out.f + 4 * (size_t)leaf1));
            } else if (mine0 >= 0) {
                asm volatile("prefetch.global.L2 [%0];" ::"l"(out.f + 4 * (size_t)leaf));
                asm volatile("prefetch.global.L2 [%0];" ::"l"(out.f + 4 * (size_t)(leaf + 4)));
            }
            // adds up to 32 list places from base to acc
            auto add32 = [&](uint32_t base, Acc3<T>(&acc)[2]) {
                const uint32_t p = base + lane;
                int src = 0;
#pragma unroll
                for (int k = 0; k < 7; ++k) src += p >= __shfl_sync(FULLM, incl, k) ? 1 : 0;
                const uint32_t rf = __shfl_sync(FULLM, first, src);
                MarkerRec<T> r;
                int rel[3] = {64, 64, 64};
                if (p < total) {
                    r = recs[rf + p];
                    const uint32_t off = bits_of(r.off);
#pragma unroll
                    for (int k = 0; k < 3; ++k) rel[k] = (int)((off >> (8 * k)) & 0xffu) - 8 - 4 * ((src >> k) & 1);
                }
                bool over = true;  // the stencil overlaps the tile
#pragma unroll
                for (int k = 0; k < 3; ++k) over = over && rel[k] > -W && rel[k] < 4;
                if (valid != 0xffu) {  // does it overlap a block that is not there?
                    unsigned blocks = over ? 0xffu : 0u;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const unsigned upper = k == 0 ? 0xAAu : k == 1 ? 0xCCu : 0xF0u;
                        blocks &= (rel[k] <= 1 && rel[k] + W > 0 ? ~upper : 0u) |
                                  (rel[k] <= 3 && rel[k] + W > 2 ? upper : 0u);
                    }
                    missing = missing || (blocks & ~valid & 0xffu);
                }
                const unsigned m = __ballot_sync(FULLM, over);
                const int cnt = __popc(m), at = __popc(m & lt);
                bool odd = false;  // a force that is not finite: 0 F is no longer 0
                if (over) {
                    T ax[4], ay[4], az[4];
                    align_weights<T>(r.w[0], rel[0], ax);
                    align_weights<T>(r.w[1], rel[1], ay);
                    align_weights<T>(r.w[2], rel[2], az);
#pragma unroll
                    for (int c = 0; c < 16; ++c) sg.wxy[c][at] = ax[c & 3] * ay[c >> 2];
#pragma unroll
                    for (int c = 0; c < 4; ++c) sg.wz[c >> 1][at][c & 1] = az[c];
                    store4(sg.F[at], r.F[0], r.F[1], r.F[2], T(0));
                    odd = !(is_finite(r.F[0]) && is_finite(r.F[1]) && is_finite(r.F[2]));
                }
                const bool slow = __any_sync(FULLM, odd);
                if (slow && over) {  // the cells that the stencil covers, 4 bits per axis
                    uint32_t cover = 0;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const uint32_t b = rel[k] >= 0 ? ((1u << W) - 1u) << rel[k] : ((1u << W) - 1u) >> -rel[k];
                        cover |= (b & 0xfu) << (4 * k);
                    }
                    sg.F[at][3] = bits_to(cover, T(0));
                }
                __syncwarp();
                if (!slow) {
                    if constexpr (HALVES) {
                        // (a loop per half: a product that is only predicated off takes the pipe all the same)
                        const unsigned reach[2] = {__ballot_sync(FULLM, over && rel[2] <= 1),
                                                   __ballot_sync(FULLM, over && rel[2] + W > 2)};
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
#pragma unroll 2
                            for (unsigned todo = reach[e]; todo; todo &= todo - 1u) {
                                const int j = __popc(m & ((todo & (0u - todo)) - 1u));  // its place in the stage
                                T Fj[4];
                                load4(sg.F[j], Fj);
                                acc[e].add(sg.wxy[lane & 15][j] * sg.wz[e][j][zh], Fj[0], Fj[1], Fj[2]);
                            }
                        }
                    } else {
#pragma unroll 4
                        for (int j = 0; j < cnt; ++j) {
                            const T xy = sg.wxy[lane & 15][j];
                            T Fj[4];
                            load4(sg.F[j], Fj);
                            acc[0].add(xy * sg.wz[zh][j][0], Fj[0], Fj[1], Fj[2]);
                            acc[1].add(xy * sg.wz[zh][j][1], Fj[0], Fj[1], Fj[2]);
                        }
                    }
                } else {  // the stencil's own cells only
                    for (int j = 0; j < cnt; ++j) {
                        const uint32_t cover = bits_of(sg.F[j][3]);
                        if ((cover & cells) != cells) continue;
#pragma unroll
                        for (int e = 0; e < 2; ++e)
                            if ((cover >> (8 + (HALVES ? zh + 2 * e : 2 * zh + e))) & 1u)
                                acc[e].add(sg.wxy[lane & 15][j] * (HALVES ? sg.wz[e][j][zh] : sg.wz[zh][j][e]),
                                           sg.F[j][0], sg.F[j][1], sg.F[j][2]);
                    }
                }
                __syncwarp();
            };
            Acc3<T> sum[2];
            if (!wide) {
                for (uint32_t base = 0; base < total; base += SEG) {
                    Acc3<T> acc[2];
                    for (uint32_t b = base; b < base + SEG && b < total; b += 32) add32(b, acc);
                    sum[0].add(acc[0]), sum[1].add(acc[1]);
                }
            } else {
                for (uint32_t base = 0; base < total; base += NW * SEG) {
                    const uint32_t own = base + warp * SEG;
                    Acc3<T> acc[2];
                    for (uint32_t b = own; b < own + SEG && b < total; b += 32) add32(b, acc);
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        s_part[warp][3 * e][lane] = acc[e].x, s_part[warp][3 * e + 1][lane] = acc[e].y,
                        s_part[warp][3 * e + 2][lane] = acc[e].z;
                    __syncthreads();
                    for (int w = 0; w < NW && base + w * SEG < total; ++w)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            sum[e].x += s_part[w][3 * e][lane];
                            sum[e].y += s_part[w][3 * e + 1][lane];
                            sum[e].z += s_part[w][3 * e + 2][lane];
                        }
                    __syncthreads();
                }
                if (warp != 0) continue;  // every warp has the sums; one writes them
            }
            if constexpr (HALVES) {
                if (mine0 >= 0 && !sum[0].zero()) out.add(leaf, sum[0]);
                if (mine1 >= 0 && !sum[1].zero()) out.add(leaf1, sum[1]);
            } else if (mine0 >= 0) {
                if (!sum[0].zero()) out.add(leaf, sum[0]);
                if (!sum[1].zero()) out.add(leaf + 4, sum[1]);
            }
        }
    }
    if (missing) atomicOr(t.err, (unsigned)OT_DEV_STENCIL);
}

// lmax = 1: 8 finest leaves, smaller than a tile, which (nearly) every marker reaches.  A thread keeps the
// sums of all 8 for the markers of its stride, from the marker's weights per axis and half; they are
// added up in a fixed tree per block, and the blocks' in a fixed tree by a last block.  The number of
// blocks depends on n only, so the order does too.  2M markers 77 us in FP32 and 1.24 ms in FP64, whose
// pipe bounds it (one thread per leaf over all markers, as before, took 2.2 s in FP32).
constexpr int UNIT_T = 256, UNIT_BLOCKS = 608;
int64_t unit_blocks(int64_t n) { return std::min<int64_t>(UNIT_BLOCKS, (n + UNIT_T - 1) / UNIT_T); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) v += __shfl_xor_sync(0xffffffffu, v, k);
    return v;
}
template <typename T>
__device__ __forceinline__ void add_unit(T* f, int leaf, T x, T y, T z) {
    Acc3<T> a;
    a.x = x, a.y = y, a.z = z;
    if (!a.zero()) add_leaf<false>(f, leaf, a);
}

// part (24 sums per block) is not written by a single block, which adds to f.
template <typename T, int K>
__global__ void __launch_bounds__(UNIT_T) k_spread_unit(TreeView t, const double* __restrict__ x,
                                                        const double* __restrict__ y, const double* __restrict__ z,
                                                        const T* __restrict__ F, const T* __restrict__ dV, int64_t n,
                                                        T* __restrict__ part, T* __restrict__ f) {
    constexpr int W = Stencil<K>::W, NW = UNIT_T / 32;
    __shared__ T s_part[NW][24];
    Acc3<T> acc[8];
    bool out = false, miss = false;
    for (int64_t k = blockIdx.x * (int64_t)UNIT_T + threadIdx.x; k < n; k += (int64_t)gridDim.x * UNIT_T) {
        uint64_t X[3];
        if (!fixpoint3(x[k], y[k], z[k], X)) {
            out = true;
            continue;
        }
        int i0[3];
        T w[3][W];
        stencil_weights<K, T>(1, X, i0, w);
        const T vol = marker_volume(dV, k, 1);
        const T F0 = F[k] * vol, F1 = F[n + k] * vol, F2 = F[2 * n + k] * vol;
        T wd[3][2];  // per axis and half, the stencil cells that lie in (or wrap onto) it
        unsigned any = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            wd[d][0] = wd[d][1] = T(0);
#pragma unroll
            for (int a = 0; a < W; ++a) {
                const int c = t.periodic ? (i0[d] + a) & 1 : i0[d] + a;
                if (c < 0 || c > 1) {
                    miss = true;
                    continue;
                }
                if (c == 0) wd[d][0] += w[d][a];
                else wd[d][1] += w[d][a];
                any |= 1u << (2 * d + c);
            }
        }
#pragma unroll
        for (int leaf = 0; leaf < 8; ++leaf) {
            const int c[3] = {leaf & 1, (leaf >> 1) & 1, leaf >> 2};
            const unsigned need = (1u << c[0]) | (4u << c[1]) | (16u << c[2]);
            if ((any & need) == need) acc[leaf].add(wd[0][c[0]] * wd[1][c[1]] * wd[2][c[2]], F0, F1, F2);
        }
    }
    if (out) atomicOr(t.err, (unsigned)OT_DEV_OUTSIDE);
    if (miss) atomicOr(t.err, (unsigned)OT_DEV_STENCIL);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int leaf = 0; leaf < 8; ++leaf) {
        const T a[3] = {warp_sum(acc[leaf].x), warp_sum(acc[leaf].y), warp_sum(acc[leaf].z)};
        if (lane == 0)
#pragma unroll
            for (int d = 0; d < 3; ++d) s_part[warp][3 * leaf + d] = a[d];
    }
    __syncthreads();
    if (threadIdx.x < 24) {
        T a = T(0);
#pragma unroll
        for (int w = 0; w < NW; ++w) a += s_part[w][threadIdx.x];
        if (gridDim.x > 1) part[24 * (int64_t)blockIdx.x + threadIdx.x] = a;
        else s_part[0][threadIdx.x] = a;  // (this thread's alone)
    }
    if (gridDim.x > 1) return;
    __syncthreads();
    if (threadIdx.x < 8) {
        const T* a = s_part[0] + 3 * threadIdx.x;
        add_unit(f, (int)threadIdx.x, a[0], a[1], a[2]);
    }
}
// Warp w: leaf w's sums over the blocks.
template <typename T>
__global__ void __launch_bounds__(256) k_spread_unit_sum(const T* __restrict__ part, int nb, T* __restrict__ f) {
    const int lane = threadIdx.x & 31, leaf = threadIdx.x >> 5;
    T a[3] = {T(0), T(0), T(0)};
    for (int b = lane; b < nb; b += 32)
#pragma unroll
        for (int d = 0; d < 3; ++d) a[d] += part[24 * b + 3 * leaf + d];
#pragma unroll
    for (int d = 0; d < 3; ++d) a[d] = warp_sum(a[d]);
    if (lane == 0) add_unit(f, leaf, a[0], a[1], a[2]);
}

template <typename Kern>
unsigned grid_for(Kern k, int block, size_t smem, int64_t n) {
    const int per_sm = blocks_per_sm((const void*)k, block, smem);
    int64_t need = (n + block - 1) / block;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms() * per_sm, need));
}

size_t align_up(size_t b) { return (b + 255) & ~(size_t)255; }

int index_bits(int64_t n) {
    int b = 1;
    while (b < 40 && ((int64_t)1 << b) < n) ++b;
    return b;
}

// Places of the run table: a power of two, at least 1.5 per marker.
uint64_t table_size(int64_t n) {
    uint64_t p = 64;
    while (2 * p < 3 * (uint64_t)n) p <<= 1;
    return p;
}

size_t sorted_ws_bytes(int64_t n, size_t rec) {
    return 2 * align_up((size_t)n * 8) + align_up(radix_ws_bytes(n)) + align_up((size_t)n * rec) +
           align_up((size_t)table_size(n) * 8) + align_up((size_t)n * 4) + 256 + 256;
}

// What a sorted spreading keeps in its workspace.
template <typename T> struct TilePlan {
    TileOrder o;
    MarkerRec<T>* recs;
    RunTable rt;
    uint32_t *runs, *n_runs;
};

// Sorts the markers by home tile and writes records (forces from F when given) and runs.
template <typename T, int K>
ot_status plan_tiles(const ot_octree* t, const double* x, const double* y, const double* z, const T* F, const T* dV,
                     int64_t n, void* ws, cudaStream_t s, TilePlan<T>& pl) {
    // from a 256-byte boundary (records are read in 16-byte pieces)
    char* p = reinterpret_cast<char*>(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    auto take = [&p](size_t bytes) {
        char* r = p;
        p += align_up(bytes);
        return r;
    };
    uint64_t* pairs = reinterpret_cast<uint64_t*>(take((size_t)n * 8));
    uint64_t* tmp = reinterpret_cast<uint64_t*>(take((size_t)n * 8));
    void* rws = take(radix_ws_bytes(n));
    pl.recs = reinterpret_cast<MarkerRec<T>*>(take((size_t)n * sizeof(MarkerRec<T>)));
    pl.rt = RunTable{reinterpret_cast<unsigned long long*>(take((size_t)table_size(n) * 8)),
                     (uint32_t)(table_size(n) - 1)};
    pl.runs = reinterpret_cast<uint32_t*>(take((size_t)n * 4));
    pl.n_runs = reinterpret_cast<uint32_t*>(take(4));
    const int bits = 3 * (t->lmax - 2), ib = index_bits(n), room = 64 - ib;
    TileOrder& o = pl.o;
    o = TileOrder{pairs, x, y, z, n, ib, bits <= room, t->lmax, t->periodic};
    ot_status st;
    if (n <= SMALL_SORT && o.whole) {
        auto k = k_tile_sort_small<K>;
        OT_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM));
        k<<<1, SMALL_T, SMALL_SMEM, s>>>(o, bits, pairs, pl.rt, pl.n_runs);
        count_launch();
    } else {
        uint64_t* cur = nullptr;  // the markers' order so far (null: as given)
        for (int sh = 0; sh == 0 || sh < bits; sh += room) {
            const int nb = std::min(bits - sh, room);
            uint64_t* a = cur ? cur : pairs;
            auto k = k_tile_keys<K>;
            k<<<grid_for(k, 256, 0, n), 256, 0, s>>>(o, cur, sh, nb, a, pl.rt, pl.n_runs);
            count_launch();
            if ((st = radix_sort_u64_ws(a, a == pairs ? tmp : pairs, n, ib, ib + nb, rws, s, &cur)) != OT_OK)
                return st;
        }
        o.pairs = cur;
    }
    auto kr = k_tile_records<T, K>;
    kr<<<grid_for(kr, REC_T, 0, n), REC_T, 0, s>>>(o, F, dV, pl.recs, pl.rt, pl.runs, pl.n_runs, t->d_err);
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

// Sums to f and, scaled, to u (nullable).  (Whether they allow wide accesses is a template argument: asked
// per leaf it cost multi-direct forcing on few markers 2%.)
template <typename T, int K>
ot_status reduce_tiles(const TreeView& v, const TilePlan<T>& pl, T* f, T* u, T scale, cudaStream_t s) {
    auto launch = [&](auto vec) {
        constexpr bool VEC = decltype(vec)::value;
        auto kt = k_tile_reduce<T, K, VEC>;
        kt<<<grid_for(kt, TILE_T, 0, pl.o.n * 8 * TILE_T), TILE_T, 0, s>>>(v, pl.o, pl.rt, pl.runs, pl.n_runs, pl.recs,
                                                                         TileOut<T, VEC>{f, u, scale});
    };
    if (sizeof(T) == 8 || (((uintptr_t)f | (uintptr_t)u) & 15) == 0)
        launch(std::true_type{});
    else
        launch(std::bool_constant<sizeof(T) == 8>{});
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

template <typename T, int K>
ot_status spread_sorted(const ot_octree* t, const double* x, const double* y, const double* z, const T* F,
                        const T* dV, int64_t n, T* f, void* ws, cudaStream_t s) {
    TreeView v = tree_view(t);
    if (t->lmax < 2) {
        // 24 sums per 256 markers: less than the 16 bytes per marker of the workspace's first part
        T* part = reinterpret_cast<T*>(ws);
        const int nb = (int)unit_blocks(n);
        k_spread_unit<T, K><<<nb, UNIT_T, 0, s>>>(v, x, y, z, F, dV, n, part, f);
        count_launch();
        if (nb > 1) {
            k_spread_unit_sum<T><<<1, 256, 0, s>>>(part, nb, f);
            count_launch();
        }
        OT_CUDA(cudaGetLastError());
        return OT_OK;
    }
    TilePlan<T> pl;
    const ot_status st = plan_tiles<T, K>(t, x, y, z, F, dV, n, ws, s, pl);
    return st == OT_OK ? reduce_tiles<T, K>(v, pl, f, nullptr, T(0), s) : st;
}

// Marker forces of a round of multi-direct forcing, in home-tile order: the velocity interpolated at
// each marker, F = (U - u) / dt times the volume factor into its record, and the squared slip
// summed into *slip2 (nullable; FP64, one atomic per block).  forces 0: the slip only.
// A warp takes `per` consecutive markers (at most 32).  The records hold the weights, and the
// markers of a run share the 4x4x4 blocks of finest leaves from their home tile on, looked up
// once per run; then 8 lanes per marker sum its stencil as delta_sum does.
template <int K>
__global__ void __launch_bounds__(REC_T) k_tile_forces(TreeView t, TileOrder o, MarkerRec<float>* __restrict__ recs,
                                                       const float* __restrict__ field, const float* __restrict__ U,
                                                       const float* __restrict__ dV, float inv_dt, int per, int forces,
                                                       double* __restrict__ slip2) {
    constexpr int W = Stencil<K>::W;
    constexpr unsigned FULLM = 0xffffffffu;
    __shared__ int s_blk[REC_T / 32][64];
    __shared__ double s_part[REC_T / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ch = lane & 7;
    int* blk = s_blk[warp];
    const int64_t n = o.n, nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int nb = 1 << (o.lmax - 1);  // blocks per axis
    const int shb = MAXLEVEL - (o.lmax - 1);
    double slip = 0.0;
    bool missing = false;
    for (int64_t base = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * per; base < n; base += nwarps * per) {
        const int cnt = (int)min((int64_t)per, n - base);
        const uint64_t tile = lane < cnt ? tile_at<K>(o, base + lane) : ~0ULL;
        for (int s0 = 0; s0 < cnt;) {  // the warp's markers of one tile: s0 .. s1 - 1
            const uint64_t here = __shfl_sync(FULLM, tile, s0);
            const unsigned rest = ~__ballot_sync(FULLM, tile == here) & (FULLM << s0);
            const int s1 = rest ? min(__ffs(rest) - 1, cnt) : cnt;
            uint32_t h[3];
            demorton3(here, h[0], h[1], h[2]);
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int k = lane + 32 * r, b[3] = {k & 3, (k >> 2) & 3, k >> 4};
                bool inside = true;
                uint64_t q = 0;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    int v = 2 * (int)h[d] + b[d];
                    if (o.periodic) v &= nb - 1;
                    inside = inside && v < nb;
                    q |= part1by2((uint32_t)v << shb) << d;
                }
                blk[k] = inside ? find_block<false>(t, q) : -1;
            }
            __syncwarp();
            for (int m = s0 + (lane >> 3); __any_sync(FULLM, m < s1); m += 4) {
                float u0 = 0.0f, u1 = 0.0f, u2 = 0.0f;
                uint32_t off = OFF_NONE;
                if (m < s1) off = bits_of(recs[base + m].off);
                const bool ok = off != OFF_NONE;
                if (ok) {
                    const MarkerRec<float>& rc = recs[base + m];
                    float w[3][2];
                    int b0[3];
                    bool two[3];
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const int rel = (int)((off >> (8 * d)) & 0xffu) - 8, par = rel & 1, cd = (ch >> d) & 1;
                        const int a = cd ^ par;
                        b0[d] = (rel >> 1) + (par & ~cd);
                        two[d] = W == 4 || a == 0;
                        w[d][0] = rc.w[d][a];
                        w[d][1] = rc.w[d][a + 2];
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int ex = e & 1, ey = (e >> 1) & 1, ez = e >> 2;
                        if ((ex && !two[0]) || (ey && !two[1]) || (ez && !two[2])) continue;
                        const int bx = b0[0] + ex, by = b0[1] + ey, bz = b0[2] + ez;
                        // (a stencil that starts outside the cube: blocks before the tile's)
                        const int first = (bx | by | bz) >= 0 ? blk[bx + 4 * by + 16 * bz] : -1;
                        missing = missing || first < 0;
                        if (first < 0) continue;
                        const float4 f = Vec4<float>::load(field, first + ch);
                        const float wt = w[0][ex] * w[1][ey] * w[2][ez];
                        u0 += wt * f.x;
                        u1 += wt * f.y;
                        u2 += wt * f.z;
                    }
                }
#pragma unroll
                for (int k = 1; k < 8; k <<= 1) {
                    u0 += __shfl_xor_sync(FULLM, u0, k);
                    u1 += __shfl_xor_sync(FULLM, u1, k);
                    u2 += __shfl_xor_sync(FULLM, u2, k);
                }
                if (m < s1 && ch < 3) {
                    const int64_t k = (int64_t)(o.pairs[base + m] & ((1ULL << o.ib) - 1));
                    const float uk = ok ? (ch == 0 ? u0 : ch == 1 ? u1 : u2) : qnan<float>();
                    const float e = U[ch * n + k] - uk;
                    if (forces && ok) recs[base + m].F[ch] = e * inv_dt * marker_volume(dV, k, o.lmax);
                    slip += (double)e * (double)e;
                }
            }
            s0 = s1;
        }
    }
    if (missing) atomicOr(t.err, (unsigned)OT_DEV_STENCIL);
    if (!slip2) return;
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) slip += __shfl_xor_sync(FULLM, slip, k);
    if (lane == 0) s_part[warp] = slip;
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0.0;
        for (int w = 0; w < REC_T / 32; ++w) b += s_part[w];
        atomicAdd(slip2, b);
    }
}

template <int K>
ot_status mdf_tiles(const ot_octree* t, const double* x, const double* y, const double* z, const float* U,
                    const float* dV, int64_t n, float rho, float dt, int n_iter, float* u, float* f, double* slip2,
                    void* ws, cudaStream_t s) {
    TreeView v = tree_view(t);
    TilePlan<float> pl;
    ot_status st = plan_tiles<float, K>(t, x, y, z, nullptr, dV, n, ws, s, pl);
    auto k = k_tile_forces<K>;
    const unsigned grid = grid_for(k, REC_T, 0, n * 8);
    const int64_t warps = (int64_t)grid * (REC_T / 32);
    const int per = (int)std::min<int64_t>(32, std::max<int64_t>(4, (n + warps - 1) / warps));
    for (int it = 0; st == OT_OK && it <= n_iter; ++it) {
        if (it == n_iter && !slip2) break;  // the last interpolation is for the slip alone
        k<<<grid, REC_T, 0, s>>>(v, pl.o, pl.recs, u, U, dV, 1.0f / dt, per, it < n_iter, slip2 ? slip2 + it : nullptr);
        count_launch();
        if (it < n_iter) st = reduce_tiles<float, K>(v, pl, f, u, dt / rho, s);
    }
    OT_CUDA(cudaGetLastError());
    return st;
}

} // namespace

size_t spread_ws_bytes(const ot_octree* t, int kernel, int64_t n) {
    (void)t, (void)kernel;
    return sorted_ws_bytes(n, sizeof(MarkerRec<double>));
}

template <typename T>
ot_status launch_spread(const ot_octree* t, int kernel, int mode, const double* x, const double* y, const double* z,
                        const T* F, const T* dV, int64_t n, T* f, void* ws, size_t ws_bytes, cudaStream_t s) {
    if (n == 0) return OT_OK;
    if (mode == OT_SORTED) {
        if (ws_bytes < spread_ws_bytes(t, kernel, n)) return OT_ERR_ARG;
        if (kernel == OT_PESKIN4) return spread_sorted<T, OT_PESKIN4>(t, x, y, z, F, dV, n, f, ws, s);
        return spread_sorted<T, OT_ROMA3>(t, x, y, z, F, dV, n, f, ws, s);
    }
    TreeView v = tree_view(t);
    if (kernel == OT_PESKIN4) {
        auto k = k_spread_atomic<T, OT_PESKIN4>;
        k<<<grid_for(k, 256, 0, n), 256, 0, s>>>(v, x, y, z, F, dV, n, f);
    } else {
        auto k = k_spread_atomic<T, OT_ROMA3>;
        k<<<grid_for(k, 256, 0, n), 256, 0, s>>>(v, x, y, z, F, dV, n, f);
    }
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

template ot_status launch_spread<float>(const ot_octree*, int, int, const double*, const double*, const double*,
                                        const float*, const float*, int64_t, float*, void*, size_t, cudaStream_t);
template ot_status launch_spread<double>(const ot_octree*, int, int, const double*, const double*, const double*,
                                         const double*, const double*, int64_t, double*, void*, size_t, cudaStream_t);

// Rounds of multi-direct forcing on trees of two levels or more (see ot_mdf.cu): the markers are
// sorted and their records written once, a round is two launches.  ws: spread_ws_bytes.
ot_status launch_mdf_tiles(const ot_octree* t, int kernel, const double* x, const double* y, const double* z,
                           const float* U, const float* dV, int64_t n, float rho, float dt, int n_iter, float* u,
                           float* f, double* slip2, void* ws, cudaStream_t s) {
    if (kernel == OT_PESKIN4)
        return mdf_tiles<OT_PESKIN4>(t, x, y, z, U, dV, n, rho, dt, n_iter, u, f, slip2, ws, s);
    return mdf_tiles<OT_ROMA3>(t, x, y, z, U, dV, n, rho, dt, n_iter, u, f, slip2, ws, s);
}

// The same spreading with caller scratch of spread_noalloc_bytes(n) bytes (FP32 records).
size_t spread_noalloc_bytes(int64_t n) { return sorted_ws_bytes(n, sizeof(MarkerRec<float>)); }

ot_status launch_spread_sorted_noalloc(const ot_octree* t, int kernel, const double* x, const double* y,
                                       const double* z, const float* F, const float* dV, int64_t n, float* f,
                                       void* scratch, cudaStream_t s) {
    if (n == 0) return OT_OK;
    if (kernel == OT_PESKIN4) return spread_sorted<float, OT_PESKIN4>(t, x, y, z, F, dV, n, f, scratch, s);
    return spread_sorted<float, OT_ROMA3>(t, x, y, z, F, dV, n, f, scratch, s);
}

} // namespace ot
