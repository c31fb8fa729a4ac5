// ot_queue.cuh -- warp-cooperative host-cell search over a per-warp task list, and the
// trilinear interpolation (Sec. 2.3.2, level-mate rule) built on it.
//
// A point needs up to 8 searches (its host, then its level-mates).  Most are answered by the
// descriptor of the key's level-map cell, one load.  Those in deeper subtrees, and the learned
// search, take up to ~12 dependent key probes, so a warp that gave each lane its own would
// idle most lanes: every corner would cost the longest lane's search.  There the lanes
// first append every search they need to a task list in shared memory (ballot + popc, no
// atomics); then each lane takes the next task whenever its current one ends and performs one
// probe per step.  The warp's step count follows the total number of probes / 32 instead of the
// sum over corners of the longest lane's.  Results are exactly those of the per-lane searches
// (the same halving over the same range).
#pragma once

#include "ot_points.cuh"

namespace ot {

constexpr int QCAP = 7 * 32;  // level-mate searches of a warp's 32 points (the host's need 32)
constexpr unsigned FULL = 0xffffffffu;

// A warp's task list: key searched, and the range to search (the uncovered level-map cell);
// lo holds the answer once the task has run.  CAP tasks: QCAP for the level-mate searches, 32
// where only the hosts are searched (the level-mate table gives the rest).
template <int CAP>
struct WarpQueueN {
    static constexpr int cap = CAP;
    uint64_t q[CAP];
    int lo[CAP];
    int len[CAP];
};
using WarpQueue = WarpQueueN<QCAP>;
using HostQueue = WarpQueueN<32>;

// The root model of the learned index, staged in shared memory by every block that searches
// with it (block-wide call; a no-op for the plain form).
template <bool LEARNED>
__device__ __forceinline__ void stage_root(const TreeView& t, RootModel& s_root) {
    if (LEARNED) {
        const int* src = reinterpret_cast<const int*>(t.root);
        int* dst = reinterpret_cast<int*>(&s_root);
        for (int i = threadIdx.x; i < (int)(sizeof(RootModel) / sizeof(int)); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
}

// Level-map lookup of key q by its cell's descriptor: true with the leaf (a) and its level (lv) when
// the cell is covered by one leaf or, for the plain search, its subtree is at most 3 levels
// deep; else false with the cell's leaf range [a, e) to search.
template <bool LEARNED>
__device__ __forceinline__ bool map_lookup(const TreeView& t, uint64_t q, int& a, int& e, int& lv) {
    const uint32_t cell = map_cell(t, q);
    const uint4 d = __ldg(t.desc + cell);
    if (LEARNED ? (d.z & DESC_COVERED) != 0 : !(d.z & DESC_DEEP) || (d.z & DESC_COVERED)) {
        desc_resolve(d, t.lmap_level, q, a, lv);
        return true;
    }
    a = (int)d.w;
    e = map_end(t, cell);
    lv = -1;
    return false;
}

// Appends a task for every lane with need set (warp-wide call); returns the lane's task index
// or -1.  n is the warp-uniform task count.
template <typename Q>
__device__ __forceinline__ int push_task(Q& w, int& n, bool need, uint64_t q, int lo, int len, unsigned lt) {
    const unsigned m = __ballot_sync(FULL, need);
    const int idx = n + __popc(m & lt);
    n += __popc(m);
    if (need) {
        w.q[idx] = q;
        w.lo[idx] = lo;
        w.len[idx] = len;
    }
    return need ? idx : -1;
}

// Runs the warp's ntask tasks (warp-wide call).  Each step, a lane without a task takes the
// next one, and every lane with a task advances it by one step of at most one memory round
// trip:
//   plain:   halving probes over the cell's leaves;
//   learned: route (root model from shared memory, then the middle model's load), leaf model
//            load and window (its prediction widened by the stored error bounds, clamped to
//            the cell), halving probes over the window, and the check key[a] <= q < key[a+1];
//            a window that missed is replaced by the whole cell (a counted fallback).
// A finished task's answer (the last index in its range whose key is <= q) replaces its lo.
// (Routing all tasks side by side before the loop was measured slower: it adds a round trip
// and registers.)
enum { ST_ROUTE = 0, ST_MODEL = 1, ST_PROBE = 2, ST_CHECK = 3, ST_DONE = 4 };

template <bool LEARNED, typename Q>
__device__ __forceinline__ void run_tasks(const TreeView& t, const RootModel& root, Q& w, int ntask,
                                          unsigned lt) {
    __syncwarp();
    int cur = -1, lo = 0, len = 0, next = 0, st = ST_DONE, clo = 0, clen = 0, j = 0;
    bool checked = false;
    uint64_t q = 0;
    for (;;) {
        const bool fin = cur >= 0 && st == ST_DONE;
        if (fin) w.lo[cur] = lo;
        const bool need = cur < 0 || fin;
        const unsigned m = __ballot_sync(FULL, need);
        if (need) {
            const int idx = next + __popc(m & lt);
            cur = -1;
            if (idx < ntask) {
                cur = idx;
                q = w.q[idx];
                lo = clo = w.lo[idx];
                len = clen = w.len[idx];
                st = LEARNED ? ST_ROUTE : ST_PROBE;
                checked = false;
            }
        }
        next += __popc(m);
        if (!__any_sync(FULL, cur >= 0)) break;
        if (cur < 0) continue;
        if (LEARNED && st == ST_ROUTE) {
            j = root_route(root, q);
            if (t.mids) j = (int)(((int64_t)leaf_predict(t.mids[j], q, t.n) * t.n_leaf) / t.n);
            st = ST_MODEL;
        } else if (LEARNED && st == ST_MODEL) {
            const LeafModel md = t.models[j];
            int wl = clo, wh = clo + clen - 1;
            if (md.count > 0) {
                const int pc = leaf_predict(md, q, t.n);
                wl = max(pc - md.err_lo - 1, clo);
                wh = min(pc + md.err_hi + 1, clo + clen - 1);
            }
            if (md.count > 0 && wl <= wh) {
                lo = wl;
                len = wh - wl + 1;
            } else {
                atomicAdd(t.fallbacks, 1ULL);
                atomicOr(t.err, (unsigned)OT_DEV_WINDOW);
                checked = true;  // the whole cell: its answer needs no check
            }
            st = ST_PROBE;
        } else if (st == ST_PROBE) {
            if (len > 1) {
                const int half = len >> 1;
                const uint64_t k = ldg_key(t.key + lo + half);
                lo = (k <= q) ? lo + half : lo;
                len -= half;
            }
            if (len <= 1) st = (LEARNED && !checked) ? ST_CHECK : ST_DONE;
        } else if (LEARNED && st == ST_CHECK) {
            const uint64_t k0 = ldg_key(t.key + lo);
            const uint64_t k1 = lo + 1 < t.n ? ldg_key(t.key + lo + 1) : ~0ULL;
            checked = true;
            st = ST_DONE;
            if (!(k0 <= q && q < k1)) {
                atomicAdd(t.fallbacks, 1ULL);
                atomicOr(t.err, (unsigned)OT_DEV_WINDOW);
                lo = clo;
                len = clen;
                st = len > 1 ? ST_PROBE : ST_DONE;
            }
        }
    }
    __syncwarp();
}

// Host leaf of the point with fixed-point coordinates X, for the lanes with ok set and no host
// given (h < 0) (warp-wide call): the level-map lookup, then the warp's task list for the lanes
// that it does not answer.  hl receives the leaf's level when the lookup gave it, else stays -1.
template <bool LEARNED, typename Q>
__device__ __forceinline__ void host_queued(const TreeView& t, const RootModel& root, Q& w, bool ok,
                                            const uint64_t X[3], int& h, int& hl) {
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    const uint64_t q = morton3((uint32_t)(X[0] >> 32), (uint32_t)(X[1] >> 32), (uint32_t)(X[2] >> 32));
    int ca = 0, ce = 0, clv = -1;
    const bool need = ok && h < 0 && !map_lookup<LEARNED>(t, q, ca, ce, clv);
    if (ok && h < 0 && !need) h = ca, hl = clv;
    if (__any_sync(FULL, need)) {
        int n = 0;
        const int ix = push_task(w, n, need, q, ca, ce - ca, lt);
        run_tasks<LEARNED>(t, root, w, n, lt);
        if (ix >= 0) h = w.lo[ix], hl = -1;
        __syncwarp();
    }
}

// Octant of the point with fixed-point coordinates X in its host leaf of level l (bit d: the
// upper half on axis d, where the host is the lower of the two level-mates) and per axis the
// weights of the lower and the upper level-mate (Sec. 2.3.2), 1 - |t_d| for the host's and
// |t_d| for the neighbour's, t_d the offset from the host's centre in cell units.
template <typename T>
__device__ __forceinline__ int tri_octant(const uint64_t X[3], int l, T f[3][2]) {
    int o = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const bool up = fix_upper_half(X[d], l);
        o |= (up ? 1 : 0) << d;
        const T td = fix_offset<T>(X[d], l);
        const T at = td < T(0) ? -td : td;
        f[d][0] = up ? T(1) - at : at;
        f[d][1] = up ? at : T(1) - at;
    }
    return o;
}

// The trilinear sum over the 8 level-mate values v by position (bit d of the corner: the upper
// cell on axis d), accumulated in that order, whichever of the 8 is the host: points around one
// grid node share its 8 values in one order.  Every form of the trilinear interpolation sums so,
// so their results are bit-identical.
template <typename T>
__device__ __forceinline__ void tri_sum(const T f[3][2], const T v[8][3], T out[3]) {
    // corner weight (f_0 f_1) f_2: the four x-y products once
    const T wxy[4] = {f[0][0] * f[1][0], f[0][1] * f[1][0], f[0][0] * f[1][1], f[0][1] * f[1][1]};
    T acc0 = T(0), acc1 = T(0), acc2 = T(0);
#pragma unroll
    for (int corner = 0; corner < 8; ++corner) {
        const T wc = wxy[corner & 3] * f[2][corner >> 2];
        acc0 += wc * v[corner][0];
        acc1 += wc * v[corner][1];
        acc2 += wc * v[corner][2];
    }
    out[0] = acc0;
    out[1] = acc1;
    out[2] = acc2;
}

// A point's host leaf and level-mates (Sec. 2.3.2 with the level-mate rule): host leaf of level l, cell
// c; t_d = offset from the cell centre; s_d = +1 if t_d >= 0; level-mates c + {0, s_d}; outside the
// cube the host's index on that axis, or the wrapped index when periodic.
template <typename T>
struct TriCorners {
    int h, l;         // host leaf and its level
    T f[3][2];        // weights per axis, lower and upper cell
    uint64_t anc[8];  // anchors of the level-mates, by position
    int a[8], lvl[8]; // the leaf that holds each anchor and its level (above l: the level-mate is refined)
    // Entry of the cell means (in values of 4) of refined corner k.
    __device__ __forceinline__ long long mean(const TreeView& t, int k) const {
        if (l <= t.pyr_level) return pyr_offset(l) + (long long)(anc[k] >> (3 * (MAXLEVEL - l)));
        return pyr_offset(t.pyr_level + 1) + (long long)(l - t.pyr_level - 1) * t.n + a[k];
    }
};

// Resolves the corners of one point per lane (warp-wide call); ok: the lane has a point inside the
// cube, with fixed-point coordinates X.  host_in >= 0 gives the host.
template <typename T, bool LEARNED>
__device__ __forceinline__ void tri_corners(const TreeView& t, const RootModel& root, WarpQueue& w, bool ok,
                                            const uint64_t X[3], int host_in, TriCorners<T>& c8) {
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    // host (and its level, when the lookup gives it)
    int h = host_in, hl = -1;
    host_queued<LEARNED>(t, root, w, ok, X, h, hl);
    if (!ok) h = 0, hl = -1;  // keeps the lane's reads in bounds; its result is discarded
    const int l = hl >= 0 ? hl : (int)t.level[h];
    c8.h = h, c8.l = l;
    const int ncell = 1 << l;
    int c[3];
    const int oct = tri_octant<T>(X, l, c8.f);
#pragma unroll
    for (int d = 0; d < 3; ++d) c[d] = (int)fix_cell(X[d], l);
    const int sh = MAXLEVEL - l;
    // per axis the lower and the upper level-mate index (the host's, and the neighbour's clamped
    // into the cube) and their Morton bits: each corner's anchor is the OR of three of these six
    unsigned self_m = 0u;
    int ix[3][2];
    uint64_t dil[3][2];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const bool up = (oct >> d) & 1;  // the neighbour is the upper one
        int nb = c[d] + (up ? 1 : -1);
        if (nb < 0 || nb >= ncell) nb = t.periodic ? (nb + ncell) & (ncell - 1) : c[d];
        ix[d][0] = up ? c[d] : nb;
        ix[d][1] = up ? nb : c[d];
#pragma unroll
        for (int k = 0; k < 2; ++k) dil[d][k] = (part1by2((uint32_t)ix[d][k]) << d) << (3 * sh);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        c8.anc[k] = dil[0][k & 1] | dil[1][(k >> 1) & 1] | dil[2][k >> 2];
        if (ix[0][k & 1] == c[0] && ix[1][(k >> 1) & 1] == c[1] && ix[2][k >> 2] == c[2]) self_m |= 1u << k;
    }
    if (!ok) self_m = 0xffu;
    // the level-map lookups of the other corners, each one descriptor load and most with the answer and
    // its level; the rest become tasks of the warp's list
    unsigned pend_m = 0u;
    int ca[8], ce[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        ca[k] = ce[k] = 0;
        c8.a[k] = h;
        c8.lvl[k] = l;
        if ((self_m >> k) & 1u) continue;
        if (map_lookup<false>(t, c8.anc[k], ca[k], ce[k], c8.lvl[k]))
            c8.a[k] = ca[k];
        else
            pend_m |= 1u << k;
    }
    if (__any_sync(FULL, pend_m != 0u)) {
        int n = 0;
        int tix[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) tix[k] = push_task(w, n, (pend_m >> k) & 1u, c8.anc[k], ca[k], ce[k] - ca[k], lt);
        run_tasks<LEARNED>(t, root, w, n, lt);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (tix[k] >= 0) {
                c8.a[k] = w.lo[tix[k]];
                c8.lvl[k] = (int)t.level[c8.a[k]];
            }
        __syncwarp();
    }
}

// Trilinear interpolation at one point per lane (warp-wide call; Sec. 2.3.2): level-mate value: leaf of
// level l -> its value; inside a coarser leaf -> that leaf's value; refined -> volume-weighted mean of
// its leaves, one load: from the dense pyramid of cell means for l <= the pyramid level, else from
// the node means of level l (both in pyr).
// Lanes with active == false take part in the warp's steps only.  host_in >= 0 gives the host.
// Returns the host leaf (-1 when inactive or outside the cube, out = NaN).
template <typename T, bool LEARNED>
__device__ __forceinline__ int trilinear_queued(const TreeView& t, const RootModel& root, const T* __restrict__ field,
                                                const T* __restrict__ pyr, WarpQueue& w, bool active, double x,
                                                double y, double z, int host_in, T out[3]) {
    using V = Vec4<T>;
    uint64_t X[3] = {0, 0, 0};
    const bool ok = active && fixpoint3(x, y, z, X);
    if (active && !ok) atomicOr(t.err, (unsigned)OT_DEV_OUTSIDE);
    TriCorners<T> c8;
    tri_corners<T, LEARNED>(t, root, w, ok, X, host_in, c8);
    if (!ok) {
        out[0] = out[1] = out[2] = qnan<T>();
        return -1;
    }
    T v[8][3];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const bool refined = c8.lvl[k] > c8.l;
        const auto fv = V::load(refined ? pyr : field, refined ? c8.mean(t, k) : (long long)c8.a[k]);
        v[k][0] = fv.x, v[k][1] = fv.y, v[k][2] = fv.z;
    }
    tri_sum<T>(c8.f, v, out);
    return c8.h;
}

// The same interpolation with the level-mates read from the octree's level-mate table (built
// by ot_octree_build_mates): host leaf h of level l, octant o of its cell (bit d: the upper
// half on axis d), then row 8h + o gives the 8 value slots -- a leaf index, or (top bit set)
// an index into the cell means in pyr.  The weights, values and summation order are those of
// trilinear_queued: the results are bit-identical.  Warp-wide call (the host search).
template <typename T, bool LEARNED, typename Q>
__device__ __forceinline__ int trilinear_mates(const TreeView& t, const RootModel& root, const T* __restrict__ field,
                                               const T* __restrict__ pyr, Q& w, bool active, double x,
                                               double y, double z, int host_in, T out[3]) {
    using V = Vec4<T>;
    uint64_t X[3] = {0, 0, 0};
    const bool ok = active && fixpoint3(x, y, z, X);
    if (active && !ok) atomicOr(t.err, (unsigned)OT_DEV_OUTSIDE);
    int h = host_in, hl = -1;
    host_queued<LEARNED>(t, root, w, ok, X, h, hl);
    if (!ok) {
        out[0] = out[1] = out[2] = qnan<T>();
        return -1;
    }
    const int l = hl >= 0 ? hl : (int)t.level[h];
    T w8[3][2];
    const int o = tri_octant<T>(X, l, w8);
    const uint4* row = t.mates + 2 * (8 * (long long)h + o);
    const uint4 r0 = __ldg(row), r1 = __ldg(row + 1);
    const uint32_t sl[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
    T v[8][3];
#pragma unroll
    for (int corner = 0; corner < 8; ++corner) {
        const uint32_t sv = sl[corner];
        const auto f = V::load((sv >> 31) ? pyr : field, (long long)(sv & 0x7FFFFFFFu));
        v[corner][0] = f.x, v[corner][1] = f.y, v[corner][2] = f.z;
    }
    tri_sum<T>(w8, v, out);
    return h;
}

} // namespace ot
