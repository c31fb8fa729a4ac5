// ot_points.cuh -- per-point device routines: delta-kernel interpolation and stencil
// enumeration on exact fixed-point coordinates (the trilinear routine, which searches
// cooperatively across the warp, is in ot_queue.cuh).
// Used by the single-op kernels, the persistent batched kernel and the spreading kernels.
#pragma once

#include "ot_common.cuh"

namespace ot {

__device__ __forceinline__ int floordiv2(int v) { return v >> 1; } // arithmetic shift: floor

template <typename T> __device__ __forceinline__ T qnan();
template <> __device__ __forceinline__ float qnan<float>() { return __int_as_float(0x7fc00000); }
template <> __device__ __forceinline__ double qnan<double>() { return __longlong_as_double(0x7ff8000000000000LL); }


// First cell of level l in the pyramid of cell means: sum_{k<l} 8^k = (8^l - 1) / 7, the octal
// number 11...1 of l digits, i.e. the top l of the 21 octal ones of 0x1249249249249249 (no
// 64-bit division).
__device__ __forceinline__ long long pyr_offset(int l) { return (long long)(0x1249249249249249ULL >> (3 * (21 - l))); }

// Stencil origin and per-axis weights of a point with fixed-point coordinates X on the
// finest level lmax (Sec. 2.2: W(x) = prod phi(x_d/dx)/dx).
template <int K, typename T>
__device__ __forceinline__ void stencil_weights(int lmax, const uint64_t X[3], int i0[3], T w[3][Stencil<K>::W]) {
    constexpr int W = Stencil<K>::W;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int c = (int)fix_cell(X[d], lmax);
        const int hi = fix_upper_half(X[d], lmax) ? 1 : 0;
        const T t = fix_offset<T>(X[d], lmax);
        i0[d] = Stencil<K>::first(c, hi);
#pragma unroll
        for (int a = 0; a < W; ++a) w[d][a] = Stencil<K>::template phi<T>(Stencil<K>::template r<T>(a, hi, t));
    }
}

// Parent blocks (2x2x2 cells of level lmax, i.e. cells of level lmax-1) overlapping the
// delta-kernel stencil whose first cell is i0.  With the parent-block table, the middle block's
// row gives every block's first child; otherwise one search per block finds it.  A parent
// whose first child is a leaf of level lmax has all 8 children as consecutive leaves.  The visitor gets
// (a0, bx, by, bz, P) with a0 the first child's index, or -1 when the parent is outside the
// cube (a periodic cube wraps it instead) or not refined to the finest level.
template <int K, bool LEARNED, typename PVisit>
__device__ __forceinline__ void visit_parents(const TreeView& t, const int i0[3], PVisit&& pvisit) {
    constexpr int W = Stencil<K>::W;
    const int lp = t.lmax - 1;     // parent level
    const int np_cells = 1 << lp;  // parents per axis
    const int shp = MAXLEVEL - lp;
    int p0[3], pn[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        p0[d] = floordiv2(i0[d]);
        pn[d] = floordiv2(i0[d] + W - 1) - p0[d] + 1;
    }
    if (t.pnbr) {
        // the parent-block table: every stencil block lies within one block of the middle one,
        // whose row gives all their first children -- one lookup and one row of loads
        int pm[3], qm[3];
        bool inside = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            pm[d] = p0[d] + (pn[d] == 3 ? 1 : 0);
            qm[d] = t.periodic ? (pm[d] + np_cells) & (np_cells - 1) : pm[d];
            inside = inside && qm[d] >= 0 && qm[d] < np_cells;
        }
        int am = -1;
        if (inside) {
            const uint64_t anchor = morton3((uint32_t)qm[0] << shp, (uint32_t)qm[1] << shp, (uint32_t)qm[2] << shp);
            am = find_block<LEARNED>(t, anchor);
        }
        if (am >= 0) {  // else (the middle block is not refined to the finest level) the walk below
            const int* __restrict__ row = t.pnbr + 32 * (size_t)(am >> 3);
            for (int bz = 0; bz < pn[2]; ++bz)
                for (int by = 0; by < pn[1]; ++by)
                    for (int bx = 0; bx < pn[0]; ++bx) {
                        const int P[3] = {p0[0] + bx, p0[1] + by, p0[2] + bz};
                        const int k = (P[0] - pm[0] + 1) + 3 * (P[1] - pm[1] + 1) + 9 * (P[2] - pm[2] + 1);
                        pvisit(__ldg(row + k), bx, by, bz, P);
                    }
            return;
        }
    }
    for (int bz = 0; bz < pn[2]; ++bz)
        for (int by = 0; by < pn[1]; ++by)
            for (int bx = 0; bx < pn[0]; ++bx) {
                const int P[3] = {p0[0] + bx, p0[1] + by, p0[2] + bz};
                // the parent's own index (wrapped around a periodic cube); P stays unwrapped for
                // the stencil offsets the visitor computes
                int Q[3] = {P[0], P[1], P[2]};
                if (t.periodic)
#pragma unroll
                    for (int d = 0; d < 3; ++d) Q[d] = (Q[d] + np_cells) & (np_cells - 1);
                const bool inside = Q[0] >= 0 && Q[1] >= 0 && Q[2] >= 0 && Q[0] < np_cells && Q[1] < np_cells &&
                                    Q[2] < np_cells;
                int a0 = -1;
                if (inside)
                    a0 = find_block<LEARNED>(
                        t, morton3((uint32_t)Q[0] << shp, (uint32_t)Q[1] << shp, (uint32_t)Q[2] << shp));
                pvisit(a0, bx, by, bz, P);
            }
}

// The stencil cells themselves: the visitor gets (leaf, ax, ay, az) for each valid stencil
// cell.  Returns false when some stencil cell was outside the cube or not a finest-level leaf
// (its weight is dropped).
template <int K, bool LEARNED, typename Visit>
__device__ __forceinline__ bool visit_stencil(const TreeView& t, const int i0[3], Visit&& visit) {
    constexpr int W = Stencil<K>::W;
    bool ok_all = true;
    visit_parents<K, LEARNED>(t, i0, [&](int a0, int, int, int, const int P[3]) {
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
            const int ax = 2 * P[0] + (ch & 1) - i0[0];
            const int ay = 2 * P[1] + ((ch >> 1) & 1) - i0[1];
            const int az = 2 * P[2] + ((ch >> 2) & 1) - i0[2];
            if (ax < 0 || ay < 0 || az < 0 || ax >= W || ay >= W || az >= W) continue;
            if (a0 < 0) {
                ok_all = false;
                continue;
            }
            visit(a0 + ch, ax, ay, az);
        }
    });
    return ok_all;
}

// Delta-kernel interpolation (Sec. 2.2, Eq. ibm_interpolate): a warp takes up to 32 markers.  First a
// lane per marker forms the marker's weights and finds its middle block; then 8 lanes per marker,
// 4 markers at a time, sum its stencil.
// Lane c of a marker takes the stencil cells that are child c of their block of 8 finest leaves
// (2x2x2 cells): whatever the stencil's parity, two cells per axis, a and a + 2 (the second one
// past the 3-point stencil in half of the cases), so 8 per lane.  The 8 block entries are
// independent loads, and so are the 8 values, which the marker's lanes read from the same lines (a
// block's 8 leaves are 128 consecutive bytes in FP32).  A lane per marker walked 8 to 27 blocks in
// turn with 64 loads, each from a line of its own: bound by L1, and for few markers by that chain.
// 2M markers 506 -> 270 us, 1M without the table (uniform level 6) 537 -> 297 us, 1,000 markers
// 79 -> 5.5 us.  Forming the weights by 8 lanes per marker too, without the stage: 392 us.
// The lanes' sums are added in a fixed tree, the same with and without the parent-block table.
template <typename T>
struct DeltaStage {
    T w[12][33];       // weights by 4 axis + slot, one column per marker
    int row[32];       // row of the middle block in the parent-block table, -1: none
    int p0[3][32];     // first block per axis
    uint32_t bits[32]; // parity of the first cell (bits 0-2), host's slot (2 bits each from 4), inside the cube (16)
    int blk[4][28];    // without the table: first leaves of the 27 blocks from p0, of 4 markers
    T off[sizeof(T) == 8 ? 3 : 1][33];  // FP64: offset from the centre of the finest cell per axis
};

// FP64: the weights of the stage's first cnt markers, an evaluation per lane and round whatever their
// number.  By a lane per marker the few markers of a warp cost the FP64 pipe as much as 32: 3,000 and
// 30,000 3-point markers 35 -> 27 and 89 -> 65 us with the table.  The slots of one branch of the
// delta function come together.
template <int K>
__device__ __forceinline__ void stage_weights(DeltaStage<double>& sg, int cnt) {
    using S = Stencil<K>;
    constexpr int W = S::W, INNER = W == 4 ? 2 : 1;  // slots per axis within one cell of the marker
    for (int i = threadIdx.x & 31; i < 3 * W * cnt; i += 32) {
        const int j = i / cnt, m = i - j * cnt, o = j - 3 * INNER;
        const int d = o < 0 ? j / INNER : o >> 1, a = o < 0 ? 1 + j % INNER : (W - 1) * (o & 1);
        const int hc = (sg.bits[m] >> (4 + 2 * d)) & 3;
        sg.w[4 * d + a][m] = S::template phi<double>((double)(hc - a) + sg.off[d][m]);
    }
}

template <typename T, int K, bool LEARNED>
__device__ __forceinline__ void delta_stage(const TreeView& t, DeltaStage<T>& sg, bool active, double x, double y,
                                            double z) {
    using S = Stencil<K>;
    constexpr int W = S::W;
    const int lane = threadIdx.x & 31;
    const int lp = t.lmax - 1, np_cells = 1 << lp, shp = MAXLEVEL - lp;
    uint64_t X[3];
    const bool ok = active && fixpoint3(x, y, z, X);
    uint32_t bits = ok ? 1u << 16 : 0u;
    int row = -1;
    if (ok) {
        int i0[3];
        if constexpr (sizeof(T) == 4) {
            T w[3][W];
            stencil_weights<K, T>(t.lmax, X, i0, w);
#pragma unroll
            for (int d = 0; d < 3; ++d)
#pragma unroll
                for (int k = 0; k < W; ++k) sg.w[4 * d + k][lane] = w[d][k];
        } else {  // stage_weights, once all markers are here
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                i0[d] = S::first((int)fix_cell(X[d], t.lmax), fix_upper_half(X[d], t.lmax) ? 1 : 0);
                sg.off[d][lane] = fix_offset<T>(X[d], t.lmax);
            }
        }
        bool inside = true;
        uint64_t q = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int par = i0[d] & 1, p0 = floordiv2(i0[d]);
            bits |= (uint32_t)par << d;
            bits |= (uint32_t)((int)fix_cell(X[d], t.lmax) - i0[d]) << (4 + 2 * d);
            sg.p0[d][lane] = p0;
            // every block of the stencil lies within one of the middle one
            int qm = p0 + (W == 4 ? par : 0);
            if (t.periodic) qm = (qm + np_cells) & (np_cells - 1);
            inside = inside && qm >= 0 && qm < np_cells;
            q |= part1by2((uint32_t)qm << shp) << d;
        }
        if (t.pnbr && inside) {
            const int am = find_block<LEARNED>(t, q);
            if (am >= 0) row = am >> 3;
        }
    }
    sg.row[lane] = row;
    sg.bits[lane] = bits;
}

// The sum of marker m of the stage by its 8 lanes (m differs between them in the warp): lanes 0 to 2
// receive its components.  Returns the host leaf when the finest cell that holds the marker is
// one, else -1.
template <typename T, int K, bool LEARNED>
__device__ __forceinline__ int delta_sum(const TreeView& t, const T* __restrict__ field, DeltaStage<T>& sg, int m,
                                         T& out) {
    using V = Vec4<T>;
    constexpr int W = Stencil<K>::W;
    constexpr unsigned FULLM = 0xffffffffu;
    const int lane = threadIdx.x & 31, ch = lane & 7;
    const uint32_t bits = sg.bits[m];
    const bool ok = (bits >> 16) & 1u;
    const int row = sg.row[m];
    constexpr bool CELLS = W == 3 && sizeof(T) == 8;  // 27 cells dealt to the lanes, below
    [[maybe_unused]] int a[3], b0[3];  // this lane's first slot, and its block relative to p0
    [[maybe_unused]] bool two[3];      // slot a + 2 is in the stencil
    [[maybe_unused]] T w[3][2];
    [[maybe_unused]] int eh = 0;       // the host's cell among this lane's, 8 or more: another lane's
    if constexpr (!CELLS) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int par = (bits >> d) & 1, cd = (ch >> d) & 1, hc = (bits >> (4 + 2 * d)) & 3;
            a[d] = cd ^ par;
            b0[d] = par & ~cd;
            two[d] = W == 4 || a[d] == 0;
            w[d][0] = sg.w[4 * d + a[d]][m];
            w[d][1] = two[d] ? sg.w[4 * d + a[d] + 2][m] : T(0);
            eh = ((hc ^ a[d]) & 1) ? 8 : eh + (((hc - a[d]) >> 1) << d);
        }
    }
    const bool search = ok && row < 0;
    if (__any_sync(FULLM, search)) {  // no table, or the middle block is not refined to the finest level
        const int lp = t.lmax - 1, np_cells = 1 << lp, shp = MAXLEVEL - lp;
        int* blk = sg.blk[lane >> 3];
        // the blocks that the stencil overlaps, 2 per axis or, for odd first cells of 4, 3: a search per
        // lane and round (1 to 4 rounds; always 1 for the 3-point stencil)
        const int n0 = 2 + (W == 4 ? (int)bits & 1 : 0), n1 = 2 + (W == 4 ? (int)(bits >> 1) & 1 : 0);
        const int cnt = search ? n0 * n1 * (2 + (W == 4 ? (int)(bits >> 2) & 1 : 0)) : 0;
        for (int i = ch; __any_sync(FULLM, i < cnt); i += 8) {
            const int r = n0 == 2 ? i >> 1 : i / 3, z = n1 == 2 ? r >> 1 : r / 3;
            const int b[3] = {i - n0 * r, r - n1 * z, z};
            bool inside = i < cnt;
            uint64_t q = 0;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                int v = sg.p0[d][m] + b[d];
                if (t.periodic) v = (v + np_cells) & (np_cells - 1);
                inside = inside && v >= 0 && v < np_cells;
                q |= part1by2((uint32_t)v << shp) << d;
            }
            int f = -1;
            if (inside) f = find_block<LEARNED>(t, q);
            if (i < cnt) blk[b[0] + 3 * b[1] + 9 * b[2]] = f;
        }
        __syncwarp();
    }
    T s0 = T(0), s1 = T(0), s2 = T(0);
    int host = -1;
    bool missing = false;
    if constexpr (CELLS) {
        // 27 cells dealt to the lanes in turn, 4 each: by children the fullest lane has 8, and the FP64 pipe
        // takes as long for one lane as for all (1M markers 1,050 -> 761 us)
        int leaf[4];  // -1 when missing, -2 past the 27
        T wt[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int c = min(ch + 8 * r, 26), cell[3] = {c % 3, (c / 3) % 3, c / 9};
            int k = 0, child = 0;
#pragma unroll
            for (int d = 0, p3 = 1; d < 3; ++d, p3 *= 3) {
                const int at = (int)((bits >> d) & 1u) + cell[d];
                k += (at >> 1) * p3;
                child |= (at & 1) << d;
            }
            int first = -2;
            if (ok && ch + 8 * r < 27)
                first = row >= 0 ? __ldg(t.pnbr + 32 * (size_t)row + 13 + k) : sg.blk[lane >> 3][k];
            leaf[r] = first < 0 ? first : first + child;
            wt[r] = sg.w[cell[0]][m] * sg.w[4 + cell[1]][m] * sg.w[8 + cell[2]][m];
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            missing = missing || leaf[r] == -1;
            if (leaf[r] < 0) continue;
            const auto f = V::load(field, leaf[r]);
            s0 += wt[r] * f.x;
            s1 += wt[r] * f.y;
            s2 += wt[r] * f.z;
            if (ch + 8 * r == 13) host = leaf[r];  // the middle cell
        }
    } else {
        int leaf[8];  // by e = ex + 2 ey + 4 ez: the cell's block, -1 when missing, -2 past the stencil
        const int k0 = b0[0] + 3 * b0[1] + 9 * b0[2];
        // the table's row starts one block before the middle one
        const int pm = W == 4 ? (int)bits & 7 : 0;
        const int kr = k0 + 13 - (pm & 1) - 3 * ((pm >> 1) & 1) - 9 * (pm >> 2);
        const int* __restrict__ rp = t.pnbr + 32 * (size_t)max(row, 0) + kr;
        const int* sp = sg.blk[lane >> 3] + k0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int ex = e & 1, ey = (e >> 1) & 1, ez = e >> 2;
            const bool in = ok && (!ex || two[0]) && (!ey || two[1]) && (!ez || two[2]);
            leaf[e] = !in ? -2 : row >= 0 ? __ldg(rp + ex + 3 * ey + 9 * ez) : sp[ex + 3 * ey + 9 * ez];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            missing = missing || leaf[e] == -1;
            if (leaf[e] < 0) continue;
            const int at = leaf[e] + ch;
            const auto f = V::load(field, at);
            const T wt = w[0][e & 1] * w[1][(e >> 1) & 1] * w[2][e >> 2];
            s0 += wt * f.x;
            s1 += wt * f.y;
            s2 += wt * f.z;
            if (e == eh) host = at;
        }
    }
    if (missing) atomicOr(t.err, (unsigned)OT_DEV_STENCIL);
    // the 8 lanes' sums, by pairs: after each exchange a lane goes on with its half of the components (4
    // additions per lane instead of 9, in the same order)
    T v = (ch & 1) ? s1 : s0;
    v += __shfl_xor_sync(FULLM, (ch & 1) ? s0 : s1, 1);
    s2 += __shfl_xor_sync(FULLM, s2, 1);
    const T give = (ch & 2) ? v : s2;
    v = (ch & 2) ? s2 : v;
    v += __shfl_xor_sync(FULLM, give, 2);
    v += __shfl_xor_sync(FULLM, v, 4);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) host = max(host, __shfl_xor_sync(FULLM, host, o));
    out = ok ? v : qnan<T>();
    return host;
}

// Markers base .. end - 1 (at most n, at most 32) of a group (warp-wide call).
template <typename T, int K, bool LEARNED>
__device__ __forceinline__ void delta_markers(const TreeView& t, const T* __restrict__ field, DeltaStage<T>& sg,
                                              const double* __restrict__ x, const double* __restrict__ y,
                                              const double* __restrict__ z, int64_t n, int64_t base, int64_t end,
                                              T* __restrict__ u, int32_t* __restrict__ host) {
    const int lane = threadIdx.x & 31, ch = lane & 7;
    if (end > n) end = n;
    const int64_t mine = base + lane;
    double px = 0.0, py = 0.0, pz = 0.0;
    if (mine < end) px = x[mine], py = y[mine], pz = z[mine];
    delta_stage<T, K, LEARNED>(t, sg, mine < end, px, py, pz);
    __syncwarp();
    if constexpr (sizeof(T) == 8) {
        stage_weights<K>(sg, (int)(end - base));
        __syncwarp();
    }
    const bool ok = (sg.bits[lane] >> 16) & 1u;
    if (mine < end && !ok) atomicOr(t.err, (unsigned)OT_DEV_OUTSIDE);
    for (int64_t b = base; b < end; b += 4) {  // warp-uniform
        const int m = (int)(b - base) + (lane >> 3);
        T o;
        const int h = delta_sum<T, K, LEARNED>(t, field, sg, m, o);
        // results in the place of the marker's weights and row, stored by all lanes together below
        if (ch < 3) sg.w[ch][m] = o;
        if (ch == 3) sg.row[m] = h;
        __syncwarp();
    }
    if (mine < end) {
#pragma unroll
        for (int d = 0; d < 3; ++d) u[d * n + mine] = sg.w[d][lane];
        if (host) {
            int h = sg.row[lane];
            uint64_t X[3];
            if (ok && h < 0 && fixpoint3(px, py, pz, X))  // the finest cell that holds it is not a leaf
                h = search_plain(t, morton3((uint32_t)(X[0] >> 32), (uint32_t)(X[1] >> 32), (uint32_t)(X[2] >> 32)));
            host[mine] = h;
        }
    }
    __syncwarp();
}

} // namespace ot
