// ot_build.cu -- octree construction on the device, leaf validation, centres, level map.
//
// Construction (Sec. 3.1 refinement + 2:1 balance, Sec. 3.3 surface-driven auxiliary forest)
// works on per-level sorted key arrays R[l] of the REFINED cells of level l (3l-bit keys):
//   1. top-down: R[lmin] = cells of level lmin meeting the criterion; R[l+1] = children of
//      R[l] meeting it;
//   2. balance, finest level first: a refined cell p of level l needs every neighbour cell
//      of level l to exist, i.e. the parents of p's neighbours (and p's own parent) must be
//      refined; missing ones are added to R[l-1].  Requirements only flow to coarser levels,
//      so one descending pass reaches the fixed point (the coarsest balanced refinement);
//   3. leaves: nodes of level l+1 are the children of R[l] (already Morton-sorted); subtree
//      leaf counts bottom-up and offsets top-down place every leaf at its rank without a
//      global sort.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

#include "ot_internal.h"

namespace ot {

namespace {

unsigned grid1d(int64_t n, int block) {
    int64_t g = (n + block - 1) / block;
    int64_t cap = (int64_t)num_sms() * 16;
    return (unsigned)std::max<int64_t>(1, std::min(g, cap));
}

#define GRID_STRIDE(i, n) \
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

// The refinement test in FP64 with every operation rounded as written (no fused multiply-add),
// in x, y, z order: max(0, |c - box|_near - r, r - |c - box|_far) <= shell.
__device__ bool box_near_surface(const double lo[3], double h, const ot_sphere& s) {
    double near2 = 0.0, far2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double c = s.c[d];
        const double hi = __dadd_rn(lo[d], h);
        const double below = __dsub_rn(lo[d], c);
        const double above = __dsub_rn(c, hi);
        double e = 0.0;
        if (below > e) e = below;
        if (above > e) e = above;
        near2 = __dadd_rn(near2, __dmul_rn(e, e));
        const double f0 = fabs(__dsub_rn(c, lo[d]));
        const double f1 = fabs(__dsub_rn(c, hi));
        const double f = f0 > f1 ? f0 : f1;
        far2 = __dadd_rn(far2, __dmul_rn(f, f));
    }
    double dist = 0.0;
    const double t0 = __dsub_rn(__dsqrt_rn(near2), s.r);
    const double t1 = __dsub_rn(s.r, __dsqrt_rn(far2));
    if (t0 > dist) dist = t0;
    if (t1 > dist) dist = t1;
    return dist <= s.shell;
}

// The same test in FP32: 1 or -1 when its distance is farther from the shell width than the
// rounding can have moved it, 0 when the FP64 test has to decide (a few cells in a thousand; the
// FP64 pipe was most of the refinement's time, 497 -> 154 us for 17.3M leaves).  Rounding: positions,
// radii and distances carry at most 2^-23 of the magnitudes involved each, some 6 of them; the
// margin is 4e-6 of their sum.  Centres whose squared distances overflow FP32 (from 1.8e19 on) are
// left to FP64 too.
__device__ __forceinline__ int near_surface_f32(const float lo[3], float h, const ot_sphere& s) {
    float near2 = 0.0f, far2 = 0.0f, mag = 1.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float c = (float)s.c[k], below = lo[k] - c, above = c - (lo[k] + h);
        const float e = fmaxf(fmaxf(below, above), 0.0f), f = fmaxf(fabsf(below), fabsf(above));
        near2 += e * e;
        far2 += f * f;
        mag += fabsf(c);
    }
    const float r = (float)s.r, w = (float)s.shell;
    const float dist = fmaxf(fmaxf(sqrtf(near2) - r, r - sqrtf(far2)), 0.0f);
    const float margin = 4e-6f * (mag + r + w);
    if (!(near2 <= FLT_MAX && far2 <= FLT_MAX)) return 0;
    return dist > w + margin ? -1 : dist < w - margin ? 1 : 0;
}

// Candidate cells of level l: the 8^l cells (parent == null, l == lmin) or the children of the
// refined parents; flag[j] = criterion, cand[j] = key.  With the sphere bins (l >= Lb), only the
// spheres listed for the cell's bin of level Lb are tested: a bin lists every sphere whose
// centre is within (r + shell) + margin of it, a superset of those near any cell inside it, so the
// result is the same as testing every sphere.
__global__ void k_refine(const uint64_t* __restrict__ parent, int64_t ncand, int l, const ot_sphere* __restrict__ sph,
                         int nsph, const int* __restrict__ bin_off, const int* __restrict__ bin_sph, int Lb,
                         uint64_t* __restrict__ cand, uint32_t* __restrict__ flag) {
    const double h = ldexp(1.0, -l);
    const float hf = (float)h;
    const bool binned = bin_off && l >= Lb;
    GRID_STRIDE(j, ncand) {
        uint64_t key = parent ? ((parent[j >> 3] << 3) | (uint64_t)(j & 7)) : (uint64_t)j;
        uint32_t i0, i1, i2;
        demorton3(key, i0, i1, i2);
        const double lo[3] = {__dmul_rn((double)i0, h), __dmul_rn((double)i1, h), __dmul_rn((double)i2, h)};
        const float lof[3] = {(float)lo[0], (float)lo[1], (float)lo[2]};
        uint32_t hit = 0;
        if (binned) {
            const int sh = l - Lb, nb = 1 << Lb;
            const int b = (int)(i0 >> sh) + nb * ((int)(i1 >> sh) + nb * (int)(i2 >> sh));
            for (int k = bin_off[b]; k < bin_off[b + 1] && !hit; ++k) {
                const ot_sphere sp = sph[bin_sph[k]];
                const int sure = near_surface_f32(lof, hf, sp);
                if (sure > 0 || (sure == 0 && box_near_surface(lo, h, sp))) hit = 1;
            }
        } else {
            for (int s = 0; s < nsph && !hit; ++s) {
                const ot_sphere sp = sph[s];
                const int sure = near_surface_f32(lof, hf, sp);
                if (sure > 0 || (sure == 0 && box_near_surface(lo, h, sp))) hit = 1;
            }
        }
        cand[j] = key;
        flag[j] = hit;
    }
}

// A sorted set of keys of one level, with the places of its first keys per bucket of leading bits
// (tab[b] .. tab[b + 1], null: none).  A search is a chain of dependent loads, some 20 in the sets of
// a large tree; the table leaves some 7: ranks 114 -> 52 us, balance 410 -> 270 us, the tables 61 us
// (17.3M leaves).
struct KeySet {
    const uint64_t* a;
    int64_t n;
    const uint32_t* tab;
    int sh;
};
__device__ __forceinline__ int64_t lower_bound(const uint64_t* __restrict__ a, int64_t lo, int64_t hi, uint64_t q) {
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (a[mid] < q)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}
__device__ __forceinline__ bool contains_sorted(const KeySet& s, uint64_t q, int64_t* at) {
    const uint64_t b = q >> s.sh;
    const int64_t lo = lower_bound(s.a, s.tab ? s.tab[b] : 0, s.tab ? s.tab[b + 1] : s.n, q);
    if (at) *at = lo;
    return lo < s.n && s.a[lo] == q;
}
__global__ void k_buckets(const uint64_t* __restrict__ a, int64_t n, int sh, int64_t nb, uint32_t* __restrict__ tab) {
    GRID_STRIDE(b, nb + 1) tab[b] = (uint32_t)(b < nb ? lower_bound(a, 0, n, (uint64_t)b << sh) : n);
}

// Balance requirement of refined cells p of level l: the parents (level l-1) of p's neighbour
// cells and of p itself must be refined: its own parent and per axis the next one on the side that p
// lies at.  Missing ones are appended to `miss`, those of a warp once each (siblings miss
// the same parents) and those of a block with one addition to their count: the additions, one per key,
// were most of the rest of its time (17.3M leaves 270 -> 170 us).
constexpr int BAL_T = 256;
__global__ void __launch_bounds__(BAL_T) k_balance_req(const uint64_t* __restrict__ R, int64_t nR, int l, KeySet Rp, int full,
                              uint64_t* __restrict__ miss, uint32_t* __restrict__ nmiss, int64_t cap) {
    constexpr unsigned FULLM = 0xffffffffu;
    const uint32_t np = 1u << (l - 1);  // parents per axis
    __shared__ uint32_t s_cnt[BAL_T / 32], s_at;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t j0 = blockIdx.x * (int64_t)BAL_T; j0 < nR; j0 += (int64_t)gridDim.x * BAL_T) {
        const int64_t j = j0 + threadIdx.x;
        const bool in = j < nR;
        uint32_t c[3];
        demorton3(in ? R[j] : 0ULL, c[0], c[1], c[2]);
        uint64_t dil[3][2];
        unsigned there = 0;  // bit d: axis d has the other parent
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const uint32_t own = c[d] >> 1, other = (c[d] & 1u) ? own + 1u : own - 1u;  // (0 - 1 is not below np)
            if (other < np) there |= 1u << d;
            dil[d][0] = part1by2(own) << d;
            dil[d][1] = part1by2(other & (np - 1u)) << d;
        }
        // the 8 searches step by step together: their loads do not wait for one another
        uint64_t key[8];
        uint32_t lo[8], len[8], most = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            // face balance: p's own parent, or the parent of a face neighbour
            const bool want = in && !(e & ~there) && (full || !(e & (e - 1)));
            key[e] = dil[0][e & 1] | dil[1][(e >> 1) & 1] | dil[2][e >> 2];
            const uint64_t b = key[e] >> Rp.sh;
            lo[e] = !want || !Rp.tab ? 0u : Rp.tab[b];
            len[e] = !want ? 0u : (Rp.tab ? Rp.tab[b + 1] : (uint32_t)Rp.n) - lo[e];
            if (!want) key[e] = ~0ULL;
            most = max(most, len[e]);
        }
        for (; most > 1u; most -= most >> 1) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint32_t half = len[e] >> 1;
                if (half && Rp.a[lo[e] + half] <= key[e]) lo[e] += half;
                len[e] -= half;
            }
        }
        uint32_t mine = 0;  // bit e: this lane appends key e
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const bool missing = key[e] != ~0ULL && !(len[e] && Rp.a[lo[e]] == key[e]);
            if (!__any_sync(FULLM, missing)) continue;
            const unsigned same = __match_any_sync(FULLM, missing ? key[e] : ~0ULL);
            if (missing && !(same & ((1u << lane) - 1u))) mine |= 1u << e;
        }
        uint32_t incl = (uint32_t)__popc(mine);
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
            const uint32_t v = __shfl_up_sync(FULLM, incl, k);
            if (lane >= k) incl += v;
        }
        if (lane == 31) s_cnt[warp] = incl;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t all = 0;
            for (int w = 0; w < BAL_T / 32; ++w) all += s_cnt[w];
            s_at = all ? atomicAdd(nmiss, all) : 0u;
        }
        __syncthreads();
        uint32_t at = s_at + incl - (uint32_t)__popc(mine);
        for (int w = 0; w < warp; ++w) at += s_cnt[w];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if ((mine >> e) & 1u) {
                if (at < cap) miss[at] = key[e];
                ++at;
            }
        __syncthreads();  // s_cnt, s_at
    }
}

__device__ __forceinline__ uint64_t node_key(const uint64_t* __restrict__ Rparent, int64_t j) {
    return Rparent ? ((Rparent[j >> 3] << 3) | (uint64_t)(j & 7)) : (uint64_t)j;
}

__global__ void k_rank(const uint64_t* __restrict__ Rparent, int64_t M, KeySet R, int32_t* __restrict__ rank) {
    GRID_STRIDE(j, M) {
        int64_t at;
        rank[j] = contains_sorted(R, node_key(Rparent, j), &at) ? (int32_t)at : -1;
    }
}

__global__ void k_count(const int32_t* __restrict__ rank, int64_t M, const uint32_t* __restrict__ cnt_child,
                        uint32_t* __restrict__ cnt) {
    GRID_STRIDE(j, M) {
        int32_t r = rank[j];
        if (r < 0) {
            cnt[j] = 1;
        } else if (!cnt_child) {
            cnt[j] = 8;
        } else {
            uint32_t s = 0;
            for (int c = 0; c < 8; ++c) s += cnt_child[8 * (int64_t)r + c];
            cnt[j] = s;
        }
    }
}

__global__ void k_child_off(const int32_t* __restrict__ rank, const uint32_t* __restrict__ off, int64_t M,
                            const uint32_t* __restrict__ cnt_child, uint32_t* __restrict__ off_child) {
    GRID_STRIDE(j, M) {
        int32_t r = rank[j];
        if (r < 0) continue;
        uint32_t run = off[j];
        for (int c = 0; c < 8; ++c) {
            off_child[8 * (int64_t)r + c] = run;
            run += cnt_child ? cnt_child[8 * (int64_t)r + c] : 1u;
        }
    }
}

__global__ void k_emit(const uint64_t* __restrict__ Rparent, const int32_t* __restrict__ rank,
                       const uint32_t* __restrict__ off, int64_t M, int l, uint64_t* __restrict__ key_out,
                       uint8_t* __restrict__ lev_out) {
    GRID_STRIDE(j, M) {
        if (rank && rank[j] >= 0) continue;
        uint32_t o = off[j];
        key_out[o] = node_key(Rparent, j) << (3 * (MAXLEVEL - l));
        lev_out[o] = (uint8_t)l;
    }
}

template <typename T>
ot_status dalloc(T** p, int64_t n, cudaStream_t s) {
    *p = nullptr;
    if (n <= 0) return OT_OK;
    OT_CUDA(pool_malloc((void**)p, sizeof(T) * (size_t)n, s));
    return OT_OK;
}

// The set of the n sorted keys a of level l.  A bucket per key at most, tab has room for 2^MAX_BUCKET
// + 1; few keys go without.
constexpr int MAX_BUCKET = 18;
KeySet key_set(const uint64_t* a, int64_t n, int l, uint32_t* tab, cudaStream_t s) {
    int bits = std::min(3 * l, MAX_BUCKET);
    while (bits > 0 && ((int64_t)1 << bits) > n) --bits;
    if (bits < 10) return KeySet{a, n, nullptr, 0};
    const int64_t nb = (int64_t)1 << bits;
    k_buckets<<<grid1d(nb + 1, 256), 256, 0, s>>>(a, n, 3 * l - bits, nb, tab);
    count_launch();
    return KeySet{a, n, tab, 3 * l - bits};
}

struct Guard {
    cudaStream_t s;
    std::vector<void*> ptrs;
    ~Guard() {
        for (void* p : ptrs)
            if (p) cudaFreeAsync(p, s);
    }
    template <typename T> T* keep(T* p) {
        ptrs.push_back((void*)p);
        return p;
    }
};

} // namespace

ot_status build_tree(const ot_sphere* h_spheres, int nsph, const ot_build_params* p, cudaStream_t s, ot_octree* t) {
    const int lmin = p->lmin, lmax = p->lmax;
    Guard g{s, {}};
    ot_sphere* d_sph = nullptr;
    if (nsph > 0) {
        OT_CUDA(pool_malloc((void**)&d_sph, sizeof(ot_sphere) * nsph, s));
        g.keep(d_sph);
        OT_CUDA(cudaMemcpyAsync(d_sph, h_spheres, sizeof(ot_sphere) * nsph, cudaMemcpyHostToDevice, s));
    }
    // sphere bins: the cells of level Lb, each listing the spheres whose centre lies within
    // (r + shell) (1 + 1e-4) + 1e-4 of the bin's box (bounding-box overlap; a superset)
    const int Lb = std::min(lmin, 5);
    int* d_bin_off = nullptr;
    int* d_bin_sph = nullptr;
    if (nsph > 0 && Lb >= 1) {
        const int nb = 1 << Lb;
        std::vector<std::vector<int>> bins((size_t)nb * nb * nb);
        for (int k = 0; k < nsph; ++k) {
            const ot_sphere& sp = h_spheres[k];
            const double R = (sp.r + sp.shell) * 1.0001 + 1e-4;
            int lo[3], hi[3];
            const auto bin_of = [nb](double v) {  // clamped in FP64 before the conversion
                return (int)std::floor(std::max(0.0, std::min((double)(nb - 1), v * nb)));
            };
            for (int d = 0; d < 3; ++d) {
                lo[d] = bin_of(sp.c[d] - R);
                hi[d] = bin_of(sp.c[d] + R);
            }
            for (int z = lo[2]; z <= hi[2]; ++z)
                for (int y = lo[1]; y <= hi[1]; ++y)
                    for (int x = lo[0]; x <= hi[0]; ++x) bins[(size_t)x + nb * ((size_t)y + nb * (size_t)z)].push_back(k);
        }
        std::vector<int> off(bins.size() + 1, 0), idx;
        for (size_t b = 0; b < bins.size(); ++b) {
            off[b + 1] = off[b] + (int)bins[b].size();
            idx.insert(idx.end(), bins[b].begin(), bins[b].end());
        }
        OT_CUDA(pool_malloc((void**)&d_bin_off, sizeof(int) * off.size(), s));
        g.keep(d_bin_off);
        OT_CUDA(pool_malloc((void**)&d_bin_sph, sizeof(int) * std::max<size_t>(idx.size(), 1), s));
        g.keep(d_bin_sph);
        OT_CUDA(cudaMemcpyAsync(d_bin_off, off.data(), sizeof(int) * off.size(), cudaMemcpyHostToDevice, s));
        if (!idx.empty())
            OT_CUDA(cudaMemcpyAsync(d_bin_sph, idx.data(), sizeof(int) * idx.size(), cudaMemcpyHostToDevice, s));
        OT_CUDA(cudaStreamSynchronize(s));  // the host vectors go out of scope
    }
    const int L = lmax + 1;
    std::vector<uint64_t*> R(L, nullptr);
    std::vector<int64_t> nR(L, 0);

    // 1. top-down refinement by the criterion
    for (int l = lmin; l < lmax; ++l) {
        const int64_t ncand = (l == lmin) ? ((int64_t)1 << (3 * lmin)) : 8 * nR[l - 1];
        if (ncand == 0) break;
        uint64_t* cand = nullptr;
        uint32_t* flag = nullptr;
        ot_status st;
        if ((st = dalloc(&cand, ncand, s)) != OT_OK) return st;
        g.keep(cand);
        if ((st = dalloc(&flag, ncand, s)) != OT_OK) return st;
        g.keep(flag);
        k_refine<<<grid1d(ncand, 256), 256, 0, s>>>(l == lmin ? nullptr : R[l - 1], ncand, l, d_sph, nsph, d_bin_off,
                                                    d_bin_sph, Lb, cand, flag);
        count_launch();
        OT_CUDA(cudaGetLastError());
        uint64_t* out = nullptr;
        if ((st = dalloc(&out, ncand, s)) != OT_OK) return st;
        g.keep(out);
        if ((st = compact_u64(cand, flag, ncand, out, &nR[l], s)) != OT_OK) return st;
        R[l] = out;
    }

    uint32_t* tab = nullptr;  // of the set searched next
    {
        const ot_status st = dalloc(&tab, ((int64_t)1 << MAX_BUCKET) + 1, s);
        if (st != OT_OK) return st;
    }
    g.keep(tab);

    // 2. balance, finest refined level first
    for (int l = lmax - 1; l >= lmin + 1; --l) {
        if (nR[l] == 0) continue;
        const int64_t cap = 8 * nR[l];
        uint64_t* miss = nullptr;
        uint32_t* nmiss = nullptr;
        ot_status st;
        if ((st = dalloc(&miss, cap, s)) != OT_OK) return st;
        g.keep(miss);
        if ((st = dalloc(&nmiss, 1, s)) != OT_OK) return st;
        g.keep(nmiss);
        OT_CUDA(cudaMemsetAsync(nmiss, 0, sizeof(uint32_t), s));
        const KeySet parents = key_set(R[l - 1], nR[l - 1], l - 1, tab, s);
        k_balance_req<<<grid1d(nR[l], BAL_T), BAL_T, 0, s>>>(R[l], nR[l], l, parents, p->balance_full, miss, nmiss, cap);
        count_launch();
        OT_CUDA(cudaGetLastError());
        uint32_t hm = 0;
        OT_CUDA(cudaMemcpyAsync(&hm, nmiss, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
        OT_CUDA(cudaStreamSynchronize(s));
        if (hm > 0) {
            const int64_t tot = nR[l - 1] + hm;
            uint64_t *u = nullptr, *tmp = nullptr;
            if ((st = dalloc(&u, tot, s)) != OT_OK) return st;
            g.keep(u);
            if ((st = dalloc(&tmp, tot, s)) != OT_OK) return st;
            g.keep(tmp);
            if (nR[l - 1] > 0)
                OT_CUDA(cudaMemcpyAsync(u, R[l - 1], sizeof(uint64_t) * nR[l - 1], cudaMemcpyDeviceToDevice, s));
            OT_CUDA(cudaMemcpyAsync(u + nR[l - 1], miss, sizeof(uint64_t) * hm, cudaMemcpyDeviceToDevice, s));
            if ((st = radix_sort_u64(u, tmp, tot, 0, 3 * (l - 1), s)) != OT_OK) return st;
            int64_t m = 0;
            if ((st = unique_u64(u, tot, tmp, &m, s)) != OT_OK) return st;
            R[l - 1] = tmp;
            nR[l - 1] = m;
        }
    }

    // 3. leaves: ranks, subtree counts (bottom-up), offsets (top-down), emission
    std::vector<int64_t> M(L + 1, 0);
    std::vector<int32_t*> rank(L + 1, nullptr);
    std::vector<uint32_t*> cnt(L + 1, nullptr), off(L + 1, nullptr);
    M[lmin] = (int64_t)1 << (3 * lmin);
    for (int l = lmin; l < lmax; ++l) M[l + 1] = 8 * nR[l];
    ot_status st;
    for (int l = lmin; l <= lmax; ++l) {
        if (M[l] == 0) continue;
        if (l < lmax) {
            if ((st = dalloc(&rank[l], M[l], s)) != OT_OK) return st;
            g.keep(rank[l]);
            const KeySet refined = key_set(R[l], nR[l], l, tab, s);
            k_rank<<<grid1d(M[l], 256), 256, 0, s>>>(l == lmin ? nullptr : R[l - 1], M[l], refined, rank[l]);
            count_launch();
        }
        if ((st = dalloc(&cnt[l], M[l], s)) != OT_OK) return st;
        g.keep(cnt[l]);
        if ((st = dalloc(&off[l], M[l], s)) != OT_OK) return st;
        g.keep(off[l]);
    }
    for (int l = lmax - 1; l >= lmin; --l) {
        if (M[l] == 0) continue;
        const uint32_t* child = (l + 1 < lmax && M[l + 1] > 0) ? cnt[l + 1] : nullptr;
        k_count<<<grid1d(M[l], 256), 256, 0, s>>>(rank[l], M[l], child, cnt[l]);
        count_launch();
    }
    uint32_t* d_tot = nullptr;
    if ((st = dalloc(&d_tot, 1, s)) != OT_OK) return st;
    g.keep(d_tot);
    if (lmin == lmax) {
        // uniform tree: every node of level lmin is a leaf
        OT_CUDA(cudaMemsetAsync(cnt[lmin], 0, sizeof(uint32_t) * M[lmin], s));
    }
    if (lmin < lmax) {
        if ((st = scan_u32(cnt[lmin], off[lmin], M[lmin], d_tot, s)) != OT_OK) return st;
    }
    for (int l = lmin; l < lmax; ++l) {
        if (M[l] == 0 || M[l + 1] == 0) continue;
        const uint32_t* child = (l + 1 < lmax) ? cnt[l + 1] : nullptr;
        k_child_off<<<grid1d(M[l], 256), 256, 0, s>>>(rank[l], off[l], M[l], child, off[l + 1]);
        count_launch();
    }
    int64_t nleaf = 0;
    if (lmin < lmax) {
        uint32_t h = 0;
        OT_CUDA(cudaMemcpyAsync(&h, d_tot, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
        OT_CUDA(cudaStreamSynchronize(s));
        nleaf = h;
    } else {
        nleaf = M[lmin];
    }
    if (nleaf <= 0 || nleaf > OT_MAX_LEAVES) return OT_ERR_LIMIT;
    OT_CUDA(pool_malloc((void**)&t->d_key, sizeof(uint64_t) * nleaf, s));
    OT_CUDA(pool_malloc((void**)&t->d_level, nleaf, s));
    for (int l = lmin; l <= lmax; ++l) {
        if (M[l] == 0) continue;
        const uint32_t* o = off[l];
        if (lmin == lmax) {
            // off = identity for a uniform tree
            std::vector<uint32_t> id(M[l]);
            for (int64_t j = 0; j < M[l]; ++j) id[j] = (uint32_t)j;
            OT_CUDA(cudaMemcpyAsync(off[l], id.data(), sizeof(uint32_t) * M[l], cudaMemcpyHostToDevice, s));
            OT_CUDA(cudaStreamSynchronize(s));
        }
        k_emit<<<grid1d(M[l], 256), 256, 0, s>>>(l == lmin ? nullptr : R[l - 1], l < lmax ? rank[l] : nullptr, o, M[l],
                                                l, t->d_key, t->d_level);
        count_launch();
    }
    OT_CUDA(cudaGetLastError());
    OT_CUDA(cudaStreamSynchronize(s));
    t->n = nleaf;
    t->lmin = lmin;
    t->lmax = lmax;
    return OT_OK;
}

// ------------------------------------------------------------------------------------------
// Validation of caller leaves.
// ------------------------------------------------------------------------------------------
namespace {

__global__ void k_check_tiling(const uint64_t* __restrict__ key, const uint8_t* __restrict__ lev, int64_t n,
                               unsigned* __restrict__ bad, int* __restrict__ lrange) {
    GRID_STRIDE(i, n) {
        int l = lev[i];
        bool ok = l <= OT_MAX_LEVEL;
        uint64_t sp = ok ? key_span(l) : 0;
        if (ok) {
            ok = (key[i] & (sp - 1)) == 0;
            if (i == 0) ok = ok && key[0] == 0;
            if (i + 1 < n)
                ok = ok && key[i] + sp == key[i + 1];
            else
                ok = ok && key[i] + sp == (1ULL << 63);
        }
        if (!ok) atomicAdd(bad, 1u);
        atomicMin(&lrange[0], l);
        atomicMax(&lrange[1], l);
    }
}

__global__ void k_check_balance(const uint64_t* __restrict__ key, const uint8_t* __restrict__ lev, int n, int full,
                                unsigned* __restrict__ bad) {
    GRID_STRIDE(b, (int64_t)n) {
        const int lb = lev[b];
        uint32_t x, y, z;
        demorton3(key[b], x, y, z);
        const int sh = MAXLEVEL - lb;
        const int64_t ci = x >> sh, cj = y >> sh, ck = z >> sh, nc = (int64_t)1 << lb;
        for (int dz = -1; dz <= 1; ++dz)
            for (int dy = -1; dy <= 1; ++dy)
                for (int dx = -1; dx <= 1; ++dx) {
                    int nz = (dx != 0) + (dy != 0) + (dz != 0);
                    if (nz == 0 || (!full && nz != 1)) continue;
                    int64_t a = ci + dx, bq = cj + dy, c = ck + dz;
                    if (a < 0 || bq < 0 || c < 0 || a >= nc || bq >= nc || c >= nc) continue;
                    uint64_t q = morton3((uint32_t)(a << sh), (uint32_t)(bq << sh), (uint32_t)(c << sh));
                    int at = search_range(key, 0, n, q);
                    if ((int)lev[at] + 2 <= lb) atomicAdd(bad, 1u);
                }
    }
}

} // namespace

ot_status validate_leaves(const uint64_t* d_key, const uint8_t* d_level, int64_t n, int full, cudaStream_t s, int* lmin,
                          int* lmax) {
    unsigned* bad = nullptr;  // two counts, then the level range
    Guard g{s, {}};
    OT_CUDA(pool_malloc((void**)&bad, 2 * sizeof(unsigned) + 2 * sizeof(int), s));
    g.keep(bad);
    int* lr = reinterpret_cast<int*>(bad + 2);
    int init[2] = {1 << 20, -1};
    OT_CUDA(cudaMemsetAsync(bad, 0, 2 * sizeof(unsigned), s));
    OT_CUDA(cudaMemcpyAsync(lr, init, sizeof(init), cudaMemcpyHostToDevice, s));
    k_check_tiling<<<grid1d(n, 256), 256, 0, s>>>(d_key, d_level, n, bad, lr);
    count_launch();
    unsigned hb[2] = {0, 0};
    int hr[2];
    OT_CUDA(cudaMemcpyAsync(hb, bad, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    OT_CUDA(cudaMemcpyAsync(hr, lr, sizeof(hr), cudaMemcpyDeviceToHost, s));
    OT_CUDA(cudaStreamSynchronize(s));
    ot_status st = OT_OK;
    if (hb[0] != 0) {
        st = OT_ERR_UNSORTED;
    } else {
        k_check_balance<<<grid1d(n, 256), 256, 0, s>>>(d_key, d_level, (int)n, full, bad + 1);
        count_launch();
        OT_CUDA(cudaMemcpyAsync(hb + 1, bad + 1, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
        OT_CUDA(cudaStreamSynchronize(s));
        if (hb[1] != 0) st = OT_ERR_UNBALANCED;
    }
    *lmin = hr[0];
    *lmax = hr[1];
    OT_CUDA(cudaGetLastError());
    return st;
}

// ------------------------------------------------------------------------------------------
// Centres, search sample, diagnostics words.
// ------------------------------------------------------------------------------------------
namespace {

__global__ void k_centres(const uint64_t* __restrict__ key, const uint8_t* __restrict__ lev, int64_t n,
                          double* __restrict__ out) {
    GRID_STRIDE(i, n) {
        uint32_t x, y, z;
        demorton3(key[i], x, y, z);
        const double half = 0.5 * (double)(1u << (MAXLEVEL - lev[i]));
        const double sc = 0x1p-21;
        out[i] = ((double)x + half) * sc;
        out[n + i] = ((double)y + half) * sc;
        out[2 * n + i] = ((double)z + half) * sc;
    }
}

// lmap[c] = the leaf holding the anchor of level-L cell c: the last key <= its anchor.
__global__ void k_lmap(const uint64_t* __restrict__ key, int n, int L, int64_t ncell, uint32_t* __restrict__ out) {
    GRID_STRIDE(c, ncell) out[c] = (uint32_t)search_range(key, 0, n, (uint64_t)c << (3 * (MAXLEVEL - L)));
}

} // namespace

ot_status leaf_centres(const ot_octree* t, double* d_xyz, cudaStream_t s) {
    k_centres<<<grid1d(t->n, 256), 256, 0, s>>>(t->d_key, t->d_level, t->n, d_xyz);
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

// Descriptors of the level-map cells of level L (see desc_resolve): first leaf and, where it covers
// the cell, its level; then every leaf below a cell that is the first of its child or grandchild
// adds its bit (a thread per leaf: one per cell would walk up to 8^3 leaves in turn).
__global__ void k_desc_cells(const uint8_t* __restrict__ level, int n, const uint32_t* __restrict__ lmap, int64_t ncell,
                             uint4* __restrict__ desc) {
    GRID_STRIDE(c, ncell) {
        const int a = (int)lmap[c];
        const int e = c + 1 < ncell ? (int)lmap[c + 1] : n;
        // a refined cell holds at least 8 leaves, the first starting at its anchor
        desc[c] = make_uint4(0u, 0u, e - a <= 1 ? DESC_COVERED | ((uint32_t)level[a] << 16) : 0u, (uint32_t)a);
    }
}
__global__ void k_desc_leaves(const uint64_t* __restrict__ key, const uint8_t* __restrict__ level, int n, int L,
                              uint32_t* __restrict__ desc) {
    GRID_STRIDE(i, (int64_t)n) {
        const int l = level[i];
        if (l < L + 2) continue;
        const uint64_t k = key[i];
        uint32_t* d = desc + 4 * (size_t)(k >> (3 * (MAXLEVEL - L)));
        const int c1 = (int)(k >> (3 * (MAXLEVEL - L - 1))) & 7, c2 = (int)(k >> (3 * (MAXLEVEL - L - 2))) & 7;
        if ((k & (key_span(L + 1) - 1)) == 0) atomicOr(d + 2, 1u << c1);
        if (l >= L + 3 && (k & (key_span(L + 2) - 1)) == 0) atomicOr(d + (c1 >> 2), 1u << (8 * (c1 & 3) + c2));
        if (l > L + 3 && (k & (key_span(L + 3) - 1)) == 0) atomicOr(d + 2, DESC_DEEP);
    }
}

ot_status finish_tree(ot_octree* t, cudaStream_t s, int map_level) {
    // default: level 7, or 8 for trees deeper than 10 levels (the descriptors then reach lmax)
    const int L = map_level >= 0 ? std::min(map_level, t->lmax)
                                 : std::min(t->lmax, std::max(7, std::min(8, t->lmax - 3)));
    const int Lp = std::min(t->lmax, 7);
    if (!t->d_pmap) {
        const int64_t np = (int64_t)1 << (3 * Lp);
        OT_CUDA(pool_malloc((void**)&t->d_pmap, sizeof(uint32_t) * np, s));
        k_lmap<<<grid1d(np, 256), 256, 0, s>>>(t->d_key, (int)t->n, Lp, np, t->d_pmap);
        count_launch();
        t->pyr_level = Lp;
        ot_status st = build_node_lists(t, s);
        if (st != OT_OK) return st;
    }
    // the new map beside the old one, which stays in place when there is no memory for another
    const int64_t ncell = (int64_t)1 << (3 * L);
    uint32_t* lmap = t->d_pmap;
    uint4* desc = nullptr;
    auto fail = [&](cudaError_t e) {
        if (lmap && lmap != t->d_pmap) cudaFreeAsync(lmap, s);
        if (desc) cudaFreeAsync(desc, s);
        return cuda_status(e);
    };
    cudaError_t e;
    if (L != Lp) {
        if ((e = pool_malloc((void**)&lmap, sizeof(uint32_t) * ncell, s)) != cudaSuccess) return fail(e);
        k_lmap<<<grid1d(ncell, 256), 256, 0, s>>>(t->d_key, (int)t->n, L, ncell, lmap);
        count_launch();
    }
    if ((e = pool_malloc((void**)&desc, sizeof(uint4) * ncell, s)) != cudaSuccess) return fail(e);
    k_desc_cells<<<grid1d(ncell, 256), 256, 0, s>>>(t->d_level, (int)t->n, lmap, ncell, desc);
    count_launch();
    if (L + 2 <= t->lmax) {
        k_desc_leaves<<<grid1d(t->n, 256), 256, 0, s>>>(t->d_key, t->d_level, (int)t->n, L,
                                                       reinterpret_cast<uint32_t*>(desc));
        count_launch();
    }
    if (!t->d_err) {
        if ((e = pool_malloc((void**)&t->d_err, 64, s)) != cudaSuccess) return fail(e);
        if ((e = cudaMemsetAsync(t->d_err, 0, 64, s)) != cudaSuccess) return fail(e);
        t->d_fallbacks = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(t->d_err) + 8);
    }
    if ((e = cudaGetLastError()) != cudaSuccess || (e = cudaStreamSynchronize(s)) != cudaSuccess) return fail(e);
    // (a change of the map level: work on other streams may still read the old map)
    if (t->d_desc && !wait_device(t->device)) return fail(cudaErrorUnknown);
    if (t->d_lmap && t->d_lmap != t->d_pmap) cudaFree(t->d_lmap);
    if (t->d_desc) cudaFree(t->d_desc);
    t->d_lmap = lmap;
    t->d_desc = desc;
    t->lmap_level = L;
    return OT_OK;
}

TreeView tree_view(const ot_octree* t) {
    TreeView v{};
    v.key = t->d_key;
    v.level = t->d_level;
    v.n = (int)t->n;
    v.lmin = t->lmin;
    v.lmax = t->lmax;
    v.lmap = t->d_lmap;
    v.lmap_level = t->lmap_level;
    v.desc = t->d_desc;
    v.pyr_level = t->pyr_level;
    v.periodic = t->periodic;
    v.mates = reinterpret_cast<const uint4*>(t->d_mates);
    v.pnbr = (t->d_mates && t->lmax >= 1)
                 ? reinterpret_cast<const int*>(reinterpret_cast<const char*>(t->d_mates) + (size_t)256 * t->n)
                 : nullptr;
    v.root = t->d_root;
    v.models = t->d_models;
    v.mids = t->d_mids;
    v.n_leaf = t->n_models;
    v.err = t->d_err;
    v.fallbacks = t->d_fallbacks;
    return v;
}

} // namespace ot
