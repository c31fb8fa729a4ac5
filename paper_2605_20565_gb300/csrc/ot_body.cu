// ot_body.cu -- per-body linear and angular sums of a marker quantity (Sec. 2.3, rigid bodies):
//   lin_b = scale sum_{k in b} v_k w_k,   ang_b = scale sum_{k in b} (X_k - x_b) x v_k w_k.
// With v the velocity interpolated at the internal markers and scale = rho_f these are the
// internal fluid's linear and angular momenta P and L; with v = F_k at the surface markers and
// scale = -1, the IBM force and torque.  Accumulation to FP64 precision or better in a fixed order
// (thread-strided, then a fixed tree over the threads and blocks of a body): bit-identical from run
// to run.
#include <cooperative_groups.h>

#include "ot_internal.h"
#include "ot_sum.cuh"

namespace ot {

namespace {

namespace cg = cooperative_groups;

constexpr int BT = 256;

// x 2^62 as an integer (what lies below 2^-62 cut off: possible below 2^-9, noted in cut), or false
// for |x| >= 1 and NaN.
__device__ __forceinline__ bool to_fixed(double x, long long& f, bool& cut) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(u >> 52) & 0x7FF, sh = e - 1013;
    const unsigned long long m = (u & 0xFFFFFFFFFFFFFULL) | (e ? 1ULL << 52 : 0ULL);
    const long long v = (long long)(sh >= 0 ? m << (sh & 15) : sh > -64 ? m >> -sh : 0ULL);
    f = (u >> 63) ? -v : v;
    cut = sh < 0 && m != 0ULL;
    return e < 1023;
}
// g - f carries FP64's precision: nothing was cut, or no more than 2^-53 of it.
__device__ __forceinline__ bool precise(long long g, long long f, bool cut) {
    return !cut || (unsigned long long)(g - f) + (1ULL << 54) >= 1ULL << 55;
}
// An integer of up to 22 bits and a sign to float by its bits (no conversion instruction).
__device__ __forceinline__ float small_int(int c) { return __fsub_rn(__int_as_float(0x4B400000 + c), 12582912.0f); }
// r 2^-62 in three floats of 21 bits each, the largest first: exact.
__device__ __forceinline__ void to_limbs(long long r, float l[3]) {
    const int c0 = (int)((unsigned)r << 11) >> 11;
    const long long r1 = (r - c0) >> 21;
    const int c1 = (int)((unsigned)r1 << 11) >> 11;
    l[0] = small_int((int)((r1 - c1) >> 21)) * 0x1p-20f;
    l[1] = small_int(c1) * 0x1p-41f;
    l[2] = small_int(c0) * 0x1p-62f;
}
// s += r v, r in limbs: the products' rounding errors (fused multiply-add) are added too, down to 2^-64
// of the product.
__device__ __forceinline__ void add_product(Sum3& s, const float r[3], float v) {
    const float p = __fmul_rn(r[0], v), q = __fmul_rn(r[1], v);
    s.add(p);
    s.low(__fmaf_rn(r[0], v, -p));
    s.low(q);
    s.last(__fmaf_rn(r[2], v, __fmaf_rn(r[1], v, -q)));
}
// The same for v some 2^-24 below the other terms.
__device__ __forceinline__ void add_small_product(Sum3& s, const float r[3], float v) {
    const float p = __fmul_rn(r[0], v);
    s.low(p);
    s.last(__fmaf_rn(r[1], v, __fmaf_rn(r[0], v, -p)));
}

// One thread-block cluster per body; its blocks share the body's markers and the first adds the
// blocks' partial sums in rank order from their shared memory (there is no workspace to keep them
// in, and atomics would leave the order open).
// The FP64 pipe bounded it (12 operations per marker, 418 us for 7.5M markers and 130 us for 2M with
// volumes, on all SMs), so a thread's sums are kept in three floats each: X - x_b is formed in
// integers at 2^-62, cut into three floats, and the products and their rounding errors are added
// up (some 300 FP32 and integer instructions: 315 and 93 us).  That carries more bits than FP64 does;
// markers with a coordinate of 1 or more, closer to their body's centre than the cut at 2^-62
// allows, or with a value that floats cannot multiply exactly (below 2^-40, above 2^74, not
// finite) are summed in FP64.
// DV: marker volumes given.  MINB: blocks per SM that the registers allow.
template <bool DV, int MINB>
__global__ void __launch_bounds__(BT, MINB) k_body_sums(const double* __restrict__ x, const double* __restrict__ y,
                                                  const double* __restrict__ z, const float* __restrict__ v,
                                                  const float* __restrict__ dV, float w, int64_t n,
                                                  const int64_t* __restrict__ start, const double* __restrict__ xb,
                                                  double scale, double* __restrict__ lin, double* __restrict__ ang) {
    __shared__ float s_float[6][BT / 32][3];
    __shared__ double s_double[6][BT / 32];
    __shared__ bool s_used[BT / 32];
    __shared__ double s_sum[6];
    cg::cluster_group cluster = cg::this_cluster();
    const int nb = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int b = blockIdx.x / nb;
    const int64_t k0 = start[b], k1 = start[b + 1];
    const double cx = xb[3 * b], cy = xb[3 * b + 1], cz = xb[3 * b + 2];
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    Sum3 sum[6];
    bool used = false;  // acc
    long long f0, f1, f2;
    bool t0, t1, t2;
    bool centre = to_fixed(cx, f0, t0);
    centre = to_fixed(cy, f1, t1) && centre;
    centre = to_fixed(cz, f2, t2) && centre;
#pragma unroll 2
    for (int64_t k = k0 + rank * BT + (int)threadIdx.x; k < k1; k += (int64_t)nb * BT) {
        const float w0 = v[k], w1 = v[n + k], w2 = v[2 * n + k], wk = DV ? dV[k] : 1.0f;
        const double X = x[k], Y = y[k], Z = z[k];
        long long g0, g1, g2;
        bool u0, u1, u2;
        bool exact = to_fixed(X, g0, u0);
        exact = to_fixed(Y, g1, u1) && exact;
        exact = to_fixed(Z, g2, u2) && exact;
        exact = exact && precise(g0, f0, t0 || u0) && precise(g1, f1, t1 || u1) && precise(g2, f2, t2 || u2);
        // with volumes the value is the product w_i wk, as its rounding p and the error q of that
        float p[3] = {w0, w1, w2}, q[3] = {0.0f, 0.0f, 0.0f};
        if (DV) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float t = __fmul_rn(p[c], wk);
                exact = exact && (t != 0.0f || p[c] == 0.0f || wk == 0.0f);  // (not a product lost below the smallest float)
                q[c] = __fmaf_rn(p[c], wk, -t);
                p[c] = t;
            }
        }
        if (exact && centre && plain(p[0]) && plain(p[1]) && plain(p[2])) {
            float r0[3], r1[3], r2[3];
            to_limbs(g0 - f0, r0);
            to_limbs(g1 - f1, r1);
            to_limbs(g2 - f2, r2);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                sum[c].add(p[c]);
                if (DV) sum[c].low(q[c]);
            }
            add_product(sum[3], r1, p[2]), add_product(sum[3], r2, -p[1]);
            add_product(sum[4], r2, p[0]), add_product(sum[4], r0, -p[2]);
            add_product(sum[5], r0, p[1]), add_product(sum[5], r1, -p[0]);
            if (DV) {
                add_small_product(sum[3], r1, q[2]), add_small_product(sum[3], r2, -q[1]);
                add_small_product(sum[4], r2, q[0]), add_small_product(sum[4], r0, -q[2]);
                add_small_product(sum[5], r0, q[1]), add_small_product(sum[5], r1, -q[0]);
            }
        } else {
            const double s0 = (double)w0 * (double)wk, s1 = (double)w1 * (double)wk, s2 = (double)w2 * (double)wk;
            const double r0 = X - cx, r1 = Y - cy, r2 = Z - cz;
            used = true;
            acc[0] += s0;
            acc[1] += s1;
            acc[2] += s2;
            acc[3] = fma(r1, s2, fma(-r2, s1, acc[3]));
            acc[4] = fma(r2, s0, fma(-r0, s2, acc[4]));
            acc[5] = fma(r0, s1, fma(-r1, s0, acc[5]));
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t mine = k1 - k0 - rank * BT;  // markers from the block's first on
    const int nw = mine <= 0 ? 0 : mine < BT ? ((int)mine + 31) / 32 : BT / 32;  // warps with markers
    if (warp < nw) {
        // the lanes' sums and then the warps', in three floats still (in FP64 the conversions and the tree were
        // most of the time of bodies of a few hundred markers: 5,000 of 200 markers 183 -> 105 us)
        const bool doubles = __any_sync(0xffffffffu, used);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                Sum3 v;
                v.a = __shfl_down_sync(0xffffffffu, sum[c].a, o);
                v.b = __shfl_down_sync(0xffffffffu, sum[c].b, o);
                v.c = __shfl_down_sync(0xffffffffu, sum[c].c, o);
                sum[c].add(v);
            }
            if (doubles)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
            if (lane == 0) {
                s_float[c][warp][0] = sum[c].a, s_float[c][warp][1] = sum[c].b, s_float[c][warp][2] = sum[c].c;
                s_double[c][warp] = acc[c];
            }
        }
        if (lane == 0) s_used[warp] = doubles;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        Sum3 a;
        double d = 0.0;
        for (int k = 0; k < nw; ++k) {
            const float* f = s_float[threadIdx.x][k];
            a.add(f[0]), a.low(f[1]), a.last(f[2]);
            if (s_used[k]) d += s_double[threadIdx.x][k];
        }
        s_sum[threadIdx.x] = d + a.value();
    }
    if (nb > 1)
        cluster.sync();
    else
        __syncthreads();
    if (rank == 0 && threadIdx.x < 6) {
        double a = 0.0;
        for (int k = 0; k < nb; ++k) a += *cluster.map_shared_rank(&s_sum[threadIdx.x], k);
        if (!DV) a *= (double)w;
        (threadIdx.x < 3 ? lin : ang)[3 * b + threadIdx.x % 3] = scale * a;
    }
    if (nb > 1) cluster.sync();  // the partial sums stay until they are read
}

template <bool DV, int MINB>
cudaError_t launch_body(int blocks, int nb, cudaStream_t s, const double* x, const double* y, const double* z,
                        const float* v, const float* dV, float w, int64_t n, const int64_t* start, const double* xb,
                        double scale, double* lin, double* ang) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(BT);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)nb;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_body_sums<DV, MINB>, x, y, z, v, dV, w, n, start, xb, scale, lin, ang);
}

} // namespace

} // namespace ot

using namespace ot;

extern "C" ot_status ot_body_sums(const double* d_x, const double* d_y, const double* d_z, const float* d_v,
                                  const float* d_dV, float w, int64_t n, const int64_t* d_start, int n_bodies,
                                  const double* d_xb, double scale, double* d_lin, double* d_ang, void* stream) {
    if (n < 0 || n_bodies < 0 || n_bodies > (1 << 24)) return OT_ERR_ARG;
    if (n_bodies == 0) return OT_OK;
    if (!d_start || !d_xb || !d_lin || !d_ang || (n > 0 && (!d_x || !d_y || !d_z || !d_v))) return OT_ERR_ARG;
    // blocks per body: up to the portable cluster size while all of them are at most 6 per SM (more than
    // are resident at once: large bodies get their share as small ones end), one when the bodies
    // alone are that many or the markers are few.  Lines of 3, 6 and 1000 per SM: 64 bodies of different
    // sizes 349, 277 and 277 us (7.5M markers), 156, 95 and 95 us (2M with volumes), 64 of one size
    // 175, 178 and 185 us, 1,000 of one size 156, 154 and 384 us
    int nb = 8;
    while (nb > 1 && ((int64_t)n_bodies * nb > 6 * (int64_t)num_sms() || (int64_t)n_bodies * nb * BT > 4 * n)) nb >>= 1;
    // registers: 99 to 121 (2 blocks per SM) while the blocks are few and long, 80 (3 blocks) for many,
    // which are short.  2 and 3 blocks: 64 bodies of 7.5M and 2M markers 379 and 433 us together, 5,000
    // bodies of 5M 206 and 177, of 1M 105 and 88, of 100,000 86 and 63
    const int blocks = n_bodies * nb;
    const bool few = blocks <= 6 * num_sms();
    const auto launch = d_dV ? (few ? launch_body<true, 2> : launch_body<true, 3>)
                             : (few ? launch_body<false, 2> : launch_body<false, 3>);
    OT_CUDA(launch(blocks, nb, (cudaStream_t)stream, d_x, d_y, d_z, d_v, d_dV, w, n, d_start, d_xb, scale, d_lin, d_ang));
    count_launch();
    return OT_OK;
}
