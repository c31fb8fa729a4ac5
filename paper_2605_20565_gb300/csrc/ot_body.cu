// ot_body.cu -- per-body linear and angular sums of a marker quantity (Sec. 2.3, rigid bodies):
//   lin_b = scale sum_{k in b} v_k w_k,   ang_b = scale sum_{k in b} (X_k - x_b) x v_k w_k.
// With v the velocity interpolated at the internal markers and scale = rho_f these are the
// internal fluid's linear and angular momenta P and L; with v = F_k at the surface markers and
// scale = -1, the IBM force and torque.  FP64 accumulation in a fixed order (thread-strided, then
// a fixed tree over the threads and blocks of a body): bit-identical from run to run.
#include <cooperative_groups.h>

#include "ot_internal.h"

namespace ot {

namespace {

namespace cg = cooperative_groups;

constexpr int BT = 256;

// One thread-block cluster per body; its blocks share the body's markers and the first adds the
// blocks' partial sums in rank order from their shared memory (there is no workspace to keep them
// in, and atomics would leave the order open).  Bound by the FP64 pipe (2 lanes per clock and SM):
// 12 FP64 operations per marker, 15 with marker volumes -- a common weight is applied to the
// sums, products go through fused multiply-adds.
// DV: marker volumes given.
template <bool DV>
__global__ void __launch_bounds__(BT) k_body_sums(const double* __restrict__ x, const double* __restrict__ y,
                                                  const double* __restrict__ z, const float* __restrict__ v,
                                                  const float* __restrict__ dV, float w, int64_t n,
                                                  const int64_t* __restrict__ start, const double* __restrict__ xb,
                                                  double scale, double* __restrict__ lin, double* __restrict__ ang) {
    __shared__ double s_warp[6][BT / 32];
    __shared__ double s_sum[6];
    cg::cluster_group cluster = cg::this_cluster();
    const int nb = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int b = blockIdx.x / nb;
    const int64_t k0 = start[b], k1 = start[b + 1];
    const double cx = xb[3 * b], cy = xb[3 * b + 1], cz = xb[3 * b + 2];
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int64_t k = k0 + rank * BT + (int)threadIdx.x; k < k1; k += (int64_t)nb * BT) {
        double v0 = (double)v[k], v1 = (double)v[n + k], v2 = (double)v[2 * n + k];
        if (DV) {
            const double wk = (double)dV[k];
            v0 *= wk, v1 *= wk, v2 *= wk;
        }
        const double r0 = x[k] - cx, r1 = y[k] - cy, r2 = z[k] - cz;
        acc[0] += v0;
        acc[1] += v1;
        acc[2] += v2;
        acc[3] = fma(r1, v2, fma(-r2, v1, acc[3]));
        acc[4] = fma(r2, v0, fma(-r0, v2, acc[4]));
        acc[5] = fma(r0, v1, fma(-r1, v0, acc[5]));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
        if (lane == 0) s_warp[c][warp] = acc[c];
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        double a = 0.0;
        for (int k = 0; k < BT / 32; ++k) a += s_warp[threadIdx.x][k];
        s_sum[threadIdx.x] = a;
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x < 6) {
        double a = 0.0;
        for (int k = 0; k < nb; ++k) a += *cluster.map_shared_rank(&s_sum[threadIdx.x], k);
        if (!DV) a *= (double)w;
        (threadIdx.x < 3 ? lin : ang)[3 * b + threadIdx.x % 3] = scale * a;
    }
    cluster.sync();  // the partial sums stay until they are read
}

template <bool DV>
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
    return cudaLaunchKernelEx(&cfg, k_body_sums<DV>, x, y, z, v, dV, w, n, start, xb, scale, lin, ang);
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
    // blocks per body: up to the portable cluster size while the chip holds all of them at once
    // (6 blocks per SM), one when the bodies alone fill it or the markers are few
    int nb = 8;
    while (nb > 1 && ((int64_t)n_bodies * nb > 6 * (int64_t)num_sms() || (int64_t)n_bodies * nb * BT > 4 * n)) nb >>= 1;
    OT_CUDA(d_dV ? launch_body<true>(n_bodies * nb, nb, (cudaStream_t)stream, d_x, d_y, d_z, d_v, d_dV, w, n, d_start,
                                     d_xb, scale, d_lin, d_ang)
                 : launch_body<false>(n_bodies * nb, nb, (cudaStream_t)stream, d_x, d_y, d_z, d_v, d_dV, w, n, d_start,
                                      d_xb, scale, d_lin, d_ang));
    count_launch();
    return OT_OK;
}
