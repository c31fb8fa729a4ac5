// ot_field.cu -- an analytic cell-centred field on the leaves: u(x) = sum_m A_m cos(2 pi n_m . x
// + phi_m) at every leaf centre, for integer wave vectors n_m (the random solenoidal fields the
// tracking driver re-samples on each new octree, standing in for the fluid solver's field).
// The phase is exact fixed point: a leaf centre at level l is (2 x + 2^(21-l)) 2^-22 per axis
// (x its level-21 anchor coordinate), so n . x in turns is an integer times 2^-22; with the
// phase rounded to 2^-32 turns the whole argument reduces modulo one turn in integer
// arithmetic, and only the final cosine is FP32 (cospif).
#include <algorithm>
#include <cmath>

#include "ot_internal.h"
#include "ot_sum.cuh"

namespace ot {

namespace {

constexpr int MAX_MODES = 64;

struct Modes {
    int m;
    int n[MAX_MODES][3];
    float amp[MAX_MODES][3];
    uint32_t phase[MAX_MODES];  // turns, 2^-32 units
};

// Four leaves per thread: a mode's seven constants are loaded once for the four, and their cosines,
// which bound the kernel, overlap (17.3M leaves and 32 modes: 669 -> 591 us).
__global__ void __launch_bounds__(256) k_field_fourier(const uint64_t* __restrict__ key,
                                                       const uint8_t* __restrict__ level, int64_t n, Modes md,
                                                       float4* __restrict__ out) {
    constexpr int R = 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < n; i0 += R * stride) {
        uint32_t c[R][3];
        float u[R][3];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t i = min(i0 + r * stride, n - 1);
            demorton3(key[i], c[r][0], c[r][1], c[r][2]);
            const uint32_t off = 1u << (MAXLEVEL - level[i]);
#pragma unroll
            for (int d = 0; d < 3; ++d) c[r][d] = 2 * c[r][d] + off, u[r][d] = 0.0f;
        }
        for (int k = 0; k < md.m; ++k) {
            const uint32_t n0 = (uint32_t)md.n[k][0], n1 = (uint32_t)md.n[k][1], n2 = (uint32_t)md.n[k][2];
            const uint32_t ph = md.phase[k];
            const float a0 = md.amp[k][0], a1 = md.amp[k][1], a2 = md.amp[k][2];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                // turns in 2^-22 units, of which one turn is the low 22 bits: modulo 2^32 is enough
                const uint32_t t = n0 * c[r][0] + n1 * c[r][1] + n2 * c[r][2];
                const uint32_t T = (t << 10) + ph;              // mod 1 turn, 2^-32 units
                const float fr = (float)(int32_t)T * 0x1p-32f;  // in [-1/2, 1/2)
                const float w = cospif(2.0f * fr);
                u[r][0] += a0 * w;
                u[r][1] += a1 * w;
                u[r][2] += a2 * w;
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (i0 + r * stride < n) out[i0 + r * stride] = make_float4(u[r][0], u[r][1], u[r][2], 0.0f);
    }
}

// Volume-weighted field sums, FP64: block b adds the leaves of its stride in a fixed order,
// then a fixed tree; a single block then adds the block partials in a fixed tree.
// FP64 additions bound it (the pipe was busy 84%), so a thread keeps its running sums in three floats
// each, which carry 72 bits, and goes to FP64 once at the end; terms that
// floats cannot take exactly are added in FP64 at once.  17.3M leaves 197 -> 61 us (the finishing block
// 32 -> 4 us).
constexpr int MT = 256;

__global__ void __launch_bounds__(MT) k_field_sum(const uint8_t* __restrict__ level, int64_t n,
                                                  const float4* __restrict__ f, double* __restrict__ part) {
    __shared__ double s[3][MT];
    constexpr int R = 4;  // leaves whose loads are in flight together
    Sum3 s0, s1, s2;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    const int64_t stride = (int64_t)gridDim.x * MT;
    for (int64_t i0 = blockIdx.x * (int64_t)MT + threadIdx.x; i0 < n; i0 += R * stride) {
        float4 v[R];
        int l[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t i = i0 + r * stride;
            v[r] = i < n ? f[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            l[r] = i < n ? (int)level[i] : 0;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (plain(v[r].x) && plain(v[r].y) && plain(v[r].z)) {
                const float vol = exp2_neg(3 * l[r]);  // 8^-level
                s0.add(vol * v[r].x), s1.add(vol * v[r].y), s2.add(vol * v[r].z);
            } else {
                const double vol = __longlong_as_double((long long)(1023 - 3 * l[r]) << 52);
                a0 += vol * v[r].x, a1 += vol * v[r].y, a2 += vol * v[r].z;
            }
        }
    }
    a0 += s0.value(), a1 += s1.value(), a2 += s2.value();
    s[0][threadIdx.x] = a0, s[1][threadIdx.x] = a1, s[2][threadIdx.x] = a2;
    __syncthreads();
    for (int o = MT / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int c = 0; c < 3; ++c) s[c][threadIdx.x] += s[c][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x < 3) part[3 * blockIdx.x + threadIdx.x] = s[threadIdx.x][0];
}

// Warp c sums component c of the partials: lane-strided, then a fixed tree.
__global__ void k_field_mean_finish(const double* __restrict__ part, int nb, double* __restrict__ mean) {
    const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double a = 0.0;
    for (int b = lane; b < nb; b += 32) a += part[3 * b + c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) mean[c] = a;  // the unit cube's volume is 1
}

__global__ void __launch_bounds__(MT) k_field_sub(float4* __restrict__ f, int64_t n, const double* __restrict__ mean) {
    const float m0 = (float)mean[0], m1 = (float)mean[1], m2 = (float)mean[2];
    for (int64_t i = blockIdx.x * (int64_t)MT + threadIdx.x; i < n; i += (int64_t)gridDim.x * MT) {
        float4 v = f[i];
        v.x -= m0, v.y -= m1, v.z -= m2;
        f[i] = v;
    }
}

} // namespace

} // namespace ot

using namespace ot;

// Block partials of the mean: at most MEAN_BLOCKS blocks, so the workspace has a fixed size.
constexpr int MEAN_BLOCKS = 1024;

extern "C" ot_status ot_field_mean_workspace_size(const ot_octree* t, size_t* bytes) {
    if (!t || !bytes) return OT_ERR_ARG;
    *bytes = sizeof(double) * (3 * (size_t)MEAN_BLOCKS + 3);
    return OT_OK;
}

extern "C" ot_status ot_field_subtract_mean(const ot_octree* t, float* d_field, double* d_mean, void* d_workspace,
                                            size_t ws_bytes, void* stream) {
    if (!t || !d_field || !d_workspace || ((uintptr_t)d_workspace & 7) ||
        ws_bytes < sizeof(double) * (3 * (size_t)MEAN_BLOCKS + 3))
        return OT_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = (int)std::max<int64_t>(
        1, std::min<int64_t>({(t->n + MT - 1) / MT, (int64_t)num_sms() * 4, (int64_t)MEAN_BLOCKS}));
    double* part = static_cast<double*>(d_workspace);
    double* mean = part + 3 * nb;
    k_field_sum<<<nb, MT, 0, s>>>(t->d_level, t->n, reinterpret_cast<const float4*>(d_field), part);
    k_field_mean_finish<<<1, 96, 0, s>>>(part, nb, mean);
    k_field_sub<<<nb, MT, 0, s>>>(reinterpret_cast<float4*>(d_field), t->n, mean);
    count_launch(3);
    if (d_mean) OT_CUDA(cudaMemcpyAsync(d_mean, mean, sizeof(double) * 3, cudaMemcpyDeviceToDevice, s));
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}

extern "C" ot_status ot_field_fourier(const ot_octree* t, int n_modes, const int32_t* h_wave, const double* h_amp,
                                      const double* h_phase, float* d_field, void* stream) {
    if (!t || n_modes < 0 || n_modes > MAX_MODES || (n_modes > 0 && (!h_wave || !h_amp || !h_phase)) || !d_field)
        return OT_ERR_ARG;
    Modes md{};
    md.m = n_modes;
    for (int k = 0; k < n_modes; ++k) {
        for (int d = 0; d < 3; ++d) {
            const int32_t w = h_wave[3 * k + d];
            if (w < -(1 << 12) || w > (1 << 12)) return OT_ERR_ARG;
            md.n[k][d] = w;
            md.amp[k][d] = (float)h_amp[3 * k + d];
        }
        double turns = h_phase[k] / (2.0 * M_PI);
        turns -= std::floor(turns);
        md.phase[k] = (uint32_t)(uint64_t)std::llround(turns * 4294967296.0);
    }
    if (t->n == 0) return OT_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((t->n + 255) / 256, (int64_t)num_sms() * 8));
    k_field_fourier<<<grid, 256, 0, s>>>(t->d_key, t->d_level, t->n, md, reinterpret_cast<float4*>(d_field));
    count_launch();
    OT_CUDA(cudaGetLastError());
    return OT_OK;
}
