// kernels_plain.cuh -- the plain FP64 path: one thread per pixel (render), per sample
// (records) or per ray (trace_rays); the whole Sect. 4 pipeline in one kernel.
// This is the comparator the optimised paths are measured against.
#pragma once
#include <cuda_runtime.h>

#include "internal.h"
#include "trace.cuh"

namespace ck {

// Threads past the last pixel, sample or ray stay with their warp (the lanes of a warp step together).
template <int VAR, int MODE, int INTEG, bool HAM>
__global__ void __launch_bounds__(128) k_render_plain(Params p, int spp, unsigned long long seed, float4 *out) {
    extern __shared__ double plain_smem[];
    const long long pix = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = pix < (long long)p.W * p.Hp;
    int i = (int)(pix % p.W), j = (int)(pix / p.W);
    float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, acc3 = 0.f;
    for (int s = 0; s < spp; ++s) {
        double o[3], d[3];
        camera_ray(p, i, j, s, spp, seed, o, d);
        cloak_record rec;
        float rgb[3];
        trace_ray<VAR, MODE, INTEG, HAM>(p, valid, o, d, plain_smem, rec, rgb);
        float w = (float)rec.weight;
        acc0 += w * rgb[0];
        acc1 += w * rgb[1];
        acc2 += w * rgb[2];
        acc3 += w;
    }
    if (!valid) return;
    float inv = 1.0f / spp;
    out[pix] = make_float4(acc0 * inv, acc1 * inv, acc2 * inv, acc3 * inv);
}

template <int VAR, int MODE, int INTEG, bool HAM>
__global__ void __launch_bounds__(128) k_records_plain(Params p, int spp, unsigned long long seed,
                                                        cloak_record *out) {
    extern __shared__ double plain_smem[];
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = idx < (long long)p.W * p.Hp * spp;
    long long pix = idx / spp;
    int s = (int)(idx - pix * spp);
    int i = (int)(pix % p.W), j = (int)(pix / p.W);
    double o[3], d[3];
    camera_ray(p, i, j, s, spp, seed, o, d);
    cloak_record rec;
    float rgb[3];
    trace_ray<VAR, MODE, INTEG, HAM>(p, valid, o, d, plain_smem, rec, rgb);
    if (valid) out[idx] = rec;
}

template <int VAR, int MODE, int INTEG, bool HAM>
__global__ void __launch_bounds__(128) k_trace_rays(Params p, const double *rays, long long n, cloak_record *out) {
    extern __shared__ double plain_smem[];
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = idx < n;
    const double *r = rays + 6 * (valid ? idx : n - 1);
    double o[3] = {r[0], r[1], r[2]}, d[3] = {r[3], r[4], r[5]};
    cloak_record rec;
    float rgb[3];
    trace_ray<VAR, MODE, INTEG, HAM>(p, valid, o, d, plain_smem, rec, rgb);
    if (valid) out[idx] = rec;
}

// ---------------------------------------------------------------- launchers (one variant per translation unit)
template <int V, int M, int I, bool HAM>
constexpr size_t plain_smem_bytes(int threads) {
    return (size_t)PlainStepper<V, M, I, HAM>::SMEM_PER_THREAD * threads;
}
template <int V, int M, int I, bool HAM>
static cudaError_t render_plain_vmi(const Params &p, int spp, unsigned long long seed, float4 *out, cudaStream_t st) {
    long long n = (long long)p.W * p.Hp;
    const int bs = 128;
    k_render_plain<V, M, I, HAM><<<(unsigned)((n + bs - 1) / bs), bs, plain_smem_bytes<V, M, I, HAM>(bs), st>>>(p, spp, seed, out);
    return cudaGetLastError();
}
template <int V, int M, int I, bool HAM>
static cudaError_t records_plain_vmi(const Params &p, int spp, unsigned long long seed, cloak_record *out,
                                     cudaStream_t st) {
    long long n = (long long)p.W * p.Hp * spp;
    const int bs = 128;
    k_records_plain<V, M, I, HAM><<<(unsigned)((n + bs - 1) / bs), bs, plain_smem_bytes<V, M, I, HAM>(bs), st>>>(p, spp, seed, out);
    return cudaGetLastError();
}
template <int V, int M, int I, bool HAM>
static cudaError_t trace_rays_vmi(const Params &p, const double *rays, long long n, cloak_record *out,
                                  cudaStream_t st) {
    const int bs = 128;
    k_trace_rays<V, M, I, HAM><<<(unsigned)((n + bs - 1) / bs), bs, plain_smem_bytes<V, M, I, HAM>(bs), st>>>(p, rays, n, out);
    return cudaGetLastError();
}

// the Hamiltonian form is refused for the test medium, which has no such kernels
#define CK_MI_SWITCH(FN, ...)                                                                        \
    if constexpr (V != V_TEST) {                                                                     \
        if (p.formulation) {                                                                         \
            if (mode == M_ORD && p.integ == I_RK4) return FN<V, M_ORD, I_RK4, true>(__VA_ARGS__);    \
            if (mode == M_ORD && p.integ == I_DP45) return FN<V, M_ORD, I_DP45, true>(__VA_ARGS__);  \
            if (mode == M_EXT && p.integ == I_RK4) return FN<V, M_EXT, I_RK4, true>(__VA_ARGS__);    \
            if (mode == M_EXT && p.integ == I_DP45) return FN<V, M_EXT, I_DP45, true>(__VA_ARGS__);  \
        }                                                                                            \
    }                                                                                                \
    if (mode == M_ORD && p.integ == I_RK4) return FN<V, M_ORD, I_RK4, false>(__VA_ARGS__);           \
    if (mode == M_ORD && p.integ == I_DP45) return FN<V, M_ORD, I_DP45, false>(__VA_ARGS__);         \
    if (mode == M_EXT && p.integ == I_RK4) return FN<V, M_EXT, I_RK4, false>(__VA_ARGS__);           \
    if (mode == M_EXT && p.integ == I_DP45) return FN<V, M_EXT, I_DP45, false>(__VA_ARGS__);         \
    return cudaErrorInvalidValue;

template <int V>
cudaError_t launch_render_plain_v(const Params &p, int mode, int spp, unsigned long long seed, float4 *out,
                                  cudaStream_t st) {
    CK_MI_SWITCH(render_plain_vmi, p, spp, seed, out, st)
}
template <int V>
cudaError_t launch_records_plain_v(const Params &p, int mode, int spp, unsigned long long seed, cloak_record *out,
                                   cudaStream_t st) {
    CK_MI_SWITCH(records_plain_vmi, p, spp, seed, out, st)
}
template <int V>
cudaError_t launch_trace_rays_v(const Params &p, int mode, const double *rays, long long n, cloak_record *out,
                                cudaStream_t st) {
    CK_MI_SWITCH(trace_rays_vmi, p, rays, n, out, st)
}

#define CK_INSTANTIATE_PLAIN(V)                                                                                   \
    template cudaError_t launch_render_plain_v<V>(const Params &, int, int, unsigned long long, float4 *,         \
                                                  cudaStream_t);                                                  \
    template cudaError_t launch_records_plain_v<V>(const Params &, int, int, unsigned long long, cloak_record *,   \
                                                   cudaStream_t);                                                 \
    template cudaError_t launch_trace_rays_v<V>(const Params &, int, const double *, long long, cloak_record *,    \
                                                cudaStream_t);

}  // namespace ck
