// kernels_plain.cuh -- the plain FP64 path: one thread per pixel (render), per sample
// (records) or per ray (trace_rays); the whole Sect. 4 pipeline in one kernel.
// This is the comparator the optimised paths are measured against.
#pragma once
#include <cuda_runtime.h>

#include "internal.h"
#include "trace.cuh"

namespace ck {

// One ray (pixel, sample) per thread, or per group of eight lanes (WIDE).  Threads past the last one stay with
// their warp (its lanes step together).
template <bool WIDE>
__device__ __forceinline__ long long plain_index() {
    return ((long long)blockIdx.x * blockDim.x + threadIdx.x) / (WIDE ? WIDE_LANES : 1);
}
template <bool WIDE>
__device__ __forceinline__ bool plain_writer() {
    return !WIDE || (threadIdx.x & (WIDE_LANES - 1)) == 0;
}
template <int VAR, int MODE, int INTEG, bool HAM, bool WIDE>
__global__ void __launch_bounds__(WIDE ? 32 : 128) k_render_plain(Params p, int spp, unsigned long long seed, float4 *out) {
    extern __shared__ double plain_smem[];
    const long long pix = plain_index<WIDE>();
    const bool valid = pix < (long long)p.W * p.Hp;
    int i = (int)(pix % p.W), j = (int)(pix / p.W);
    float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, acc3 = 0.f;
    for (int s = 0; s < spp; ++s) {
        double o[3], d[3];
        camera_ray(p, i, j, s, spp, seed, o, d);
        cloak_record rec;
        float rgb[3];
        trace_ray<VAR, MODE, INTEG, HAM, WIDE>(p, valid, o, d, plain_smem, rec, rgb);
        float w = (float)rec.weight;
        acc0 += w * rgb[0];
        acc1 += w * rgb[1];
        acc2 += w * rgb[2];
        acc3 += w;
    }
    if (!valid || !plain_writer<WIDE>()) return;
    float inv = 1.0f / spp;
    out[pix] = make_float4(acc0 * inv, acc1 * inv, acc2 * inv, acc3 * inv);
}

template <int VAR, int MODE, int INTEG, bool HAM, bool WIDE>
__global__ void __launch_bounds__(WIDE ? 32 : 128) k_records_plain(Params p, int spp, unsigned long long seed,
                                                                   cloak_record *out) {
    extern __shared__ double plain_smem[];
    const long long idx = plain_index<WIDE>();
    const bool valid = idx < (long long)p.W * p.Hp * spp;
    long long pix = idx / spp;
    int s = (int)(idx - pix * spp);
    int i = (int)(pix % p.W), j = (int)(pix / p.W);
    double o[3], d[3];
    camera_ray(p, i, j, s, spp, seed, o, d);
    cloak_record rec;
    float rgb[3];
    trace_ray<VAR, MODE, INTEG, HAM, WIDE>(p, valid, o, d, plain_smem, rec, rgb);
    if (valid && plain_writer<WIDE>()) out[idx] = rec;
}

template <int VAR, int MODE, int INTEG, bool HAM, bool WIDE>
__global__ void __launch_bounds__(WIDE ? 32 : 128) k_trace_rays(Params p, const double *rays, long long n,
                                                                cloak_record *out) {
    extern __shared__ double plain_smem[];
    const long long idx = plain_index<WIDE>();
    const bool valid = idx < n;
    const double *r = rays + 6 * (valid ? idx : n - 1);
    double o[3] = {r[0], r[1], r[2]}, d[3] = {r[3], r[4], r[5]};
    cloak_record rec;
    float rgb[3];
    trace_ray<VAR, MODE, INTEG, HAM, WIDE>(p, valid, o, d, plain_smem, rec, rgb);
    if (valid && plain_writer<WIDE>()) out[idx] = rec;
}

// ---------------------------------------------------------------- launchers (one variant per translation unit)
// Eight lanes per ray (one warp per block, spread over the chip's schedulers) as long as the warps do not crowd
// each other out, one thread per ray above.  In units of the rays that one warp on every scheduler holds (2432):
// RK4, whose rays all take about the same number of steps, up to one of rays and two of camera rays (some of
// which miss); DP5(4), where the slowest rays decide, one and a half and twelve.  Radial extraordinary rays, narrow ->
// wide: RK4 2000 rays 12.1 -> 10.9 ms, 4000 12.3 -> 13.8; DP5(4) 2000 rays 24.1 -> 16.8 ms, 4000 25.0 -> 17.4 with near-axis
// rays among them, 5000 without 1.8 -> 2.7; images RK4 64 x 48 12.0 -> 11.5, 96 x 72 11.9 -> 12.3;
// DP5(4) 192 x 144 2.29 -> 1.89, azimuthal 256 x 192 8.12 -> 8.18.
inline bool plain_wide(int integ, bool camera, long long n) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long unit = 4LL * WIDE_RAYS * sms;
    return 2 * n <= unit * (integ == I_RK4 ? (camera ? 4 : 2) : (camera ? 24 : 3));
}
#define CK_PLAIN_LAUNCH(KERNEL, n, camera, ...)                                                                  \
    if constexpr (!HAM) {                                                                                        \
        if (plain_wide(I, camera, n)) {                                                                          \
            KERNEL<V, M, I, HAM, true><<<(unsigned)(((n) + WIDE_RAYS - 1) / WIDE_RAYS), 32,                      \
                                         PlainStepper<V, M, I, HAM, true>::SMEM_PER_THREAD * 32, st>>>(__VA_ARGS__); \
            return cudaGetLastError();                                                                           \
        }                                                                                                        \
    }                                                                                                            \
    KERNEL<V, M, I, HAM, false><<<(unsigned)(((n) + 127) / 128), 128,                                            \
                                  PlainStepper<V, M, I, HAM, false>::SMEM_PER_THREAD * 128, st>>>(__VA_ARGS__);  \
    return cudaGetLastError();

template <int V, int M, int I, bool HAM>
static cudaError_t render_plain_vmi(const Params &p, int spp, unsigned long long seed, float4 *out, cudaStream_t st) {
    const long long n = (long long)p.W * p.Hp;
    CK_PLAIN_LAUNCH(k_render_plain, n, true, p, spp, seed, out)
}
template <int V, int M, int I, bool HAM>
static cudaError_t records_plain_vmi(const Params &p, int spp, unsigned long long seed, cloak_record *out,
                                     cudaStream_t st) {
    const long long n = (long long)p.W * p.Hp * spp;
    CK_PLAIN_LAUNCH(k_records_plain, n, true, p, spp, seed, out)
}
template <int V, int M, int I, bool HAM>
static cudaError_t trace_rays_vmi(const Params &p, const double *rays, long long n, cloak_record *out,
                                  cudaStream_t st) {
    CK_PLAIN_LAUNCH(k_trace_rays, n, false, p, rays, n, out)
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
