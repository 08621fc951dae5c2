// Rays stepped by the library's state machine (csrc/integrator.cuh) from a given state, for test_crossing_start_gpu.py.
#include <cstring>

#include "integrator.cuh"

namespace {

struct Slot {  // one ray, as the integrator's queue holds it
    double *x, *y, *z, *vx, *vy, *vz, *ax, *ay, *az, *t;
    int *status;
};

template <typename S, int INTEG, bool NEWTON, int LANES>
__global__ void k_lane(ck::Params p, Slot q, int vm, bool mirrors) {
    extern __shared__ double smem[];
    S st;
    st.vm = vm;
    st.bind(smem);
    ck::Lane<S, INTEG, NEWTON, true> ray;
    ray.reset();
    st.load(q, 0);
    if (threadIdx.x < LANES) ray.start(p);
    int status = -1;
    for (int n = 0; n < 5000; ++n) {
        const bool live = ray.phase != ck::PH_IDLE;
        const unsigned int lanes = __ballot_sync(0xffffffffu, live);
        if (!lanes) break;
        if (!live) continue;
        status = ray.advance(p, st, lanes, mirrors);
        if (status >= 0) ray.phase = ck::PH_IDLE;
    }
    if (threadIdx.x == 0) {
        st.store(q, 0);
        q.t[0] = (double)ray.t;
        q.status[0] = status;
    }
}

}  // namespace

// kind: 0 one thread, 1 eight lanes, 2 mixed precision with the FP64 band, 3 with the double-float band.  y: the state,
// replaced by the one at the end.  Returns the ray's status, -2 for a CUDA error.
extern "C" int lane_trace(int kind, int vm, double R1, double R2, double H, double tol, int newton, double y[6], double *t) {
    ck::Params p;
    memset(&p, 0, sizeof(p));
    p.variant = vm >> 1;
    p.R1 = R1; p.R2 = R2; p.H = H; p.halfH = 0.5 * H;
    p.K = (R2 / (R2 - R1)) * (R2 / (R2 - R1));
    p.invK = 1.0 / p.K;
    p.R1x2 = 2 * R1; p.R1sq = R1 * R1; p.R2sq = R2 * R2;
    p.gtol_lat = ck::CROSS_G_TOL * p.R2sq; p.gtol_cap = ck::CROSS_G_TOL * p.halfH; p.gtol_metal = ck::CROSS_G_TOL * p.R1sq;
    p.gtolf_lat = (float)p.gtol_lat; p.gtolf_cap = (float)p.gtol_cap; p.gtolf_metal = (float)p.gtol_metal;
    p.R1f = (float)R1; p.R2f = (float)R2; p.halfHf = (float)p.halfH; p.Kf = (float)p.K; p.invKf = (float)p.invK;
    p.R1sq_hf = (float)p.R1sq; p.R1sq_lf = (float)(p.R1sq - (double)p.R1sq_hf);
    p.R2sq_hf = (float)p.R2sq; p.R2sq_lf = (float)(p.R2sq - (double)p.R2sq_hf);
    p.halfH_hf = (float)p.halfH; p.halfH_lf = (float)(p.halfH - (double)p.halfH_hf);
    p.integ = ck::I_DP45;
    p.precision = kind < 2 ? 0 : kind - 1;
    p.band_df = kind == 3;
    p.band_limf = kind < 2 ? 0.f : (float)(R1 + 0.02);
    p.h_or_tol = tol;
    p.max_steps = 1000;
    double *d = nullptr;
    if (cudaMalloc(&d, 16 * 8) != cudaSuccess) return -2;
    double host[16];
    for (int i = 0; i < 6; ++i) {
        if (kind < 2) {
            host[i] = y[i];
        } else {
            const float hi = (float)y[i], pair[2] = {hi, (float)(y[i] - (double)hi)};
            memcpy(&host[i], pair, 8);
        }
    }
    const unsigned long long nan = 0x7ff8000000000000ull;
    memcpy(&host[6], &nan, 8);
    cudaMemcpy(d, host, 7 * 8, cudaMemcpyHostToDevice);
    const Slot q = {d, d + 1, d + 2, d + 3, d + 4, d + 5, d + 6, d + 7, d + 8, d + 9, reinterpret_cast<int *>(d + 10)};
    constexpr int V = ck::V_ANY, I = ck::I_DP45;
    const size_t smem = 32 * ck::DP_SLOTS * sizeof(double);
    if (kind == 0 && newton) k_lane<ck::Stepper64<V, V, I>, I, true, 1><<<1, 32, smem>>>(p, q, vm, vm == 0);
    else if (kind == 0) k_lane<ck::Stepper64<V, V, I>, I, false, 1><<<1, 32, smem>>>(p, q, vm, vm == 0);
    else if (kind == 1) k_lane<ck::StepperWide<V, V, I>, I, false, ck::WIDE_LANES><<<1, 32, smem>>>(p, q, vm, vm == 0);
    else k_lane<ck::StepperMixed<V, V, I>, I, false, 1><<<1, 32, smem>>>(p, q, vm, vm == 0);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(host, d, 11 * 8, cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess) return -2;
    for (int i = 0; i < 6; ++i) {
        if (kind < 2) {
            y[i] = host[i];
        } else {
            float pair[2];
            memcpy(pair, &host[i], 8);
            y[i] = (double)pair[0] + (double)pair[1];
        }
    }
    *t = host[9];
    int status;
    memcpy(&status, &host[10], 4);
    return status;
}
