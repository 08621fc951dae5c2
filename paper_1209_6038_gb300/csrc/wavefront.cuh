// wavefront.cuh -- the optimised FP64 schedule.
//
//   A  k_wf_entry      one thread per (pixel, sample): camera ray, cylinder entry, Sect. 3 entry
//                      refraction and the Eq. 12 factor of the entry face; rays that miss or hit a
//                      metal disc are shaded at once, rays that enter are appended to a compacted
//                      device queue (SoA, FP64 state).
//   B  k_wf_integrate  persistent kernel, one resident grid: every lane owns one queued ray and
//                      refills itself from the queue when its ray leaves.  Each loop iteration runs
//                      ONE uniform step evaluation (DP5(4): six right-hand sides; RK4: four) for every
//                      lane; the surface-crossing search is a lane state that reuses that same step
//                      slot with a trial step size, so root finding never serialises a warp.
//                      FP64 or mixed arithmetic (integrator.cuh).
//   C  k_wf_exit       one thread per queued ray: exit refraction, Eq. 12 factor of the exit face,
//                      room lookup.
//   D  k_wf_resolve    per pixel: mean over its samples in sample order.
//
// The arithmetic of every ray is that of the plain path (trace.cuh) step for step.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "integrator.cuh"
#include "internal.h"
#include "trace.cuh"

namespace ck {

// queue slot layout (structure of arrays; capacity = rays per image)
struct Queue {
    double *x, *y, *z, *vx, *vy, *vz;  // state on entry; final state after B
    double *ax, *ay, *az;              // dv/dt at the entry state (Fermat form, FP64), NaN where not computed
    double *w_out;                     // Eq. 12 factor of the entry face (physical exit towards the camera)
    double *t;                         // time of flight after B
    int *id;                           // sample index (pixel * spp + sample)
    int *status;                       // CLOAK_RAY_* after B (EXITED / HIT_METAL_EXITED means: crossed a face)
    int *steps;
    int *face;                         // surface crossed at exit (EV_LAT / EV_TOP / EV_BOT)
    int *key;                          // cost bucket of the ray (larger = more steps expected)
    int *perm;                         // integration order: slots sorted by descending cost bucket
    unsigned int *count;               // [0] queued rays, [1] next ray of the integration kernel,
                                       // [2] rays to integrate, [4 + v] next ray of medium segment v
    unsigned int *bins;                // [nbins] bucket sizes, [nbins] scatter cursors (nbins <= 256), then
                                       // per medium segment v: [SEG_OFFSET + 2v] first index into perm, [+1] size
    long long cap;
};

constexpr int NBINS = 64;         // cost buckets of a single image
constexpr int NBINS_BATCH = 256;  // medium/mode x cost bucket of a batch: key = vm * NBINS + cost
constexpr int SEG_OFFSET = 2 * NBINS_BATCH;
__host__ __device__ constexpr int batch_key(int vm, int cost) { return vm * NBINS + cost; }
__host__ __device__ constexpr int key_vm(int key) { return key / NBINS; }
constexpr size_t QUEUE_HEADER_BYTES = 4096;
// count[8]: medium segment of the reserved long rays, count[9]: their number, count[10]: their cursor;
// from count[DEDICATED_FLAGS]: one flag per SM id (mod 256) that hosts a long-ray block
constexpr int DEDICATED_FLAGS = 576;
constexpr int LONG_RAY_BLOCKS = 4;  // default number of blocks (SMs) for the long rays
static_assert((DEDICATED_FLAGS + 256) * 4 <= (int)QUEUE_HEADER_BYTES, "queue header too small");
static_assert(DEDICATED_FLAGS * 4 >= 64 + 4 * (SEG_OFFSET + 8), "long-ray flags overlap the bins");
// every array of the queue starts on a 256-byte boundary (the float4 per-sample buffer needs 16 bytes)
constexpr size_t queue_array_bytes(long long cap, size_t elem) { return ((size_t)cap * elem + 255) & ~(size_t)255; }
constexpr size_t queue_bytes(long long cap) {
    return QUEUE_HEADER_BYTES + 11 * queue_array_bytes(cap, sizeof(double)) + queue_array_bytes(cap, sizeof(float4)) +
           6 * queue_array_bytes(cap, sizeof(int));
}

// Lay the queue, its sort arrays and the per-sample buffer out in `base` (queue_bytes(cap) bytes,
// 256-byte aligned).  The header (counters and bins) must be zeroed before each render.
inline void carve_queue(char *base, long long cap, Queue &q, float4 **samples) {
    q.count = (unsigned int *)base;
    q.bins = (unsigned int *)(base + 64);
    char *b = base + QUEUE_HEADER_BYTES;
    double **dp[11] = {&q.x, &q.y, &q.z, &q.vx, &q.vy, &q.vz, &q.ax, &q.ay, &q.az, &q.w_out, &q.t};
    for (int i = 0; i < 11; ++i) { *dp[i] = (double *)b; b += queue_array_bytes(cap, sizeof(double)); }
    *samples = (float4 *)b;
    b += queue_array_bytes(cap, sizeof(float4));
    int **ip[6] = {&q.id, &q.status, &q.steps, &q.face, &q.key, &q.perm};
    for (int i = 0; i < 6; ++i) { *ip[i] = (int *)b; b += queue_array_bytes(cap, sizeof(int)); }
    q.cap = cap;
}

// Cost bucket of an entering ray from its axial angular momentum L = (x cross k)_z: rays that pass
// close to the inner radius (small |L|) are the slow ones (the ray speed grows like 1/L there).
__device__ __forceinline__ int cost_bucket(const Params &p, const double x[3], const double k[3]) {
    float L = fabsf((float)(x[0] * k[1] - x[1] * k[0]));
    int b = (int)(-p.cost_scale * __log2f(L + 1e-30f));
    return min(max(b, 0), NBINS - 1);
}

__device__ __forceinline__ void store_sample(float4 *samples, cloak_record *recs, long long id,
                                             const cloak_record &rec, const float rgb[3]) {
    if (samples) {
        float w = (float)rec.weight;
        samples[id] = make_float4(w * rgb[0], w * rgb[1], w * rgb[2], w);
    }
    if (recs) recs[id] = rec;
}

// Sample of a camera ray that misses the cylinder (enter): the room's colour, half of the light through a polariser.
__device__ __forceinline__ void store_missed(const Params &p, float4 *samples, long long id, const float rgb[3]) {
    const float w = p.analyzer ? 0.5f : 1.0f;
    samples[id] = make_float4(w * rgb[0], w * rgb[1], w * rgb[2], w);
}

// Per-sample output of a TOF difference render (Params::tof): (w dt, w, 0, 0).
__device__ __forceinline__ void store_tof_sample(const Params &p, float4 *samples, long long id, const double o[3],
                                                 const double d[3], const cloak_record &rec) {
    const double w = rec.weight;
    samples[id] = make_float4((float)(w * tof_difference(p, o, d, rec)), (float)w, 0.f, 0.f);
}

// State format of the queue.  FP64 renders keep (x, v) as doubles; the mixed-precision path keeps each
// component as a float-float pair (hi, lo) in the same 8-byte slot, so that its FP32 stepper loads and
// stores rays with no FP64 arithmetic (a lone refilling lane converting doubles held the SM's FP64 unit
// 16 cycles per instruction for its whole warp).
__device__ __forceinline__ void put_state(bool ff, const Queue &q, unsigned int k, const double y[6]) {
    double *a[6] = {q.x, q.y, q.z, q.vx, q.vy, q.vz};
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        if (ff) {
            const float hi = (float)y[i];
            reinterpret_cast<float2 *>(a[i])[k] = make_float2(hi, (float)(y[i] - (double)hi));
        } else {
            a[i][k] = y[i];
        }
    }
}
__device__ __forceinline__ void get_state(bool ff, const Queue &q, unsigned int k, double y[6]) {
    const double *a[6] = {q.x, q.y, q.z, q.vx, q.vy, q.vz};
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        if (ff) {
            const float2 v = reinterpret_cast<const float2 *>(a[i])[k];
            y[i] = (double)v.x + (double)v.y;
        } else {
            y[i] = a[i][k];
        }
    }
}

// Eq. 12 factors of the mixed-precision path: the field-continuity solve in FP32 where the vacuum wave meets
// the face at more than ~11.5 degrees from grazing (cos > 0.2), in FP64 otherwise (the 4x4 system loses its
// conditioning towards grazing).  The face geometry, the double refraction and the exit refraction stay
// in FP64 on every path.
constexpr double F32_EQ12_MIN_COS = 0.2;
// axis: the camera's polariser (nullable)
__device__ __forceinline__ double entry_factor(const Params &p, int mode, double eo, double ee, const double c[3],
                                               const double n[3], const double k[3], const double *axis) {
    if (p.precision != 0) {
        const double kn = dot3(k, n), kt2 = dot3(k, k) - kn * kn;  // the vacuum wave's normal part: 1 - kt2
        if (1.0 - kt2 > F32_EQ12_MIN_COS * F32_EQ12_MIN_COS) {
            const float cf[3] = {(float)c[0], (float)c[1], (float)c[2]}, nf[3] = {(float)n[0], (float)n[1], (float)n[2]},
                        kf[3] = {(float)k[0], (float)k[1], (float)k[2]};
            float af[3];
            if (axis) { af[0] = (float)axis[0]; af[1] = (float)axis[1]; af[2] = (float)axis[2]; }
            return (double)transmission_out(mode, (float)eo, (float)ee, cf, nf, kf, axis ? af : (const float *)nullptr);
        }
    }
    return transmission_out(mode, eo, ee, c, n, k, axis);
}
// cos_vac: |d . n| of the vacuum wave d at the exit face
__device__ __forceinline__ double exit_factor(const Params &p, int mode, double eo, double ee, const double c[3],
                                              const double n[3], const double d[3], double cos_vac) {
    if (p.precision != 0 && cos_vac > F32_EQ12_MIN_COS) {
        const float cf[3] = {(float)c[0], (float)c[1], (float)c[2]}, nf[3] = {(float)n[0], (float)n[1], (float)n[2]},
                    df[3] = {(float)d[0], (float)d[1], (float)d[2]};
        return (double)transmission_in(mode, (float)eo, (float)ee, cf, nf, df);
    }
    return transmission_in(mode, eo, ee, c, n, d);
}

// Append an entering ray to the queue; one atomic per warp for the slot and one per distinct key.
// a: dv/dt at y (the integrator's first stage, computed here where every lane of the warp has one), or
// null.  ff: store the state as float-float pairs (mixed precision).
__device__ __forceinline__ void queue_append(const Queue &q, const double y[6], double w_out, int id, int key,
                                             const double *a = nullptr, bool ff = false) {
    const unsigned int act = __activemask();
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(act) - 1;
    unsigned int base = 0;
    if (lane == leader) base = atomicAdd(q.count, (unsigned int)__popc(act));
    base = __shfl_sync(act, base, leader);
    unsigned int slot = base + __popc(act & ((1u << lane) - 1u));
    put_state(ff, q, slot, y);
    q.ax[slot] = a ? a[0] : __longlong_as_double(0x7ff8000000000000ll);
    q.ay[slot] = a ? a[1] : 0.0;
    q.az[slot] = a ? a[2] : 0.0;
    q.w_out[slot] = w_out;
    q.id[slot] = id;
    q.key[slot] = key;
    unsigned int same = __match_any_sync(act, key);
    if (lane == __ffs(same) - 1) atomicAdd(q.bins + key, (unsigned int)__popc(same));
}

template <int VAR, int MODE>
__global__ void __launch_bounds__(128) k_wf_entry(Params p, int spp, unsigned long long seed, Queue q,
                                                  float4 *samples, cloak_record *recs) {
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long n = (long long)p.W * p.Hp * spp;
    if (idx >= n) return;
    long long pix = idx / spp;
    int s = (int)(idx - pix * spp);
    int i = (int)(pix % p.W), j = (int)(pix / p.W);
    float rgb[3];
    if (!recs) {  // rays that miss, in single precision (records carry their FP64 direction)
        const uint64_t px = uint64_t(j) * uint64_t(p.W) + uint64_t(i);
        const float xi1 = spp > 1 ? jitter_f32(seed, px, s, 0) : 0.5f, xi2 = spp > 1 ? jitter_f32(seed, px, s, 1) : 0.5f;
        if (miss_f32(p, frame_f32(p.eye, p.fw, p.rt, p.up, p.tx, p.ty, p.W, p.Hp), i, j, xi1, xi2, rgb)) {
            store_missed(p, samples, idx, rgb);
            return;
        }
    }
    double o[3], d[3], y[6], k0[3], n_in[3], mat[5];
    camera_ray(p, i, j, s, spp, seed, o, d);
    cloak_record rec;
    if (!enter<MODE>(p, o, d, rec, rgb, y, k0, n_in, mat)) {
        store_sample(samples, recs, idx, rec, rgb);
        return;
    }
    // Eq. 12 at the entry face along the physical direction: light leaves the cloak towards the camera
    double mk0[3] = {-k0[0], -k0[1], -k0[2]}, c[3] = {mat[2], mat[3], mat[4]};
    double w_out = entry_factor(p, MODE, mat[0], mat[1], c, n_in, mk0, analyzer_axis(p));
    double dy[6];
    const bool first = p.precision == 0 && p.formulation == 0;  // the FP64 Fermat stepper's first stage
    if (first) rhs<VAR, MODE>(p, y, dy);
    queue_append(q, y, w_out, (int)idx, cost_bucket(p, y, k0), first ? dy + 3 : nullptr, p.precision != 0);
}

// Longest-first order: a counting sort of the queue by descending key.  k_wf_sort_scan turns the bucket
// sizes into scatter cursors and medium segments, k_wf_sort_scatter writes the permutation.  With the
// batch key (medium major, cost minor) every medium occupies one contiguous segment of the permutation,
// in descending cost order.
__global__ void k_wf_sort_scan(Queue q, int nbins, unsigned int reserve);
__global__ void k_wf_sort_scatter(Queue q);

// Rays of a warp on eight lanes each (StepperWide) until they are done: group g starts with the ray of slot
// `slot` (state st, progress h, t, steps, metal; slot < 0: none), and fetches the next of the `rl` reserved rays
// (from perm[first]) whenever it has none.
template <int VAR, int MODE, int INTEG, int PREC>
__device__ __noinline__ void wf_integrate_wide(const Params &kp, const Queue &q, double *smem, const double y[6],
                                                  int vm, double h, double t, int steps, bool metal, int slot,
                                                  unsigned int rl, unsigned int first) {
    typedef StepperWide<VAR, MODE, INTEG> S;
    Params p;  // what the steps read, in registers instead of behind a pointer (a load per use and step)
    p.R1 = kp.R1;
    p.R1sq = kp.R1sq;
    p.R2sq = kp.R2sq;
    p.halfH = kp.halfH;
    p.gtol_lat = kp.gtol_lat;
    p.gtol_cap = kp.gtol_cap;
    p.gtol_metal = kp.gtol_metal;
    p.R1f = kp.R1f;
    p.h_or_tol = kp.h_or_tol;
    p.max_steps = kp.max_steps;
    S st;
    st.bind(smem);
    st.vm = vm;
#pragma unroll
    for (int i = 0; i < 6; ++i) st.y[i] = y[i];
    st.begin();
    Lane<S, INTEG, INTEG == I_DP45, false> ray;
    ray.reset();
    if (slot >= 0) {
        ray.start(p);
        ray.h = h;
        ray.t = t;
        ray.steps = steps;
        ray.metal = metal;
    }
    bool more = rl > 0;
    for (;;) {
        if (ray.phase == PH_IDLE && more) {
            unsigned int k = 0;
            if (st.l == 0) k = atomicAdd(q.count + 10, 1u);
            k = __shfl_sync(st.grp, k, 0, WIDE_LANES);
            if (k < rl) {
                slot = q.perm[first + k];
                st.load(q, slot);
                ray.start(p);
            } else {
                more = false;
            }
        }
        const bool live = ray.phase != PH_IDLE;
        const unsigned int lm = __ballot_sync(0xffffffffu, live);
        if (!lm) break;
        if (!live) continue;
        const bool mirrors = (VAR == V_RADIAL && MODE == M_ORD) || (VAR == V_ANY && st.vm == 0);
        const int status = ray.advance(p, st, lm, mirrors);
        if (status >= 0) {
            if (st.l == 0) {
                st.store(q, slot);
                q.t[slot] = ray.t;
                q.status[slot] = status;
                q.steps[slot] = ray.steps;
                q.face[slot] = ray.evbest;
            }
            ray.phase = PH_IDLE;
        }
    }
}

// PREC: 0 FP64 (Fermat form), 1 mixed precision, 2 FP64 Hamiltonian form
template <int VAR, int MODE, int INTEG, int PREC>
using WfStepper = typename std::conditional<
    PREC == 0, Stepper64<VAR, MODE, INTEG>,
    typename std::conditional<PREC == 1, StepperMixed<VAR, MODE, INTEG>, StepperHam<VAR, MODE, INTEG>>::type>::type;
template <int VAR, int MODE, int INTEG, int PREC>
__device__ __forceinline__ void wf_integrate_body(const Params &p, const Queue &q) {
    typedef WfStepper<VAR, MODE, INTEG, PREC> S;
    extern __shared__ double wf_smem[];
    S st;
    st.vm = 0;
    st.bind(wf_smem);
    const int lane = threadIdx.x & 31;
    const unsigned int n = q.count[2];  // rays left to integrate after the sort
    // medium segments of the permutation (batch: one per medium/mode; a lane draws rays from its
    // warp's current segment, so that the lanes of a warp evaluate one medium's equations)
    // the first segment is chosen per SM, so that the warps resident on one SM run one medium's code
    // (a quarter of the kernel's instructions for the instruction caches)
    unsigned int smid = 0;
    if (VAR == V_ANY) asm("mov.u32 %0, %%smid;" : "=r"(smid));
    int seg = VAR == V_ANY ? 3 - (int)(smid & 3u) : 0;
    // Long-ray blocks: the sort reserved the first rl rays of the order (of medium segment rv in a
    // batch) -- those that pass closest to the inner radius, up to 3.4e4 steps each -- for the warps of
    // the first p.dedicated_blocks blocks.  The other blocks resident on those SMs leave at once, so
    // these warps share their SM's FP64 unit with no others and advance their long rays at close to
    // one warp's latency (FP64: four rays per warp, eight lanes each); on a full SM they would get a fraction
    // of it and finish last, after the rest of the queue.  (A block that misses the flag only costs speed:
    // every ray is still integrated once.)
    const unsigned int rl = q.count[9];
    const unsigned int rv = rl ? q.count[8] : 0u;
    bool reserve = false;
    if (rl) {
        if (VAR != V_ANY) asm("mov.u32 %0, %%smid;" : "=r"(smid));
        volatile unsigned int *sm_taken = q.count + DEDICATED_FLAGS;
        if ((int)blockIdx.x < p.dedicated_blocks) {
            reserve = true;
            seg = (int)rv;
            if (threadIdx.x == 0) sm_taken[smid & 255u] = 1u;
        } else {
            __nanosleep(2000);
            unsigned int f = 0;
            if ((threadIdx.x & 31u) == 0) f = sm_taken[smid & 255u];
            if (__shfl_sync(0xffffffffu, f, 0)) return;  // the whole warp leaves
        }
    }
    if constexpr (PREC == 0) {
        if (reserve) {
            const double none[6] = {0, 0, 0, 0, 0, 0};
            wf_integrate_wide<VAR, MODE, INTEG, PREC>(p, q, wf_smem, none, (int)rv, 0.0, 0.0, 0, false, -1, rl,
                                                      VAR == V_ANY ? q.bins[SEG_OFFSET + 2 * rv] : 0u);
            reserve = false;
            __syncwarp();
        }
    }
    Lane<S, INTEG, INTEG == I_DP45 && PREC != 1, false> ray;
    ray.reset();
    int slot = -1;
    bool drained = false;  // the queue had no ray left for this lane

    // Every lane of a warp stays in the loop until the whole warp is drained, and the warp reconverges
    // before the one step evaluation of each iteration, which all its live lanes then run together
    // (stepping and crossing search alike).
    for (;;) {
        // ---- refill: a lane without a ray takes the next queued one
        if (ray.phase == PH_IDLE && !drained) {
            int phase = PH_IDLE;
            if (VAR == V_ANY) {
                if (reserve) {  // a long-ray lane: the reserved rays first
                    const unsigned int k = atomicAdd(q.count + 10, 1u);
                    if (k < rl) {
                        slot = q.perm[__ldg(q.bins + SEG_OFFSET + 2 * rv) + k];
                        seg = (int)rv;
                        st.vm = seg;
                        phase = PH_STEP;
                    } else {
                        reserve = false;
                    }
                }
                // the current segment first, then the others in descending medium order (segment rv
                // without its reserved head)
                for (int tries = 0; tries < 4 && phase != PH_STEP; ++tries) {
                    const unsigned int skip = (unsigned int)seg == rv ? rl : 0u;
                    const unsigned int len = __ldg(q.bins + SEG_OFFSET + 2 * seg + 1) - skip;
                    const unsigned int k = len ? atomicAdd(q.count + 4 + seg, 1u) : 0xffffffffu;
                    if (k < len) {
                        slot = q.perm[__ldg(q.bins + SEG_OFFSET + 2 * seg) + skip + k];
                        st.vm = seg;
                        phase = PH_STEP;
                        break;
                    }
                    seg = (seg + 3) & 3;
                }
            } else {
                if (reserve) {  // a long-ray lane: the reserved head of the order first
                    const unsigned int k = atomicAdd(q.count + 10, 1u);
                    if (k < rl) {
                        slot = q.perm[k];
                        phase = PH_STEP;
                    } else {
                        reserve = false;
                    }
                }
                if (phase != PH_STEP) {
                    const unsigned int k = atomicAdd(q.count + 1, 1u) + rl;
                    if (k < n) {
                        slot = q.perm[k];
                        phase = PH_STEP;
                    }
                }
            }
            if (phase == PH_STEP) {
                st.load(q, slot);
                ray.start(p);
            }
        }
        const bool live = ray.phase != PH_IDLE;
        if (!live) drained = true;
        const unsigned int lm = __ballot_sync(0xffffffffu, live);
        if (!lm) break;     // the whole warp is drained
        if constexpr (PREC == 0) {
            // few rays left and none to refill with: eight lanes each to the end
            if (__popc(lm) <= WIDE_RAYS && __all_sync(0xffffffffu, live ? ray.phase == PH_STEP : drained)) {
                const int src = __fns(lm, 0, (lane >> 3) + 1) & 31;  // lane of this group's ray
                double yw[6];
#pragma unroll
                for (int i = 0; i < 6; ++i) yw[i] = __shfl_sync(0xffffffffu, st.y[i], src);
                const double hw = __shfl_sync(0xffffffffu, ray.h, src), tw = __shfl_sync(0xffffffffu, ray.t, src);
                const int vw = __shfl_sync(0xffffffffu, st.vm, src), nw = __shfl_sync(0xffffffffu, ray.steps, src),
                          mw = __shfl_sync(0xffffffffu, (int)ray.metal, src),
                          sw = __shfl_sync(0xffffffffu, slot, src);
                wf_integrate_wide<VAR, MODE, INTEG, PREC>(p, q, wf_smem, yw, vw, hw, tw, nw, mw != 0,
                                                          (lane >> 3) < __popc(lm) ? sw : -1, 0u, 0u);
                break;
            }
        }
        if (!live) continue;
        const bool mirrors = (VAR == V_RADIAL && MODE == M_ORD) || (VAR == V_ANY && st.vm == 0);
        const int status = ray.advance(p, st, lm, mirrors);
        if (status >= 0) {  // ray finished: write back (in the queue's state format), lane becomes idle
            st.store(q, slot);
            q.t[slot] = (double)ray.t;
            q.status[slot] = status;
            q.steps[slot] = ray.steps;
            q.face[slot] = ray.evbest;
            ray.phase = PH_IDLE;
        }
    }
}

// The FP64 integrator is held to 168 registers for three blocks per SM (the wide steps, a call of their own, would
// take 208 and leave two: 3 % slower on a full image); the mixed one to 128 for four -- its FP32 steps are
// latency-bound and gain from the extra warps, while the rare band steps near R1 may spill.
template <int VAR, int MODE, int INTEG, int PREC>
__global__ void __launch_bounds__(128, 3) k_wf_integrate(const __grid_constant__ Params p, const __grid_constant__ Queue q) {
    wf_integrate_body<VAR, MODE, INTEG, PREC>(p, q);
}
template <int VAR, int MODE, int INTEG, int PREC>
__global__ void __launch_bounds__(128, 4) k_wf_integrate_mixed(const __grid_constant__ Params p, Queue q) {
    wf_integrate_body<VAR, MODE, INTEG, PREC>(p, q);
}
template <int VAR, int MODE, int INTEG, int PREC>
constexpr auto wf_integrate_kernel() {
    if constexpr (PREC != 1) return k_wf_integrate<VAR, MODE, INTEG, PREC>;
    else return k_wf_integrate_mixed<VAR, MODE, INTEG, PREC>;
}
// Rays reserved for the long-ray blocks: reserve_per_thread for each of their threads; FP64 Fermat form, where a
// ray takes eight: reserve_per_thread for each ray that they advance at a time, four times that in a render of more than
// 2^26 samples, whose bulk lasts as long as four of the slowest rays one after the other (integration of twelve views of
// 1920 x 1080 x 4, 99.5 M samples: one 651, four 622, eight 622 ms).  In smaller ones the reserved rays end last, the
// other SMs idle: twelve views of 1920 x 1080 x 2 one 348, four 350 ms; 960 x 540 x 4 one 183, four 201; 300 x 168 one 13.3,
// four 25.6; 96 x 54 one 6.0, four 15.7; images 481 x 271 x 3 one 58.8, four 70.0, 1920 x 1080 x 4 one 188, four 209.
inline unsigned int long_ray_reserve(const Params &p, int prec, int packet, long long samples) {
    const int per_block = prec == 0 ? (samples > (1LL << 26) ? 4 : 1) * (packet / WIDE_LANES) : packet;
    return (unsigned int)(p.long_ray_blocks * per_block * p.reserve_per_thread);
}
// the kernel's precision index from the handle's settings
inline int wf_prec(const Params &p) { return p.precision ? 1 : p.formulation ? 2 : 0; }
// Launch the persistent integrator over the sorted queue: exactly the resident grid.
template <int VAR, int MODE, int INTEG, int PREC>
cudaError_t launch_wf_integrate(const Params &p, const Queue &q, int packet, int sms, cudaStream_t st) {
    constexpr auto kern = wf_integrate_kernel<VAR, MODE, INTEG, PREC>();
    const size_t smem = (size_t)WfStepper<VAR, MODE, INTEG, PREC>::SMEM_PER_THREAD * packet;
    int nb = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, packet, smem);
    if (e != cudaSuccess) return e;
    kern<<<(nb > 0 ? nb : 1) * sms, packet, smem, st>>>(p, q);
    return cudaGetLastError();
}

// Exit of queue slot k: refraction into vacuum at the crossed face, the Eq. 12 factor of the exit face
// times the stored factor of the entry face, room lookup.  d_cam: the camera ray (kept as the
// direction of rays that do not leave).
__device__ __forceinline__ void exit_slot(const Params &p, int mode, const Queue &q, unsigned int k, const double d_cam[3],
                                          cloak_record &rec, float rgb[3]) {
    double y[6];
    get_state(p.precision != 0, q, k, y);
    int status = q.status[k];
    rec.mode = mode;
    rec.tile_id = -1;
    rec.weight = 0.0;
    rec.steps = q.steps[k];
    rec.tof = q.t[k];
    rgb[0] = rgb[1] = rgb[2] = 0.f;
    if (status == CLOAK_RAY_EXITED || status == CLOAK_RAY_HIT_METAL_EXITED) {
        double x[3] = {y[0], y[1], y[2]}, nrm[3], eo, ee, c[3], kk[3];
        face_normal(q.face[k], x, nrm);
        local_material(p, x, eo, ee, c);
        if (p.formulation) set_vec(kk, y + 3);  // the Hamiltonian state carries the wave vector
        else wave_from_velocity(mode, eo, ee, c, y + 3, kk);
        double kn = dot3(kk, nrm), kt[3];
        for (int a = 0; a < 3; ++a) kt[a] = kk[a] - kn * nrm[a];
        double kt2 = dot3(kt, kt);
        set_vec(rec.exit_pos, x);
        if (kt2 > 1.0) {
            rec.status = CLOAK_RAY_TIR;
            set_vec(rec.exit_dir, d_cam);
        } else {
            double qn = sqrt(1.0 - kt2), dout[3], mdout[3];
            for (int a = 0; a < 3; ++a) {
                dout[a] = fma(qn, nrm[a], kt[a]);
                mdout[a] = -dout[a];
            }
            double tin = exit_factor(p, mode, eo, ee, c, nrm, mdout, qn);
            rec.weight = tin * q.w_out[k];
            rec.status = status;
            set_vec(rec.exit_dir, dout);
            rec.tile_id = room_hit(p, x, dout, rgb);
        }
    } else {  // STEP_LIMIT or SINGULAR
        rec.status = status;
        rec.exit_pos[0] = y[0]; rec.exit_pos[1] = y[1]; rec.exit_pos[2] = y[2];
        set_vec(rec.exit_dir, d_cam);
    }
}

template <int VAR, int MODE>
__global__ void __launch_bounds__(128) k_wf_exit(Params p, int spp, unsigned long long seed, Queue q,
                                                 float4 *samples, cloak_record *recs) {
    const unsigned int n = q.count[0];
    for (unsigned int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        if (q.key[k] < 0) continue;  // finished before the integration (learned surrogate)
        long long idx = q.id[k];
        long long pix = idx / spp;
        int s = (int)(idx - pix * spp);
        int i = (int)(pix % p.W), j = (int)(pix / p.W);
        double o[3], d[3];
        camera_ray(p, i, j, s, spp, seed, o, d);
        cloak_record rec;
        float rgb[3];
        exit_slot(p, MODE, q, k, d, rec, rgb);
        store_sample(samples, recs, idx, rec, rgb);
    }
}

__global__ void k_wf_resolve(int npix, int spp, const float4 *samples, float4 *out);

}  // namespace ck

namespace ck {

template <int V, int M, int I, int PREC>
static cudaError_t wavefront_vmip(const Params &p, int spp, unsigned long long seed, const Queue &q, float4 *samples,
                                 cloak_record *recs, int packet, cudaStream_t st, cudaEvent_t *ev, const WfHook *hook) {
    long long n = (long long)p.W * p.Hp * spp;
    const int bs = 128;
    k_wf_entry<V, M><<<(unsigned)((n + bs - 1) / bs), bs, 0, st>>>(p, spp, seed, q, samples, recs);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (hook && (e = hook->fn(hook->ctx, q, st)) != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int pk = packet > 0 ? packet : 128;
    // the slowest rays go to the warps of LONG_RAY_BLOCKS blocks that have their SMs to themselves
    k_wf_sort_scan<<<1, 32, 0, st>>>(q, NBINS, long_ray_reserve(p, PREC, pk, n));
    k_wf_sort_scatter<<<sms * 8, 256, 0, st>>>(q);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (ev) cudaEventRecord(ev[1], st);
    Params pl = p;
    pl.dedicated_blocks = p.long_ray_blocks;
    if ((e = launch_wf_integrate<V, M, I, PREC>(pl, q, pk, sms, st)) != cudaSuccess) return e;
    if (ev) cudaEventRecord(ev[2], st);
    k_wf_exit<V, M><<<sms * 16, 128, 0, st>>>(p, spp, seed, q, samples, recs);
    e = cudaGetLastError();
    if (ev) cudaEventRecord(ev[3], st);
    return e;
}

template <int V, int M, int I>
static cudaError_t wavefront_vmi(const Params &p, int spp, unsigned long long seed, const Queue &q, float4 *samples,
                                 cloak_record *recs, int packet, cudaStream_t st, cudaEvent_t *ev, const WfHook *hook) {
    const int prec = wf_prec(p);
    if (prec == 1) return wavefront_vmip<V, M, I, 1>(p, spp, seed, q, samples, recs, packet, st, ev, hook);
    if constexpr (V != V_TEST) {
        if (prec == 2) return wavefront_vmip<V, M, I, 2>(p, spp, seed, q, samples, recs, packet, st, ev, hook);
    }
    return wavefront_vmip<V, M, I, 0>(p, spp, seed, q, samples, recs, packet, st, ev, hook);
}

template <int V>
cudaError_t launch_wavefront_v(const Params &p, int mode, int spp, unsigned long long seed, const Queue &q,
                               float4 *samples, cloak_record *recs, int packet, cudaStream_t st, cudaEvent_t *ev,
                               const WfHook *hook) {
    if (mode == M_ORD && p.integ == I_RK4)
        return wavefront_vmi<V, M_ORD, I_RK4>(p, spp, seed, q, samples, recs, packet, st, ev, hook);
    if (mode == M_ORD && p.integ == I_DP45)
        return wavefront_vmi<V, M_ORD, I_DP45>(p, spp, seed, q, samples, recs, packet, st, ev, hook);
    if (mode == M_EXT && p.integ == I_RK4)
        return wavefront_vmi<V, M_EXT, I_RK4>(p, spp, seed, q, samples, recs, packet, st, ev, hook);
    if (mode == M_EXT && p.integ == I_DP45)
        return wavefront_vmi<V, M_EXT, I_DP45>(p, spp, seed, q, samples, recs, packet, st, ev, hook);
    return cudaErrorInvalidValue;
}

#define CK_INSTANTIATE_WAVEFRONT(V)                                                                        \
    template cudaError_t launch_wavefront_v<V>(const Params &, int, int, unsigned long long, const Queue &, \
                                               float4 *, cloak_record *, int, cudaStream_t, cudaEvent_t *, const WfHook *);

}  // namespace ck
