// integrator.cuh -- the persistent integration kernel of the wavefront schedule, templated on a
// stepper that fixes the arithmetic:
//
//   Stepper64     FP64 throughout (the arithmetic of the plain path, step for step).
//   StepperMixed  right-hand sides of Eq. 2 / Eq. 8 and the stage combinations in FP32; the state
//                 (x, v) accumulated as float-float (TwoSum, Knuth 1969), so rounding does not build
//                 up over thousands of steps, and stage positions kept as float-float so r - R1 is
//                 formed without cancellation; whole steps in FP64 where r < R1 + 0.02 (where
//                 f -> 0); step control in FP32 on the part of the embedded error estimate that
//                 exceeds its own FP32 rounding bound (the estimate is a difference of nearly equal
//                 stage combinations, so without this the controller would chase rounding noise).
//
//   StepperMixed with the band in double-float (CLOAK_MIXED_FF): the steps within the band are taken
//                 in double-float (pairs of FP32 numbers, ~48 bits, dfloat.cuh) instead of FP64.
//
// Each lane owns one queued ray and refills from the queue when it finishes.  Every loop iteration
// runs ONE uniform step evaluation for all lanes; the surface-crossing search (bisection prefix,
// then Illinois regula falsi, or Newton steps: Lane below) reuses that slot with a trial size.
#pragma once

#include "dfloat.cuh"
#include "physics.cuh"

namespace ck {

// ------------------------------------------------------------------ FP64 steppers
// What the FP64 steppers share: state, trial end point, event functions, metal mirror.
template <int INTEG>
struct State64 {
    typedef double real;
    static constexpr bool FP64 = true;
    double y[6], y1[6], e6[6];
    bool need_k1;
    int vm;  // 2 * variant + mode when VAR = MODE = V_ANY

    // DP5(4) step control (physics.cuh: dp_control); fac is the next-step factor
    __device__ __forceinline__ bool control(double tol, double &fac) const { return dp_control(y, y1, e6, tol, fac); }
    __device__ __forceinline__ double chord(const Params &p) const {
        if (!chord_near(s64_truncate(y[0]), s64_truncate(y[1]), s64_truncate(y1[0]), s64_truncate(y1[1]), p.R1f)) return 0.0;
        return metal_chord(y[0], y[1], y1[0], y1[1], p.R1sq);
    }
    __device__ __forceinline__ double g_start(const Params &p, int ev) const { return event_g(p, ev, y); }
    __device__ __forceinline__ double g_end(const Params &p, int ev) const { return event_g(p, ev, y1); }
    __device__ __forceinline__ double g_end_rr(const Params &p, int ev) const { return event_g(p, ev, rr, y1[2]); }
    double rr;  // r^2 at y1, where the step leaves it (DP5(4) of the Fermat form)
    // surfaces behind the end point: bit ev is set iff event_g(ev, y1) > 0, decided by integer comparisons; none is
    // where the end point is NaN (a fixed RK4 step that lands on r = R1 exactly: no step control rejects it)
    template <bool RR>
    __device__ __forceinline__ unsigned int crossed_rr(const Params &p, int nev) const {
        const double r2 = RR ? rr : fma(y1[0], y1[0], __dmul_rn(y1[1], y1[1])), az = s64_abs(y1[2]);
        unsigned int m = 0;
        if (s64_gt_pos(r2, p.R2sq)) m |= 1u << EV_LAT;
        if (s64_gt_pos(az, p.halfH)) m |= __double2hiint(y1[2]) < 0 ? 1u << EV_BOT : 1u << EV_TOP;
        if (nev == 4 && s64_gt_pos(p.R1sq, r2)) m |= 1u << EV_METAL;
        return m;
    }
    __device__ __forceinline__ unsigned int crossed(const Params &p, int nev) const { return crossed_rr<false>(p, nev); }
    // d/ds of the event function at the end of the last trial step of size s, with the end point's
    // derivative taken as the flow's, f(y1) (position part): the Newton slope of the crossing search
    __device__ __forceinline__ double g_rate(int ev) const { return event_dg(ev, y1, y1 + 3); }
    // the same at the start of the step, from f(y)
    __device__ __forceinline__ double g_rate_start(int ev) const { return event_dg(ev, y, y + 3); }
    __device__ __forceinline__ void take_crossing() {
#pragma unroll
        for (int i = 0; i < 6; ++i) y[i] = y1[i];
        need_k1 = true;
    }
    __device__ __forceinline__ void mirror() {  // Sect. 4: single mirror ray at the metal cylinder
        double r = hypot(y[0], y[1]), nm0 = y[0] / r, nm1 = y[1] / r;
        double vn = y[3] * nm0 + y[4] * nm1;
        y[3] -= 2.0 * vn * nm0;
        y[4] -= 2.0 * vn * nm1;
        need_k1 = true;
    }
    // after a change of y from outside
    __device__ __forceinline__ void begin() { need_k1 = true; }
    // final state into queue slot k (FP64 format)
    template <typename Q>
    __device__ __forceinline__ void store(const Q &q, int k) const {
        q.x[k] = y[0]; q.y[k] = y[1]; q.z[k] = y[2];
        q.vx[k] = y[3]; q.vy[k] = y[4]; q.vz[k] = y[5];
    }
};

// Fermat form: the compact steps, stages in shared memory (bind)
template <int VAR, int MODE, int INTEG>
struct Stepper64 : State64<INTEG> {
    using B = State64<INTEG>;
    using B::need_k1;
    using B::vm;
    using B::y;
    using B::y1;
    using B::e6;
    using B::rr;
    __device__ __forceinline__ unsigned int crossed(const Params &p, int nev) const {
        return B::template crossed_rr<INTEG == I_DP45>(p, nev);
    }
    __device__ __forceinline__ double g_end(const Params &p, int ev) const {
        return INTEG == I_DP45 ? B::g_end_rr(p, ev) : B::g_end(p, ev);
    }
    static constexpr int SMEM_PER_THREAD = INTEG == I_DP45 ? DP_SLOTS * (int)sizeof(double) : 0;
    double *kb;
    int ks;
    __device__ __forceinline__ void bind(double *smem) {
        kb = smem + threadIdx.x;
        ks = blockDim.x;
    }
    // state of queue slot k; the first stage comes with it when the entry kernel computed it
    template <typename Q>
    __device__ __forceinline__ void load(const Q &q, int k) {
        y[0] = q.x[k]; y[1] = q.y[k]; y[2] = q.z[k];
        y[3] = q.vx[k]; y[4] = q.vy[k]; y[5] = q.vz[k];
        const double a0 = q.ax[k];
        need_k1 = s64_isnan(a0);
        if (INTEG == I_DP45 && !need_k1) {
            kb[0] = y[3]; kb[ks] = y[4]; kb[2 * ks] = y[5];
            kb[3 * ks] = a0; kb[4 * ks] = q.ay[k]; kb[5 * ks] = q.az[k];
        }
    }
    template <int V, int M>
    __device__ __forceinline__ void eval_medium(const Params &p, double s, bool first) {
        if (INTEG == I_RK4) rk4_fermat<V, M>(p, y, s, y1);
        else dp45_fermat<V, M>(p, y, s, first, kb, ks, y1, e6, rr);
    }
    // lanes: the lanes of the warp that evaluate with this one; whole: the error estimate and the derivative at the end
    // are wanted too (StepperHam on the plain path; the others form them in any case)
    __device__ __forceinline__ void eval(const Params &p, double s, unsigned int lanes, bool) {
        const bool first = INTEG == I_DP45 && __any_sync(lanes, need_k1);
        if (VAR != V_ANY) {
            eval_medium<VAR, MODE>(p, s, first);
        } else {
            switch (vm) {
            case 0: eval_medium<V_RADIAL, M_ORD>(p, s, first); break;
            case 1: eval_medium<V_RADIAL, M_EXT>(p, s, first); break;
            case 2: eval_medium<V_AZIMUTHAL, M_ORD>(p, s, first); break;
            default: eval_medium<V_AZIMUTHAL, M_EXT>(p, s, first); break;
            }
        }
        need_k1 = false;
    }
    __device__ __forceinline__ void take_step() {
#pragma unroll
        for (int i = 0; i < 6; ++i) y[i] = y1[i];
        if (INTEG == I_DP45) {
#pragma unroll
            for (int i = 0; i < 6; ++i) kb[i * ks] = kb[(36 + i) * ks];  // first stage of the next step (FSAL)
        }
    }
};

// ------------------------------------------------------------------ eight lanes per ray
// The same steps with a ray on the eight lanes of a group (four rays per warp), for warps that have few rays
// left and for calls with few rays.  An FP64 instruction blocks its warp for 64 cycles however many lanes take
// part, and a warp alone has no other to fill them, so what counts there is instructions per step, not per ray.
// Lane l keeps component l of the stages (lanes 6 and 7 follow along): each term of a stage combination is one FMA
// instead of six, the scaled tableau is formed a column per lane, the step control checks a component per lane; the
// right-hand side and the crossing search run alike on all lanes of the group on copies of the state.  Terms and
// roundings are those of the narrow steps in their order: the results are the same bit for bit.  One ray alone, one
// thread -> eight lanes, per DP5(4) step: azimuthal extraordinary 13.7 -> 8.9 us, azimuthal ordinary 14.2 -> 9.5,
// radial extraordinary 15.5 -> 11; per RK4 step 5.8 -> 5.2.  (Independent products of the right-hand side on
// different lanes, 1912 instead of 4060 instructions per step, took as long: what the FP64 instructions saved went
// to shuffles.)
// Scaled tableau rows of stages 2 .. 7 and of the error estimate: columns 0 .. 5 the coefficients of k1 .. k6
// without the row's last one, which is in column 7.
static __constant__ double c_dp_wide[7][8] = {
    {0, 0, 0, 0, 0, 0, 0, DP::a21},
    {DP::a31, 0, 0, 0, 0, 0, 0, DP::a32},
    {DP::a41, DP::a42, 0, 0, 0, 0, 0, DP::a43},
    {DP::a51, DP::a52, DP::a53, 0, 0, 0, 0, DP::a54},
    {DP::a61, DP::a62, DP::a63, DP::a64, 0, 0, 0, DP::a65},
    {DP::b1, 0, DP::b3, DP::b4, DP::b5, 0, 0, DP::b6},
    {DP::e1, 0, DP::e3, DP::e4, DP::e5, DP::e6, 0, DP::e7}};
constexpr int WIDE_LANES = 8, WIDE_RAYS = 32 / WIDE_LANES;

template <int VAR, int MODE, int INTEG>
struct StepperWide : State64<INTEG> {
    using B = State64<INTEG>;
    using B::need_k1;
    using B::vm;
    using B::y;
    using B::y1;
    using B::rr;
    __device__ __forceinline__ unsigned int crossed(const Params &p, int nev) const {
        return B::template crossed_rr<INTEG == I_DP45>(p, nev);
    }
    __device__ __forceinline__ double g_end(const Params &p, int ev) const {
        return INTEG == I_DP45 ? B::g_end_rr(p, ev) : B::g_end(p, ev);
    }
    static constexpr int SMEM_PER_THREAD = INTEG == I_DP45 ? 14 * (int)sizeof(double) : 0;
    double *tab;  // this group's scaled tableau (7 rows of 8, ks doubles apart), then the tableau itself
    int ks, l;    // l: lane of the group
    unsigned int grp;  // the group's lanes
    double yo, y1o, eo, k1o, k7o;

    __device__ __forceinline__ void bind(double *smem) {
        const int lane = threadIdx.x & 31;
        l = lane & (WIDE_LANES - 1);
        grp = 0xffu << (lane - l);
        tab = smem + (threadIdx.x - l);
        ks = blockDim.x;
        if (INTEG == I_DP45) {
#pragma unroll
            for (int r = 0; r < 7; ++r) tab[(7 + r) * ks + l] = c_dp_wide[r][l];
        }
    }
    __device__ __forceinline__ double own(const double a[6]) const {
        return l == 0 ? a[0] : l == 1 ? a[1] : l == 2 ? a[2] : l == 3 ? a[3] : l == 4 ? a[4] : a[5];
    }
    __device__ __forceinline__ double from(double a, int lane) const { return __shfl_sync(grp, a, lane, WIDE_LANES); }
    __device__ __forceinline__ void begin() {
        yo = own(y);
        need_k1 = true;
    }
    template <typename Q>
    __device__ __forceinline__ void load(const Q &q, int k) {
        y[0] = q.x[k]; y[1] = q.y[k]; y[2] = q.z[k];
        y[3] = q.vx[k]; y[4] = q.vy[k]; y[5] = q.vz[k];
        begin();
    }
    // this lane's component of the right-hand side at the point whose components are t; g: all of the point's
    template <int V, int M>
    __device__ __forceinline__ double derivative(const Params &p, double t, double g[6]) {
        g[0] = from(t, 0); g[1] = from(t, 1); g[2] = from(t, 2);
        g[3] = from(t, 3); g[4] = from(t, 4); g[5] = from(t, 5);
        double a[3];
        accel64<V, M>(p.R1, g[0], g[1], g[3], g[4], g[5], a[0], a[1], a[2], rr);
        return l == 0 ? g[3] : l == 1 ? g[4] : l == 2 ? g[5] : l == 3 ? a[0] : l == 4 ? a[1] : a[2];
    }
    template <int V, int M>
    __device__ __forceinline__ void eval_medium(const Params &p, double h) {
        if constexpr (V == V_TEST || (V == V_RADIAL && M == M_ORD)) {  // straight lines
            if (INTEG == I_RK4) {
                rk4_fermat<V, M>(p, y, h, y1);
            } else {
                dp45_fermat<V, M>(p, y, h, false, nullptr, 0, y1, B::e6, rr);
                eo = own(B::e6);
            }
            y1o = own(y1);
        } else if constexpr (INTEG == I_RK4) {
            double acc = 0.0, t = yo, k = 0.0, g[6];
            const double hh = 0.5 * h;
#pragma unroll 1
            for (int s = 0; s < 4; ++s) {
                k = derivative<V, M>(p, t, g);
                if (s == 3) break;
                acc = s == 0 ? k : fma(2.0, k, acc);
                t = fma(s < 2 ? hh : h, k, yo);
            }
            y1o = fma(h * (1.0 / 6.0), acc + k, yo);
#pragma unroll
            for (int i = 0; i < 6; ++i) y1[i] = from(y1o, i);
        } else {
            // the tableau times h, a column per lane
#pragma unroll
            for (int r = 0; r < 7; ++r) {
                const double c = tab[(7 + r) * ks + l];
                const bool zero = s64_is_zero(c);
                tab[r * ks + l] = s64_clear(zero, s64_mul(h, s64_nonzero(zero, c)));
            }
            __syncwarp(grp);
            // stages not known yet enter with a zero coefficient, so they have to be finite
            double k1 = need_k1 ? 0.0 : k1o, k2 = 0.0, k3 = 0.0, k4 = 0.0, k5 = 0.0, k6 = 0.0, k = k1, t = yo;
            const double *row = tab;
            if (!need_k1) t = fma(row[7], k, yo);
#pragma unroll 1
            for (int s = need_k1 ? 1 : 2; s < 8; ++s) {
                row = tab + (s - 1) * ks;
                double pre = s == 7 ? 0.0 : yo;
                if (s > 1) pre = fma(row[1], k2, fma(row[0], k1, pre));
                if (s > 3) pre = fma(row[3], k4, fma(row[2], k3, pre));
                if (s > 5) pre = fma(row[5], k6, fma(row[4], k5, pre));
                y1o = t;
                k = derivative<V, M>(p, t, y1);
                k1 = s == 1 ? k : k1;
                k2 = s == 2 ? k : k2;
                k3 = s == 3 ? k : k3;
                k4 = s == 4 ? k : k4;
                k5 = s == 5 ? k : k5;
                k6 = s == 6 ? k : k6;
                t = fma(row[7], k, pre);
            }
            k1o = k1;
            k7o = k;
            eo = t;
            __syncwarp(grp);  // the table has been read
        }
        need_k1 = false;
    }
    __device__ __forceinline__ void eval(const Params &p, double h, unsigned int, bool) {
        if (VAR != V_ANY) {
            eval_medium<VAR, MODE>(p, h);
        } else {
            switch (vm) {
            case 0: eval_medium<V_RADIAL, M_ORD>(p, h); break;
            case 1: eval_medium<V_RADIAL, M_EXT>(p, h); break;
            case 2: eval_medium<V_AZIMUTHAL, M_ORD>(p, h); break;
            default: eval_medium<V_AZIMUTHAL, M_EXT>(p, h); break;
            }
        }
    }
    // dp_control, a component per lane
    __device__ __forceinline__ bool control(double tol, double &fac) const {
        const double sc = fma(tol, fmax(s64_abs(yo), s64_abs(y1o)), tol), ae = s64_abs(eo);
        bool ok = true, bad = false, le = s64_bits(ae) <= s64_bits(sc);
        float fe = __fdividef(s64_to_float(ae, ok), s64_to_float(sc, ok));
        if (!ok) {
            bad = ae != ae;
            le = ae <= sc;
            fe = __fdividef((float)ae, (float)sc);
        }
        const bool acc = __all_sync(grp, le);
        if (__any_sync(grp, bad)) { fac = 0.2; return false; }
        fe = fmaxf(fe, 0.f);  // NaN (infinite over infinite) counts for nothing, as in dp_control
#pragma unroll
        for (int o = WIDE_LANES / 2; o; o >>= 1) fe = fmaxf(fe, __shfl_xor_sync(grp, fe, o));
        fac = dp_factor(fe);
        return acc;
    }
    __device__ __forceinline__ void take_step() {
#pragma unroll
        for (int i = 0; i < 6; ++i) y[i] = y1[i];
        yo = y1o;
        k1o = k7o;  // first stage of the next step (FSAL)
    }
    __device__ __forceinline__ void take_crossing() {
        B::take_crossing();
        begin();
    }
    __device__ __forceinline__ void mirror() {
        B::mirror();
        begin();
    }
};

// Hamiltonian form: state (x, k), stages in registers
template <int VAR, int MODE, int INTEG>
struct StepperHam : State64<INTEG> {
    using B = State64<INTEG>;
    using B::need_k1;
    using B::vm;
    using B::y;
    using B::y1;
    using B::e6;
    static constexpr int SMEM_PER_THREAD = 0;
    double k1[6], k7[6];
    __device__ __forceinline__ void bind(double *) {}
    template <typename Q>
    __device__ __forceinline__ void load(const Q &q, int k) {
        y[0] = q.x[k]; y[1] = q.y[k]; y[2] = q.z[k];
        y[3] = q.vx[k]; y[4] = q.vy[k]; y[5] = q.vz[k];
        need_k1 = true;
    }
    __device__ __forceinline__ void eval(const Params &p, double s, unsigned int, bool whole) {
        if (INTEG == I_RK4) {
            rk4_step<VAR, MODE>(p, y, s, y1, vm);
        } else {
            if (need_k1) rhs_ham<VAR, MODE>(p, y, k1, vm);
            need_k1 = false;
            dp45_step<VAR, MODE>(p, y, k1, s, y1, whole, e6, k7, vm);
        }
    }
    __device__ __forceinline__ double g_rate(int ev) const { return event_dg(ev, y1, k7); }
    __device__ __forceinline__ double g_rate_start(int ev) const { return event_dg(ev, y, k1); }
    __device__ __forceinline__ void take_step() {
#pragma unroll
        for (int i = 0; i < 6; ++i) y[i] = y1[i];
        if (INTEG == I_DP45) {
#pragma unroll
            for (int i = 0; i < 6; ++i) k1[i] = k7[i];  // first stage of the next step (FSAL)
        }
    }
};

// ------------------------------------------------------------------ mixed stepper
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
// (hi, lo) + d  ->  renormalised (hi', lo')
__device__ __forceinline__ void ff_add(float hi, float lo, float d, float &oh, float &ol) {
    float s, e;
    two_sum(hi, d, s, e);
    e += lo;
    oh = s + e;
    ol = e - (oh - s);
}

// dv/dt of Eq. 8 / Eq. 2 in FP32 with the fast reciprocal square root and division.  The position
// comes as float-float (xh + xl, yh + yl) so that u = r - R1 keeps its relative precision close to
// the inner radius: r^2 is formed exactly (TwoProd / TwoSum) and u = (r^2 - R1^2) / (r + R1) with
// R1^2 as float-float (r^2 - R1^2 is then free of cancellation error).
template <int VAR, int MODE>
__device__ __forceinline__ void accel_f32_fixed(float R1, float R1sq_h, float R1sq_l, float K, float invK, float xh,
                                                float xl, float yh, float yl, float vx, float vy, float vz, float &ax,
                                                float &ay, float &az) {
    if (VAR == V_TEST || (VAR == V_RADIAL && MODE == M_ORD)) {
        ax = 0.f; ay = 0.f; az = 0.f;
        return;
    }
    float px = xh * xh, ex = fmaf(xh, xh, -px);
    float py = yh * yh, ey = fmaf(yh, yh, -py);
    float r2h, r2l;
    two_sum(px, py, r2h, r2l);
    r2l += ex + ey + 2.f * (xh * xl + yh * yl);
    float r2 = r2h + r2l;
    float ir = rsqrtf(r2);
    float r = r2 * ir;
    float x = xh + xl, y = yh + yl;
    float cx = x * ir, cy = y * ir;
    float vr = vx * cx + vy * cy;
    float vt = vy * cx - vx * cy;
    float u = __fdividef((r2h - R1sq_h) + (r2l - R1sq_l), r + R1);
    float g = __fdividef(2.f * R1 * ir, u);  // f'/f
    float ar, at, azz;
    if (MODE == M_EXT) {  // the simplified radial terms of accel_fixed
        const float gvr = -g * vr;
        at = gvr * vt;
        const float R1ir2 = R1 * ir * ir;
        if (VAR == V_RADIAL) {
            ar = R1ir2 * ir * (u * vz * vz - r * vt * vt);
            azz = gvr * vz;
        } else {
            ar = -R1ir2 * vt * vt;
            azz = 0.f;
        }
        (void)K; (void)invK;
    } else {
        float hg = 0.5f * g;
        ar = hg * (vt * vt + vz * vz - vr * vr);
        at = -g * vr * vt;
        azz = -g * vr * vz;
    }
    ax = ar * cx - at * cy;
    ay = ar * cy + at * cx;
    az = azz;
}

// dy/dt of the mixed stepper for one medium, inlined.  t: stage point (float), tl: low parts of its x and
// y.  The batch's medium is chosen once per step (StepperMixed::eval), not per right-hand side: each
// medium's step is one contiguous block of code with its seven right-hand sides inline.  (Inlining all
// four media at every one of the seven call sites overflowed the instruction caches -- "no instruction"
// was three quarters of the warps' stall cycles; one out-of-line right-hand side with the switch inside
// paid a call per stage; the switch per step is 2.5 % faster than that, with identical results.)
template <int VAR, int MODE>
__device__ __forceinline__ void rhs_f32(const Params &p, const float t[6], const float tl[2], float d[6]) {
    d[0] = t[3]; d[1] = t[4]; d[2] = t[5];
    accel_f32_fixed<VAR, MODE>(p.R1f, p.R1sq_hf, p.R1sq_lf, p.Kf, p.invKf, t[0], tl[0], t[1], tl[1], t[3], t[4], t[5],
                               d[3], d[4], d[5]);
}

// ------------------------------------------------------------------ double-float steps (the band near R1)
// The same right-hand side and the same Dormand-Prince / RK4 updates as the FP64 path, in double-float.
struct df3 {
    df x, y, z;
};
template <int VAR, int MODE>
__device__ __noinline__ df3 accel_df_call(df R1, df x, df y, df vx, df vy, df vz, int vm) {
    const df unused;  // K and 1/K: the simplified accelerations of accel_fixed do not read them
    df3 a;
    accel<VAR, MODE, df>(R1, unused, unused, x, y, vx, vy, vz, a.x, a.y, a.z, vm);
    return a;
}
// one medium: inline; the batch's any-medium form: one out-of-line copy with the switch inside
template <int VAR, int MODE>
__device__ __forceinline__ void rhs_df(df R1, const df y[6], df d[6], int vm) {
    d[0] = y[3]; d[1] = y[4]; d[2] = y[5];
    if (VAR != V_ANY) {
        const df unused;  // K and 1/K: the simplified accelerations of accel_fixed do not read them
        accel_fixed<VAR, MODE, df>(R1, unused, unused, y[0], y[1], y[3], y[4], y[5], d[3], d[4], d[5]);
    } else {
        const df3 a = accel_df_call<VAR, MODE>(R1, y[0], y[1], y[3], y[4], y[5], vm);
        d[3] = a.x; d[4] = a.y; d[5] = a.z;
    }
}
template <int VAR, int MODE>
__device__ __forceinline__ void rk4_step_df(df R1, const df y[6], df h, df out[6], int vm) {
    df k[6], acc[6], t[6];
    const df hh = h * 0.5f, h6 = h * df(1.0 / 6.0);
    rhs_df<VAR, MODE>(R1, y, k, vm);
#pragma unroll
    for (int i = 0; i < 6; ++i) { acc[i] = k[i]; t[i] = df_fma(hh, k[i], y[i]); }
    rhs_df<VAR, MODE>(R1, t, k, vm);
#pragma unroll
    for (int i = 0; i < 6; ++i) { acc[i] = acc[i] + k[i] * 2.0f; t[i] = df_fma(hh, k[i], y[i]); }
    rhs_df<VAR, MODE>(R1, t, k, vm);
#pragma unroll
    for (int i = 0; i < 6; ++i) { acc[i] = acc[i] + k[i] * 2.0f; t[i] = df_fma(h, k[i], y[i]); }
    rhs_df<VAR, MODE>(R1, t, k, vm);
#pragma unroll
    for (int i = 0; i < 6; ++i) out[i] = df_fma(h6, acc[i] + k[i], y[i]);
}

// The band's steps near R1 (FP64 or double-float), out of line: rare, large, and kept out of the
// instruction stream of the FP32 steps.  Inputs and outputs pass through the caller's local memory.
template <int VAR, int MODE, int INTEG>
__device__ __forceinline__ void band_medium_f64(const Params &p, const double *y, double s, double *yo, double *e,
                                                double *kb, int ks) {
    double rr;
    if (INTEG == I_RK4) rk4_fermat<VAR, MODE>(p, y, s, yo);
    else dp45_fermat<VAR, MODE>(p, y, s, true, kb, ks, yo, e, rr);
}
template <int VAR, int MODE, int INTEG>
__device__ __noinline__ void band_step_f64(const Params &p, const double *y, double s, double *yo, double *e,
                                           double *kb, int ks, int vm) {
    if (VAR != V_ANY) {
        band_medium_f64<VAR, MODE, INTEG>(p, y, s, yo, e, kb, ks);
    } else {
        switch (vm) {
        case 0: band_medium_f64<V_RADIAL, M_ORD, INTEG>(p, y, s, yo, e, kb, ks); break;
        case 1: band_medium_f64<V_RADIAL, M_EXT, INTEG>(p, y, s, yo, e, kb, ks); break;
        case 2: band_medium_f64<V_AZIMUTHAL, M_ORD, INTEG>(p, y, s, yo, e, kb, ks); break;
        default: band_medium_f64<V_AZIMUTHAL, M_EXT, INTEG>(p, y, s, yo, e, kb, ks); break;
        }
    }
}
// a double constant as a double-float pair
#define CK_DF2(c) {(float)(c), (float)((c) - (double)(float)(c))}
// The tableau in double-float (c_dp_a, c_dp_e of the FP64 form)
static __constant__ float2 c_dp_a_df[20] = {CK_DF2(DP::a21), CK_DF2(DP::a31), CK_DF2(DP::a32), CK_DF2(DP::a41),
                                            CK_DF2(DP::a42), CK_DF2(DP::a43), CK_DF2(DP::a51), CK_DF2(DP::a52),
                                            CK_DF2(DP::a53), CK_DF2(DP::a54), CK_DF2(DP::a61), CK_DF2(DP::a62),
                                            CK_DF2(DP::a63), CK_DF2(DP::a64), CK_DF2(DP::a65), CK_DF2(DP::b1),
                                            CK_DF2(DP::b3),  CK_DF2(DP::b4),  CK_DF2(DP::b5),  CK_DF2(DP::b6)};
static __constant__ float2 c_dp_e_df[5] = {CK_DF2(DP::e1), CK_DF2(DP::e3), CK_DF2(DP::e4), CK_DF2(DP::e5),
                                           CK_DF2(DP::e6)};
__device__ __forceinline__ df df_of(float2 v) { return df(v.x, v.y); }
// DP5(4) step of one medium from y, its first stage included: the stages in shared memory (kb: this thread's
// column, ks threads per row) and one copy of the right-hand side in a loop over them, as in dp45_fermat, because
// the seven inlined copies of the unrolled form (3500 instructions per medium) left the mixed kernel's warps
// waiting for instructions.
template <int VAR, int MODE>
__device__ __forceinline__ void dp45_band_df(df R1, const df *y, df h, df *yo, df *e, float2 *kb, int ks) {
    const df unused;
    if constexpr (VAR == V_TEST || (VAR == V_RADIAL && MODE == M_ORD)) {  // straight lines: no band (island)
#pragma unroll
        for (int i = 0; i < 6; ++i) { yo[i] = y[i]; e[i] = unused; }
    } else {
        df t[6], a[3];
        int row = 0;
#pragma unroll 1
        for (int s = 0; s < 7; ++s) {
#pragma unroll
            for (int i = 0; i < 6; ++i) t[i] = y[i];
            const int terms = s < 6 ? s : 5;
            const float2 *k = kb;
#pragma unroll 1
            for (int q = 0; q < terms; ++q) {
                const df c = h * df_of(c_dp_a_df[row + q]);
                df kq[6];
#pragma unroll
                for (int i = 0; i < 6; ++i) kq[i] = df_of(k[i * ks]);
                t[0] = df_fma(c, kq[0], t[0]);
                t[1] = df_fma(c, kq[1], t[1]);
#pragma unroll
                for (int i = 3; i < 6; ++i) t[i] = df_fma(c, kq[i], t[i]);
                if (s == 6) {
                    const df ce = h * df_of(c_dp_e_df[q]);
                    t[2] = df_fma(c, kq[2], t[2]);
#pragma unroll
                    for (int i = 0; i < 6; ++i) e[i] = q == 0 ? ce * kq[i] : df_fma(ce, kq[i], e[i]);
                    if (q == 0) k += 6 * ks;  // no second stage in the solution
                }
                k += 6 * ks;
            }
            row += s;
            accel_fixed<VAR, MODE, df>(R1, unused, unused, t[0], t[1], t[3], t[4], t[5], a[0], a[1], a[2]);
            float2 *ko = kb + 6 * s * ks;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                ko[i * ks] = make_float2(t[3 + i].hi, t[3 + i].lo);
                ko[(3 + i) * ks] = make_float2(a[i].hi, a[i].lo);
            }
        }
        const df c7 = h * df(DP::e7);
#pragma unroll
        for (int i = 0; i < 6; ++i) yo[i] = t[i];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            e[i] = df_fma(c7, t[3 + i], e[i]);
            e[3 + i] = df_fma(c7, a[i], e[3 + i]);
        }
    }
}
template <int VAR, int MODE, int INTEG>
__device__ __noinline__ void band_step_df(float R1h, float R1l, const df *y, float s, df *yo, df *e, float2 *kb, int ks,
                                          int vm) {
    const df R1(R1h, R1l), hs(s, 0.f);
    if (INTEG == I_RK4) {
        rk4_step_df<VAR, MODE>(R1, y, hs, yo, vm);
    } else if (VAR == V_ANY) {  // the batch's medium chosen once per step
        switch (vm) {
        case 0: dp45_band_df<V_RADIAL, M_ORD>(R1, y, hs, yo, e, kb, ks); break;
        case 1: dp45_band_df<V_RADIAL, M_EXT>(R1, y, hs, yo, e, kb, ks); break;
        case 2: dp45_band_df<V_AZIMUTHAL, M_ORD>(R1, y, hs, yo, e, kb, ks); break;
        default: dp45_band_df<V_AZIMUTHAL, M_EXT>(R1, y, hs, yo, e, kb, ks); break;
        }
    } else {
        dp45_band_df<VAR, MODE>(R1, y, hs, yo, e, kb, ks);
    }
}

template <int VAR, int MODE, int INTEG>
struct StepperMixed {
    typedef float real;
    static constexpr bool FP64 = false;
    static constexpr int SMEM_PER_THREAD = INTEG == I_DP45 ? DP_SLOTS * (int)sizeof(double) : 0;  // the band's stages
    double *kb;
    int ks;
    float yh[6], yl[6], k1[6];  // state (float-float) and first stage
    float y1h[6], y1l[6], e6[6], k7[6];
    float n6[6];  // rounding bound of the FP32 error estimate (noise floor)
    bool need_k1;
    int vm;  // 2 * variant + mode when VAR = MODE = V_ANY

    __device__ __forceinline__ void bind(double *smem) {
        kb = smem + threadIdx.x;
        ks = blockDim.x;
    }
    // the queue holds the mixed path's states as float-float pairs: no conversion
    template <typename Q>
    __device__ __forceinline__ void load(const Q &q, int k) {
        const double *a[6] = {q.x, q.y, q.z, q.vx, q.vy, q.vz};
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const float2 v = reinterpret_cast<const float2 *>(a[i])[k];
            yh[i] = v.x;
            yl[i] = v.y;
        }
        need_k1 = true;
    }
    template <typename Q>
    __device__ __forceinline__ void store(const Q &q, int k) const {
        double *a[6] = {q.x, q.y, q.z, q.vx, q.vy, q.vz};
#pragma unroll
        for (int i = 0; i < 6; ++i) reinterpret_cast<float2 *>(a[i])[k] = make_float2(yh[i], yl[i]);
    }
    __device__ __forceinline__ bool island(const Params &p) const {
        if (VAR == V_TEST || (VAR == V_RADIAL && MODE == M_ORD) || (VAR == V_ANY && vm == 0)) return false;
        float x = yh[0] + yl[0], y = yh[1] + yl[1];
        const float lim = p.band_limf;  // 0 without a band
        if (!(lim > 0.f)) return false;
        return x * x + y * y < lim * lim;
    }
    // stage point y + d: x, y as float-float (t, tl), the rest in FP32
    __device__ __forceinline__ void stage(const float d[6], float t[6], float tl[2]) const {
        ff_add(yh[0], yl[0], d[0], t[0], tl[0]);
        ff_add(yh[1], yl[1], d[1], t[1], tl[1]);
#pragma unroll
        for (int i = 2; i < 6; ++i) t[i] = yh[i] + (yl[i] + d[i]);
    }
    __device__ __forceinline__ void eval(const Params &p, float s, unsigned int, bool) {
        if (p.band_df && island(p)) {  // double-float step from the float-float state
            df y[6], yo[6], e[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) y[i] = df(yh[i], yl[i]);
            const df R1(p.R1);
            band_step_df<VAR, MODE, INTEG>(R1.hi, R1.lo, y, s, yo, e, reinterpret_cast<float2 *>(kb), ks, vm);
            if (INTEG == I_DP45) {
#pragma unroll
                for (int i = 0; i < 6; ++i) { e6[i] = e[i].hi + e[i].lo; n6[i] = 0.f; }
            }
#pragma unroll
            for (int i = 0; i < 6; ++i) { y1h[i] = yo[i].hi; y1l[i] = yo[i].lo; }
            need_k1 = true;
            return;
        }
        if (island(p)) {  // FP64 step from the float-float state
            double y[6], yo[6], e[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) y[i] = (double)yh[i] + (double)yl[i];
            band_step_f64<VAR, MODE, INTEG>(p, y, (double)s, yo, e, kb, ks, vm);
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                y1h[i] = (float)yo[i];
                y1l[i] = (float)(yo[i] - (double)y1h[i]);
                if (INTEG == I_DP45) { e6[i] = (float)e[i]; n6[i] = 0.f; }
            }
            need_k1 = true;
            return;
        }
        if (VAR == V_ANY) {
            switch (vm) {
            case 0: eval_f32<V_RADIAL, M_ORD>(p, s); break;
            case 1: eval_f32<V_RADIAL, M_EXT>(p, s); break;
            case 2: eval_f32<V_AZIMUTHAL, M_ORD>(p, s); break;
            default: eval_f32<V_AZIMUTHAL, M_EXT>(p, s); break;
            }
        } else {
            eval_f32<VAR, MODE>(p, s);
        }
    }
    // the FP32 step (RK4, or DP5(4) with its error estimate) of medium V2 / M2 from the float-float state
    template <int V2, int M2>
    __device__ __forceinline__ void eval_f32(const Params &p, float s) {
        float t[6], tl[2], d[6], k2[6], k3[6], k4[6], k5[6], k6[6];
        if (INTEG == I_RK4) {
            float acc[6], kk[6];
            const float z6[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            stage(z6, t, tl);
            rhs_f32<V2, M2>(p, t, tl, kk);
#pragma unroll
            for (int i = 0; i < 6; ++i) { acc[i] = kk[i]; d[i] = 0.5f * s * kk[i]; }
            stage(d, t, tl);
            rhs_f32<V2, M2>(p, t, tl, kk);
#pragma unroll
            for (int i = 0; i < 6; ++i) { acc[i] = fmaf(2.f, kk[i], acc[i]); d[i] = 0.5f * s * kk[i]; }
            stage(d, t, tl);
            rhs_f32<V2, M2>(p, t, tl, kk);
#pragma unroll
            for (int i = 0; i < 6; ++i) { acc[i] = fmaf(2.f, kk[i], acc[i]); d[i] = s * kk[i]; }
            stage(d, t, tl);
            rhs_f32<V2, M2>(p, t, tl, kk);
#pragma unroll
            for (int i = 0; i < 6; ++i) ff_add(yh[i], yl[i], s * (1.f / 6.f) * (acc[i] + kk[i]), y1h[i], y1l[i]);
            return;
        }
        if (need_k1) {
            const float z6[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            stage(z6, t, tl);
            rhs_f32<V2, M2>(p, t, tl, k1);
            need_k1 = false;
        }
        const float a21 = (float)DP::a21, a31 = (float)DP::a31, a32 = (float)DP::a32, a41 = (float)DP::a41,
                    a42 = (float)DP::a42, a43 = (float)DP::a43, a51 = (float)DP::a51, a52 = (float)DP::a52,
                    a53 = (float)DP::a53, a54 = (float)DP::a54, a61 = (float)DP::a61, a62 = (float)DP::a62,
                    a63 = (float)DP::a63, a64 = (float)DP::a64, a65 = (float)DP::a65, b1 = (float)DP::b1,
                    b3 = (float)DP::b3, b4 = (float)DP::b4, b5 = (float)DP::b5, b6 = (float)DP::b6,
                    c1 = (float)DP::e1, c3 = (float)DP::e3, c4 = (float)DP::e4, c5 = (float)DP::e5,
                    c6 = (float)DP::e6, c7 = (float)DP::e7;
#pragma unroll
        for (int i = 0; i < 6; ++i) d[i] = s * (a21 * k1[i]);
        stage(d, t, tl);
        rhs_f32<V2, M2>(p, t, tl, k2);
#pragma unroll
        for (int i = 0; i < 6; ++i) d[i] = s * (a31 * k1[i] + a32 * k2[i]);
        stage(d, t, tl);
        rhs_f32<V2, M2>(p, t, tl, k3);
#pragma unroll
        for (int i = 0; i < 6; ++i) d[i] = s * (a41 * k1[i] + a42 * k2[i] + a43 * k3[i]);
        stage(d, t, tl);
        rhs_f32<V2, M2>(p, t, tl, k4);
#pragma unroll
        for (int i = 0; i < 6; ++i) d[i] = s * (a51 * k1[i] + a52 * k2[i] + a53 * k3[i] + a54 * k4[i]);
        stage(d, t, tl);
        rhs_f32<V2, M2>(p, t, tl, k5);
#pragma unroll
        for (int i = 0; i < 6; ++i) d[i] = s * (a61 * k1[i] + a62 * k2[i] + a63 * k3[i] + a64 * k4[i] + a65 * k5[i]);
        stage(d, t, tl);
        rhs_f32<V2, M2>(p, t, tl, k6);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            float dd = s * (b1 * k1[i] + b3 * k3[i] + b4 * k4[i] + b5 * k5[i] + b6 * k6[i]);
            ff_add(yh[i], yl[i], dd, y1h[i], y1l[i]);
            t[i] = y1h[i];
        }
        tl[0] = y1l[0];
        tl[1] = y1l[1];
#pragma unroll
        for (int i = 2; i < 6; ++i) t[i] = y1h[i] + y1l[i];
        rhs_f32<V2, M2>(p, t, tl, k7);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            e6[i] = s * (c1 * k1[i] + c3 * k3[i] + c4 * k4[i] + c5 * k5[i] + c6 * k6[i] + c7 * k7[i]);
            // each k_j carries a relative rounding error of a few FP32 ulps; so does their combination
            n6[i] = 8.f * 5.96e-8f * fabsf(s) *
                    (fabsf(c1 * k1[i]) + fabsf(c3 * k3[i]) + fabsf(c4 * k4[i]) + fabsf(c5 * k5[i]) +
                     fabsf(c6 * k6[i]) + fabsf(c7 * k7[i]));
        }
    }
    __device__ __forceinline__ bool control(float tol, float &fac) const {
        bool acc = true, bad = false;
        float fe = 0.f;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            float sc = tol + tol * fmaxf(fabsf(yh[i]), fabsf(y1h[i]));
            float ae = fmaxf(0.f, fabsf(e6[i]) - n6[i]);  // truncation error above the rounding noise
            if (e6[i] != e6[i]) bad = true;
            if (!(ae <= sc)) acc = false;
            fe = fmaxf(fe, __fdividef(ae, sc));
        }
        if (bad) { fac = 0.2f; return false; }
        fac = fe == 0.f ? 5.f : fminf(5.f, fmaxf(0.2f, 0.9f * __powf(fe, -0.2f)));
        if (!(fe < 3.0e38f)) fac = 0.2f;
        return acc;
    }
    // Event functions with the roots and signs of event_g (r^2 - R2^2, z - H/2, -z - H/2, R1^2 - r^2) from
    // the float-float position: r^2 is formed exactly (products by FMA, sums by TwoSum) and the surface
    // constants are float-float, so g keeps its precision where it is small -- next to the root, where the
    // crossing search reads it.  (In plain FP32, g carries an absolute error ~1e-7; on the short chords of
    // grazing rays, where g changes by little more than that, the crossing moved by up to 1e-4.)
    static __device__ __forceinline__ float gval(const Params &p, int ev, const float h[6], const float l[6]) {
        float r2h, r2l;
        radius_sq(h, l, r2h, r2l);
        // one difference for every surface: lanes of a warp that cross different ones do not diverge
        const bool lat = ev == EV_LAT, metal = ev == EV_METAL, bot = ev == EV_BOT;
        const float ah = lat ? r2h : metal ? p.R1sq_hf : bot ? -h[2] : h[2], bh = lat ? p.R2sq_hf : metal ? r2h : p.halfH_hf;
        const float al = lat ? r2l : metal ? p.R1sq_lf : bot ? -l[2] : l[2], bl = lat ? p.R2sq_lf : metal ? r2l : p.halfH_lf;
        return (ah - bh) + (al - bl);
    }
    static __device__ __forceinline__ void radius_sq(const float h[6], const float l[6], float &r2h, float &r2l) {
        const float px = h[0] * h[0], ex = fmaf(h[0], h[0], -px);
        const float py = h[1] * h[1], ey = fmaf(h[1], h[1], -py);
        two_sum(px, py, r2h, r2l);
        r2l += ex + ey + 2.f * (h[0] * l[0] + h[1] * l[1]);
    }
    __device__ __forceinline__ float chord(const Params &p) const {
        return metal_chord(yh[0] + yl[0], yh[1] + yl[1], y1h[0] + y1l[0], y1h[1] + y1l[1], p.R1sq_hf);
    }
    __device__ __forceinline__ float g_start(const Params &p, int ev) const { return gval(p, ev, yh, yl); }
    __device__ __forceinline__ float g_end(const Params &p, int ev) const { return gval(p, ev, y1h, y1l); }
    __device__ __forceinline__ unsigned int crossed(const Params &p, int nev) const {
        // gval of the four surfaces in straight code, r^2 formed once
        float r2h, r2l;
        radius_sq(y1h, y1l, r2h, r2l);
        unsigned int m = 0;
        if ((r2h - p.R2sq_hf) + (r2l - p.R2sq_lf) > 0.f) m |= 1u << EV_LAT;
        if ((y1h[2] - p.halfH_hf) + (y1l[2] - p.halfH_lf) > 0.f) m |= 1u << EV_TOP;
        if ((-y1h[2] - p.halfH_hf) + (-y1l[2] - p.halfH_lf) > 0.f) m |= 1u << EV_BOT;
        if (nev == 4 && (p.R1sq_hf - r2h) + (p.R1sq_lf - r2l) > 0.f) m |= 1u << EV_METAL;
        return m;
    }
    __device__ __forceinline__ float g_rate(int) const { return 1.f; }  // the search takes no Newton steps
    __device__ __forceinline__ float g_rate_start(int) const { return 0.f; }
    __device__ __forceinline__ void take_step() {
#pragma unroll
        for (int i = 0; i < 6; ++i) { yh[i] = y1h[i]; yl[i] = y1l[i]; }
        if (INTEG == I_DP45 && !need_k1) {
#pragma unroll
            for (int i = 0; i < 6; ++i) k1[i] = k7[i];
        }
    }
    __device__ __forceinline__ void take_crossing() {
#pragma unroll
        for (int i = 0; i < 6; ++i) { yh[i] = y1h[i]; yl[i] = y1l[i]; }
        need_k1 = true;
    }
    __device__ __forceinline__ void mirror() {
        double y[6];
        state(y);
        double r = hypot(y[0], y[1]), nm0 = y[0] / r, nm1 = y[1] / r;
        double vn = y[3] * nm0 + y[4] * nm1;
        y[3] -= 2.0 * vn * nm0;
        y[4] -= 2.0 * vn * nm1;
#pragma unroll
        for (int i = 3; i < 6; ++i) {
            yh[i] = (float)y[i];
            yl[i] = (float)(y[i] - (double)yh[i]);
        }
        need_k1 = true;
    }
    __device__ __forceinline__ void state(double out[6]) const {
#pragma unroll
        for (int i = 0; i < 6; ++i) out[i] = (double)yh[i] + (double)yl[i];
    }
};

// ------------------------------------------------------------------ one lane's ray: steps, crossings, mirror
enum { PH_STEP = 0, PH_CROSS = 1, PH_FINAL = 2, PH_IDLE = 3 };

// Comparisons of step sizes and event values: on the integer pipes for FP64 (each FP64 comparison would take a
// slot of the FP64 unit for the whole warp).  a may be any value, lo and hi are not negative.
__device__ __forceinline__ bool inside(double a, double lo, double hi) {
    return __double_as_longlong(a) > __double_as_longlong(lo) && __double_as_longlong(a) < __double_as_longlong(hi);
}
__device__ __forceinline__ bool inside(float a, float lo, float hi) { return a > lo && a < hi; }
__device__ __forceinline__ bool positive(double a) { return s64_positive(a); }
__device__ __forceinline__ bool positive(float a) { return a > 0.f; }
__device__ __forceinline__ bool le_pos(double a, double b) { return s64_le_pos(a, b); }  // 0 <= a, b, or NaN
__device__ __forceinline__ bool le_pos(float a, float b) { return a <= b; }
__device__ __forceinline__ bool gt_pos(double a, double b) { return s64_gt_pos(a, b); }  // 0 <= a, b, or NaN
__device__ __forceinline__ bool gt_pos(float a, float b) { return a > b; }
__device__ __forceinline__ bool not_positive(double a) { return s64_not_positive(a); }
__device__ __forceinline__ bool not_positive(float a) { return a <= 0.f; }
__device__ __forceinline__ bool not_negative(double a) { return s64_not_negative(a); }
__device__ __forceinline__ bool not_negative(float a) { return a >= 0.f; }
__device__ __forceinline__ bool same(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }
__device__ __forceinline__ bool same(float a, float b) { return a == b; }
// a <= f b for sizes 0 <= a <= b whose ratio is decided to single precision: both divided by b's power of two, so that
// lengths of any scale compare alike
__device__ __forceinline__ bool below(double a, float f, double b) {
    const int e = (s64_hi(b) & 0x7ff00000) - 0x3ff00000;
    const double am = s64_make((uint32_t)max(s64_hi(a) - e, 0), (uint32_t)s64_lo(a));
    return s64_truncate(am) <= f * s64_truncate(s64_make((uint32_t)(s64_hi(b) - e), (uint32_t)s64_lo(b)));
}
__device__ __forceinline__ bool below(float a, float f, float b) { return a <= f * b; }
__device__ __forceinline__ double mag(double a) { return s64_abs(a); }
__device__ __forceinline__ float mag(float a) { return fabsf(a); }

// The ray of one lane: adaptive steps, the search for the surface that a step crosses, the metal mirror.  One
// call of advance evaluates the stepper once, for stepping and searching lanes alike.
// NEWTON: FP64 DP5(4) renders: when the ray moves towards the surface at both ends of the crossing step (one
// crossing inside it), the search takes safeguarded Newton steps on the step function itself, the slope from the
// end point's derivative f(y1), starting from a Newton step off the coarse step's end; otherwise, and for the
// other paths, a bisection prefix and Illinois regula falsi.
// EXACT: the regula falsi quotient as an IEEE division (the plain path) instead of a reciprocal product.
template <typename S, int INTEG, bool NEWTON, bool EXACT>
struct Lane {
    typedef typename S::real R;
    static constexpr float NEWTON_LAST = 1e-6f;
    static constexpr int prefix = bisect_prefix<INTEG>();
    R h, t;
    int steps, phase;
    bool metal;
    // crossing state
    R hs, fac, lo, hi, glo, ghi, sbest, g1[4];
    int ev, evbest, side, it;
    bool newton, fin;
    R snext;
    unsigned int pending;

    __device__ __forceinline__ void reset() {
        phase = PH_IDLE;
        h = t = hs = fac = lo = hi = glo = ghi = sbest = snext = (R)0;
        steps = 0;
        metal = newton = fin = false;
        ev = side = it = 0;
        evbest = -1;
        pending = 0;
    }
    __device__ __forceinline__ void start(const Params &p) {
        h = INTEG == I_RK4 ? (R)p.h_or_tol : (R)1e-3;
        t = 0; steps = 0; metal = false;
        phase = PH_STEP;
    }
    // One evaluation of st for the lanes `lanes` of the warp, which all call this together; mirrors: rays
    // that reach the metal cylinder are mirrored (the others end there).  Returns the ray's status, -1 while
    // it continues.
    __device__ __forceinline__ int advance(const Params &p, S &st, unsigned int lanes, bool mirrors) {
        const int nev = p.R1 > 0.0 ? 4 : 3;
        const R tol = (R)p.h_or_tol;
        const float conv = sizeof(R) == 8 ? (float)CROSS_REL_TOL : 2.4e-7f;  // bracket resolution of the search
        int status = -1;
        if (phase == PH_STEP && (steps >= p.max_steps || (INTEG == I_DP45 && gt_pos((R)1e-14, h))))
            status = CLOAK_RAY_STEP_LIMIT;
        R s = phase == PH_STEP ? h : sbest;
        if (phase == PH_CROSS) {
            // next trial point: Newton (see above), or a bisection prefix, then Illinois regula falsi
            if (newton) s = snext;
            else if (it < prefix) s = (R)0.5 * (lo + hi);
            else if (it - prefix < 60 && ghi > glo)
                s = EXACT ? fma(lo, ghi, -(hi * glo)) / (ghi - glo) : fma(lo, ghi, -(hi * glo)) * rcp_nr(ghi - glo);
            else s = (R)0.5 * (lo + hi);
            if (!inside(s, lo, hi)) s = (R)0.5 * (lo + hi);
        }
        // the lanes that evaluate, where the stepper asks (FP64: its first stage is uniform over them)
        const unsigned int on = S::FP64 ? __ballot_sync(lanes, status < 0) : 0u;
        __syncwarp(lanes);  // a convergence point: keeps the compiler from splitting the evaluation by phase
        if (status >= 0) return status;
        st.eval(p, s, on, !EXACT || phase == PH_STEP);
        bool land = false;
        // mixed: the search for the next pending surface starts at one place (gnew: the surface's value at the end point),
        // which keeps a warp's lanes together: images of 128 x 96 and below 1 to 2 % faster; FP64 RK4 rays 3 % slower
        bool begin = false;
        R gnew = 0;
        if (phase == PH_STEP) {
            ++steps;
            fac = 1;
            bool accept = true;
            if (INTEG == I_DP45) {
                if (!st.control(tol, fac)) {
                    h *= fmin(fac, (R)1);
                    fac = 1;
                    accept = false;
                }
            }
            if (accept) {
                pending = st.crossed(p, nev);
                R sc = 0;
                if (INTEG == I_DP45 && nev == 4 && !(pending & (1u << EV_METAL))) sc = st.chord(p);
                if (positive(sc)) {
                    h *= sc;  // retried: the step's chord passes through the metal cylinder
                } else if (!pending) {
                    st.take_step();
                    t += h;
                    h *= fac;
                } else {
                    // the values at the end point, of the further surfaces only if there are any
                    gnew = st.g_end(p, __ffs(pending) - 1);
                    if (pending & (pending - 1)) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) g1[e] = st.g_end(p, e);
                    }
                    hs = h;
                    sbest = (R)(S::FP64 ? 1e300 : 1e30);  // above any step
                    evbest = -1;
                    newton = false;
                    fin = false;
                    if (S::FP64) search(p, st, gnew);
                    else begin = true;
                    if (NEWTON) {
                        const R d0 = (R)st.g_rate_start(ev), d1 = (R)st.g_rate(ev);
                        if (not_negative(d0) && positive(d1)) {
                            newton = true;
                            R s0 = fma(-ghi, rcp_nr(d1), hs);
                            if (!inside(s0, (R)0, hs)) s0 = hs * (-glo / (ghi - glo));
                            if (!inside(s0, (R)0, hs)) s0 = (R)0.5 * hs;
                            snext = s0;
                        }
                    }
                    phase = PH_CROSS;
                }
            }
        } else if (phase == PH_CROSS) {
            bool done = false;
            R gtol;
            cross_g_tol(p, ev, gtol);
            if (!inside(s, lo, hi)) {
                done = true;
            } else if (NEWTON && newton) {
                // safeguarded Newton: keep the bracket, bisect when the step would leave it
                const R gs = st.g_end(p, ev);
                if (positive(gs)) { hi = s; ghi = gs; } else { lo = s; glo = gs; }
                ++it;
                if (fin || le_pos(mag(gs), gtol)) {
                    // on the surface to rounding, or the trial point of a Newton correction below
                    // NEWTON_LAST x the step: quadratic convergence put it within ~1e-12 of the step
                    lo = s;
                    hi = s;
                    done = true;
                } else {
                    const R dg = (R)st.g_rate(ev);
                    R sn = fma(-gs, rcp_nr(dg), s);
                    if (!inside(sn, lo, hi)) sn = (R)0.5 * (lo + hi);
                    else if (below(mag(sn - s), NEWTON_LAST, hs)) fin = true;
                    snext = sn;
                    if (below(hi - lo, conv, hi) || it >= 100) done = true;
                }
            } else {
                R gs = st.g_end(p, ev);
                if (it < prefix) {
                    if (positive(gs)) { hi = s; ghi = gs; } else { lo = s; glo = gs; }
                } else if (positive(gs)) {
                    hi = s; ghi = gs;
                    if (side == 1) glo *= (R)0.5;
                    side = 1;
                } else {
                    lo = s; glo = gs;
                    if (side == -1) ghi *= (R)0.5;
                    side = -1;
                }
                ++it;
                if (it >= prefix && below(hi - lo, conv, hi)) done = true;
                // or a regula falsi trial point lies on the surface to rounding (Illinois approaches
                // the root from one side, so the far end of the bracket may lag for many iterations)
                if (!done && it > prefix && le_pos(mag(gs), gtol)) {
                    lo = s;
                    hi = s;
                    done = true;
                }
                if (it >= prefix + 200) done = true;
            }
            if (done) {
                R se = ev == EV_METAL ? lo : hi;
                if (inside(se, (R)-1, sbest)) { sbest = se; evbest = ev; }
                pending &= ~(1u << ev);
                if (pending) {
                    newton = false;  // the coarse step's end point is gone: bisection for further surfaces
                    const int e = __ffs(pending) - 1;
                    gnew = e == 0 ? g1[0] : e == 1 ? g1[1] : e == 2 ? g1[2] : g1[3];
                    if (S::FP64) search(p, st, gnew);
                    else begin = true;
                } else if (!positive(sbest)) {
                    land = true;  // the step starts on the surface, or behind it by rounding: no trial point before it
                } else if (S::FP64 && same(sbest, s) && evbest == ev) {
                    land = true;  // the last trial step ended on the crossing: no re-evaluation
                } else {
                    phase = PH_FINAL;
                }
            }
        } else {
            land = true;  // PH_FINAL: the evaluation landed on the crossing
        }
        if (!S::FP64 && begin) search(p, st, gnew);
        if (land) {
            if (positive(sbest)) st.take_crossing();  // else the state at the step's start, which is still there
            t += sbest;
            h = hs * fac;
            phase = PH_STEP;
            if (evbest == EV_METAL) {
                if (mirrors) {
                    st.mirror();
                    metal = true;
                } else {
                    status = CLOAK_RAY_SINGULAR;
                }
            } else {
                status = metal ? CLOAK_RAY_HIT_METAL_EXITED : CLOAK_RAY_EXITED;
            }
        }
        return status;
    }
    // start the search for the next pending surface; g: its event function at the end point of the step
    __device__ __forceinline__ void search(const Params &p, const S &st, R g) {
        ev = __ffs(pending) - 1;
        lo = 0; hi = hs; glo = st.g_start(p, ev); ghi = g;
        if (!not_positive(glo)) glo = 0;
        side = 0; it = 0;
    }
};

}  // namespace ck
