// trace.cuh -- one camera/test ray through the cloak in FP64 (Sect. 4 pipeline):
// cylinder entry, Sect. 3 double refraction into the chosen mode, integration of
// Eq. 2 / Eq. 8 (RK4 at fixed h, or Dormand-Prince 5(4)), crossing of the exit face,
// the metal mirror at r = R1 for radial ordinary rays, exit refraction, Eq. 12
// weights along the physical direction of light, and the room lookup.
#pragma once

#include <type_traits>

#include "integrator.cuh"
#include "physics.cuh"

namespace ck {

__device__ __forceinline__ void set_vec(double *dst, const double *src) {
    dst[0] = src[0]; dst[1] = src[1]; dst[2] = src[2];
}

// Time-of-flight difference of one camera sample (TOF images, Sect. 4 after Ref. [10]); c0 = 1, so a time
// of flight is a vacuum path length plus the time t spent inside the cloak.  The light the sample
// receives travels from the room point its final vacuum ray reaches, back along that ray, through the
// cloak and to the camera; subtracted is the time from the room point the straight camera ray reaches.
// Rays that miss the cylinder give 0, as do records that carry no light.
__device__ __forceinline__ double tof_difference(const Params &p, const double o[3], const double d[3],
                                                 const cloak_record &rec) {
    int face;
    const double t_ref = room_distance(p, o, d, face);
    double t, pt[3], n[3];
    if (rec.status == CLOAK_RAY_METAL_CAP) {
        for (int i = 0; i < 3; ++i) pt[i] = rec.exit_pos[i];
        t = 0.0;
    } else if (rec.status == CLOAK_RAY_EXITED || rec.status == CLOAK_RAY_HIT_METAL_EXITED) {
        if (cylinder_entry(p, o, d, pt, n) < 0) return 0.0;
        t = rec.tof;
    } else {
        return 0.0;
    }
    const double dx = pt[0] - o[0], dy = pt[1] - o[1], dz = pt[2] - o[2];
    t += sqrt(dx * dx + dy * dy + dz * dz) + room_distance(p, rec.exit_pos, rec.exit_dir, face);
    return t - t_ref;
}

// Entry part: returns true when the ray continues into the medium with state y (x, v).
// Otherwise rec and rgb are final.
template <int MODE>
__device__ __forceinline__ bool enter(const Params &p, const double o[3], const double d[3], cloak_record &rec,
                                      float rgb[3], double y[6], double k0[3], double n_in[3], double mat_in[5]) {
    rec.mode = MODE;
    rec.tile_id = -1;
    rec.steps = 0;
    rec.tof = 0.0;
    rec.weight = 0.0;
    rgb[0] = rgb[1] = rgb[2] = 0.f;
    double pt[3];
    int face = cylinder_entry(p, o, d, pt, n_in);
    // unpolarised room light through the camera's polariser: half of it
    const double vac = p.analyzer ? 0.5 : 1.0;
    if (face < 0) {
        rec.status = CLOAK_RAY_MISSED;
        rec.weight = vac;
        set_vec(rec.exit_pos, o);
        set_vec(rec.exit_dir, d);
        rec.tile_id = room_hit(p, o, d, rgb);
        return false;
    }
    if (face != EV_LAT && p.R1 > 0.0 && hypot(pt[0], pt[1]) <= p.R1) {  // metal end disc: mirror
        double dr[3], dn = dot3(d, n_in);
        for (int i = 0; i < 3; ++i) dr[i] = d[i] - 2.0 * dn * n_in[i];
        rec.status = CLOAK_RAY_METAL_CAP;
        rec.weight = vac;
        set_vec(rec.exit_pos, pt);
        set_vec(rec.exit_dir, dr);
        rec.tile_id = room_hit(p, pt, dr, rgb);
        return false;
    }
    double eo, ee, c[3];
    local_material(p, pt, eo, ee, c);
    double dn = dot3(d, n_in), kt[3], v0[3];
    for (int i = 0; i < 3; ++i) kt[i] = d[i] - dn * n_in[i];
    if (!refract_in(MODE, eo, ee, c, n_in, kt, k0, v0)) {
        rec.status = CLOAK_RAY_NO_TRANSMISSION;
        set_vec(rec.exit_pos, pt);
        set_vec(rec.exit_dir, d);
        return false;
    }
    mat_in[0] = eo; mat_in[1] = ee; mat_in[2] = c[0]; mat_in[3] = c[1]; mat_in[4] = c[2];
    y[0] = pt[0]; y[1] = pt[1]; y[2] = pt[2];
    // the state's second half: ray velocity (Fermat form) or wave vector (Hamiltonian form)
    const double *w = p.formulation ? k0 : v0;
    y[3] = w[0]; y[4] = w[1]; y[5] = w[2];
    return true;
}

// Exit part: refraction into vacuum at the crossed face, Eq. 12 weights, room lookup.
template <int MODE>
__device__ __forceinline__ void leave(const Params &p, int ev, const double y[6], const double d_cam[3],
                                      const double k0[3], const double n_in[3], const double mat_in[5], bool metal,
                                      double t, int steps, cloak_record &rec, float rgb[3]) {
    double x[3] = {y[0], y[1], y[2]}, n[3], eo, ee, c[3], k[3];
    face_normal(ev, x, n);
    local_material(p, x, eo, ee, c);
    if (p.formulation) set_vec(k, y + 3);
    else wave_from_velocity(MODE, eo, ee, c, y + 3, k);
    double kn = dot3(k, n), kt[3];
    for (int i = 0; i < 3; ++i) kt[i] = k[i] - kn * n[i];
    double kt2 = dot3(kt, kt);
    rec.steps = steps;
    rec.tof = t;
    set_vec(rec.exit_pos, x);
    if (kt2 > 1.0) {
        rec.status = CLOAK_RAY_TIR;
        set_vec(rec.exit_dir, d_cam);
        return;
    }
    double qn = sqrt(1.0 - kt2), dout[3], mdout[3], mk0[3];
    for (int i = 0; i < 3; ++i) {
        dout[i] = fma(qn, n[i], kt[i]);
        mdout[i] = -dout[i];
        mk0[i] = -k0[i];
    }
    // light enters from the room at this face and leaves towards the camera at the entry face
    double tin = transmission_in(MODE, eo, ee, c, n, mdout);
    double cin[3] = {mat_in[2], mat_in[3], mat_in[4]};
    double tout = transmission_out(MODE, mat_in[0], mat_in[1], cin, n_in, mk0, analyzer_axis(p));
    rec.weight = tin * tout;
    rec.status = metal ? CLOAK_RAY_HIT_METAL_EXITED : CLOAK_RAY_EXITED;
    set_vec(rec.exit_dir, dout);
    rec.tile_id = room_hit(p, x, dout, rgb);
}

// Whole ray, FP64, by the lanes of a warp together: `valid` lanes have a ray (one each, or one per group of eight
// lanes when WIDE); smem: the block's shared memory of the stepper.  HAM: Hamiltonian form.  rgb receives the room
// colour (0 when there is none).
template <int VAR, int MODE, int INTEG, bool HAM, bool WIDE>
using PlainStepper = typename std::conditional<
    HAM, StepperHam<VAR, MODE, INTEG>,
    typename std::conditional<WIDE, StepperWide<VAR, MODE, INTEG>, Stepper64<VAR, MODE, INTEG>>::type>::type;
template <int VAR, int MODE, int INTEG, bool HAM, bool WIDE>
__device__ __forceinline__ void trace_ray(const Params &p, bool valid, const double o[3], const double d[3], double *smem,
                                          cloak_record &rec, float rgb[3]) {
    typedef PlainStepper<VAR, MODE, INTEG, HAM, WIDE> S;
    S st;
    st.vm = 2 * VAR + MODE;
    st.bind(smem);
    double k0[3], n_in[3], mat_in[5];
    Lane<S, INTEG, false, true> ray;
    ray.reset();
    if (valid && enter<MODE>(p, o, d, rec, rgb, st.y, k0, n_in, mat_in)) ray.start(p);
    st.begin();
    int status = -1;
    for (;;) {
        const bool live = ray.phase != PH_IDLE;
        const unsigned int lm = __ballot_sync(0xffffffffu, live);
        if (!lm) break;
        if (!live) continue;
        status = ray.advance(p, st, lm, VAR == V_RADIAL && MODE == M_ORD);
        if (status >= 0) ray.phase = PH_IDLE;
    }
    if (status < 0) return;  // never entered
    if (status == CLOAK_RAY_EXITED || status == CLOAK_RAY_HIT_METAL_EXITED) {
        leave<MODE>(p, ray.evbest, st.y, d, k0, n_in, mat_in, ray.metal, ray.t, ray.steps, rec, rgb);
        return;
    }
    // STEP_LIMIT or SINGULAR
    rec.status = status;
    rec.steps = ray.steps;
    rec.tof = ray.t;
    rec.exit_pos[0] = st.y[0]; rec.exit_pos[1] = st.y[1]; rec.exit_pos[2] = st.y[2];
    set_vec(rec.exit_dir, d);
}

}  // namespace ck
