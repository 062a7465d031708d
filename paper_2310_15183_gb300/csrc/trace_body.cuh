// trace_body.cuh -- camera set-up and the body of the persistent RK4 ray-queue kernels (sm_103a),
// compiled by trace.cu and, with flush-to-zero FP32 arithmetic, by trace_fp32.cu.
//
// One lane integrates one ray.  In the persistent form a grid of a few blocks per
// SM loops until the global ray queue is empty: whenever lanes of a warp finish,
// the warp counts them with __ballot_sync, one elected lane claims that many new
// ray ids with a single atomicAdd, and the lanes rebuild their initial data from
// the pixel index (camera initialisation is fused -- there are no input arrays).
// Rays that stop early (horizon) therefore do not leave their lanes idle.  Every
// ray runs the same instruction sequence whatever lane, warp or launch shape it
// lands in, so results are bitwise independent of the launch configuration.
//
// Method (Sec. 3.1.2 RK4; appendix listing's propagation kernel for the step rule
// and exit tests):
//   k1 = F(x);  h = |sp / k1.q^t|;  k2 = F(x + h/2 k1);  k3 = F(x + h/2 k2);
//   k4 = F(x + h k3);  x += h w (k1 + 2 k2 + 2 k3 + k4),  w = 1/6 (0.1667 compat);
//   then r > 1.5 r0 -> ESCAPED, else h < sp 3e-5 -> HORIZON, else n_steps -> MAXSTEPS;
//   a non-finite step -> NONFINITE keeping the last finite state.
// Only (r, theta, p_r, p_theta) enter F; t and phi are quadratures and p_t, p_phi
// are constants of motion, so the state is 6 evolving numbers plus 2 constants.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/geotrace.h"
#include "camera.cuh"
#include "compensated.cuh"
#include "internal.cuh"
#include "spacetime.cuh"

namespace gt {
namespace { // each translation unit compiles its own

#define FULL_MASK 0xffffffffu

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ------------------------------------------------------------------ camera set-up
// Spacetime constants (Sec. 2.2.2: a = S/M; Sec. 2.2.3: alpha, k, beta), the pixel
// ranges V = tan(FOV/2)/r0 and H = atan(tan(V) res_x/res_y) of the listing, and the
// lower metric at the camera (inverse of g^{mu nu}'s (t, phi) block and diagonal).
// Three-float form of a double-double.
__device__ __forceinline__ TF tf_from2(double hi, double lo)
{
    TF t;
    t.a = (float)hi;
    const double r = (hi - (double)t.a) + lo;
    t.b = (float)r;
    t.c = (float)(r - (double)t.b);
    return t;
}

// Constants of the double-float step.  Kerr's r_+ = M + sqrt(M^2 - a^2) and Manko-Novikov's
// M + k are carried beyond 53 bits, so that r - r_+ vanishes where the metric's Delta does.
__device__ void setup_pair(const SpacetimeC &st, PairSpacetime &p)
{
    p.kind = st.kind;
    double rt, rt_lo = 0.0; // r_+ - M
    if (st.kind == KIND_KERR) {
        const double m2 = st.M * st.M, m2l = fma(st.M, st.M, -m2);
        const double a2l = fma(st.a, st.a, -st.a2);
        const double d = m2 - st.a2; // M >= a: the error of the difference
        const double dl = ((m2 - d) - st.a2) + (m2l - a2l);
        rt = sqrt(d + dl);
        rt_lo = rt > 0.0 ? (fma(-rt, rt, d) + dl) / (2.0 * rt) : 0.0;
        p.a = DF(st.a);
        p.a2 = DF(st.a2);
        p.r_hard = -1.0f;
    } else {
        rt = st.k;
        p.ik = tf_from(st.ik);
        p.alpha = tf_from(st.alpha);
        p.two_beta = DF(st.two_beta);
        p.three_beta2 = DF(st.three_beta2);
        p.c_g = tf_from(st.c_g);
        p.w_inf = tf_from(st.w_inf);
        p.k2 = tf_from(st.k2);
        p.inv_k2 = tf_from(st.inv_k2);
        p.two_k = tf_from(st.two_k);
        p.r_hard = (float)(4.0 * st.M - st.r_plus);
    }
    const double s = st.M + rt, e = rt - (s - st.M); // M >= rt: Fast2Sum
    p.r_plus = tf_from2(s, e + rt_lo);
    p.r_plus2 = DF(s);
    p.split = DF(2.0 * rt);
}

__device__ void setup_desc(CamDesc &d, int flags, double r_switch)
{
    SpacetimeC st = {};
    st.M = d.M;
    if (d.Q != 0.0) {
        st.kind = KIND_MN;
        const double sm = d.S / d.M;
        const double al = (-d.M + sqrt(d.M * d.M - sm * sm)) / sm;
        const double k = d.M * (1.0 - al * al) / (1.0 + al * al);
        st.alpha = al;
        st.k = k;
        st.ik = 1.0 / k;
        st.beta = d.Q * d.M * d.M * d.M / (k * k * k);
        st.two_beta = 2.0 * st.beta;
        st.three_beta2 = 3.0 * st.beta * st.beta;
        st.c_g = (1.0 - al * al) * (1.0 - al * al) / (k * k);
        st.w_inf = 4.0 * k * al / (1.0 - al * al);
        st.k2 = k * k;
        st.inv_k2 = 1.0 / (k * k);
        st.two_k = 2.0 * k;
        st.r_plus = d.M + k;
    } else {
        st.kind = KIND_KERR;
        st.a = d.S / d.M;
        st.a2 = st.a * st.a;
        st.r_plus = d.M + sqrt(d.M * d.M - st.a2);
    }
    d.st = st;
    setup_pair(st, d.pair);
    d.V = tan(0.5 * d.fov_deg / 180.0 * M_PI) / d.r0;
    d.H = atan(tan(d.V) * (double)d.res_x / (double)d.res_y);
    d.inv_sin_th0 = (flags & GT_FLAG_COMPAT_CAMERA) ? 1.0 : 1.0 / sin(d.th0);
    double g[5];
    upper_metric(st, d.r0, d.th0, g);
    const double det = g[0] * g[2] - g[1] * g[1];
    d.gl_tt = g[2] / det;
    d.gl_tph = -g[1] / det;
    d.gl_phph = g[0] / det;
    d.gl_rr = 1.0 / g[3];
    d.gl_thth = 1.0 / g[4];
    d.r_escape = 1.5 * d.r0;
    if (r_switch > 0.0) {
        d.r_switch = r_switch;
    } else if (r_switch < 0.0) {
        d.r_switch = 0.0;
    } else if (st.kind == KIND_KERR) {
        // Kerr needs no FP64 zone: with the compensated FP32 state, escape/capture and the
        // end directions agree with the FP64 path from a = 0.5M to 0.99M and inclinations
        // 5-85 deg, while a zone covering the horizon approach costs 7-35x in time
        d.r_switch = 0.0;
    } else {
        // Manko-Novikov: the photon region and the horizon approach in FP64 (its metric
        // exponentials come close to the FP32 range there, and FP32 there misclassifies
        // about 0.2 % of the rays of the listing's spacetime)
        d.r_switch = 4.0 * d.M;
    }
    d.valid = (d.gl_tt < 0.0 && isfinite(d.gl_tt) && isfinite(d.gl_phph) && isfinite(d.gl_rr) &&
               isfinite(d.gl_thth) && d.gl_rr > 0.0 && d.gl_thth > 0.0)
                  ? 1
                  : 0;
}

template <int KIND>
__device__ __forceinline__ void rates_any(const SpacetimeC &st, double r, double s, double cs,
                                          double pr, double pth, double pt, double pph,
                                          Rates<double> &o)
{
    if (KIND == KIND_KERR || (KIND == KIND_ANY && st.kind == KIND_KERR))
        kerr_rates_sc<double>(st, r, s, cs, pr, pth, pt, pph, o);
    else
        mn_rates_sc<double>(st, r, s, cs, pr, pth, pt, pph, o);
}

// The listing's numerics (KIND_FD): the inverse metric at (r, theta) and the forward
// differences d_r g ~ (g(r + delta, theta) - g(r, theta))/delta, d_theta likewise, with
// delta = derPrecision = 1e-8 -- three metric evaluations -- contracted into
// dp = -1/2 d g^{nu sigma} p_nu p_sigma component by component.
constexpr double FD_DELTA = 1e-8;

__device__ __forceinline__ double fd_quad(const double d[5], double pr, double pth, double pt,
                                          double pph)
{
    return d[0] * pt * pt + 2.0 * d[1] * pt * pph + d[2] * pph * pph + d[3] * pr * pr +
           d[4] * pth * pth;
}

__device__ __forceinline__ void rates_fd(const SpacetimeC &st, double r, double th, double pr,
                                         double pth, double pt, double pph, Rates<double> &o)
{
    double g0[5], gr[5], gt[5], dr[5], dt[5];
    upper_metric(st, r, th, g0);
    upper_metric(st, r + FD_DELTA, th, gr);
    upper_metric(st, r, th + FD_DELTA, gt);
#pragma unroll
    for (int i = 0; i < 5; i++) {
        dr[i] = (gr[i] - g0[i]) / FD_DELTA;
        dt[i] = (gt[i] - g0[i]) / FD_DELTA;
    }
    o.dt = g0[0] * pt + g0[1] * pph;
    o.dph = g0[1] * pt + g0[2] * pph;
    o.dr = g0[3] * pr;
    o.dth = g0[4] * pth;
    o.dpr = -0.5 * fd_quad(dr, pr, pth, pt, pph);
    o.dpth = -0.5 * fd_quad(dt, pr, pth, pt, pph);
}

// One FP64 RK4 step; returns h and writes the candidate state to y.  sin and cos of
// theta are evaluated once per step and rotated to the later stages by their small
// angle offsets (Taylor series, FP64 accurate); the forward-difference kind evaluates
// its metric at each stage's theta as the listing does.
template <int KIND>
__device__ __forceinline__ double rk4_step64(const SpacetimeC &st, const Ray64 &x, double sp,
                                             double w6, Ray64 &y)
{
    Rates<double> k1, k2, k3, k4;
    double h, hh;
    if constexpr (KIND == KIND_FD) {
        rates_fd(st, x.r, x.th, x.pr, x.pth, x.pt, x.pph, k1);
        h = fabs(sp / k1.dt);
        hh = 0.5 * h;
        rates_fd(st, x.r + hh * k1.dr, x.th + hh * k1.dth, x.pr + hh * k1.dpr,
                 x.pth + hh * k1.dpth, x.pt, x.pph, k2);
        rates_fd(st, x.r + hh * k2.dr, x.th + hh * k2.dth, x.pr + hh * k2.dpr,
                 x.pth + hh * k2.dpth, x.pt, x.pph, k3);
        rates_fd(st, x.r + h * k3.dr, x.th + h * k3.dth, x.pr + h * k3.dpr,
                 x.pth + h * k3.dpth, x.pt, x.pph, k4);
    } else {
        double s1, c1, s, c;
        sincos(x.th, &s1, &c1);
        rates_any<KIND>(st, x.r, s1, c1, x.pr, x.pth, x.pt, x.pph, k1);
        h = fabs(sp / k1.dt);
        hh = 0.5 * h;
        rotate_sc(s1, c1, x.th, hh * k1.dth, &s, &c);
        rates_any<KIND>(st, x.r + hh * k1.dr, s, c, x.pr + hh * k1.dpr, x.pth + hh * k1.dpth,
                        x.pt, x.pph, k2);
        rotate_sc(s1, c1, x.th, hh * k2.dth, &s, &c);
        rates_any<KIND>(st, x.r + hh * k2.dr, s, c, x.pr + hh * k2.dpr, x.pth + hh * k2.dpth,
                        x.pt, x.pph, k3);
        rotate_sc(s1, c1, x.th, h * k3.dth, &s, &c);
        rates_any<KIND>(st, x.r + h * k3.dr, s, c, x.pr + h * k3.dpr, x.pth + h * k3.dpth, x.pt,
                        x.pph, k4);
    }
    const double hw = h * w6;
    y.t = x.t + hw * (k1.dt + 2.0 * k2.dt + 2.0 * k3.dt + k4.dt);
    y.r = x.r + hw * (k1.dr + 2.0 * k2.dr + 2.0 * k3.dr + k4.dr);
    y.th = x.th + hw * (k1.dth + 2.0 * k2.dth + 2.0 * k3.dth + k4.dth);
    y.ph = x.ph + hw * (k1.dph + 2.0 * k2.dph + 2.0 * k3.dph + k4.dph);
    y.pr = x.pr + hw * (k1.dpr + 2.0 * k2.dpr + 2.0 * k3.dpr + k4.dpr);
    y.pth = x.pth + hw * (k1.dpth + 2.0 * k2.dpth + 2.0 * k3.dpth + k4.dpth);
    y.pt = x.pt;
    y.pph = x.pph;
    return h;
}

// One explicit Euler step (Sec. 3.1.1): x += h F(x) with the same step rule.
template <int KIND>
__device__ __forceinline__ double euler_step64(const SpacetimeC &st, const Ray64 &x, double sp,
                                               Ray64 &y)
{
    Rates<double> k1;
    if constexpr (KIND == KIND_FD) {
        rates_fd(st, x.r, x.th, x.pr, x.pth, x.pt, x.pph, k1);
    } else {
        double s1, c1;
        sincos(x.th, &s1, &c1);
        rates_any<KIND>(st, x.r, s1, c1, x.pr, x.pth, x.pt, x.pph, k1);
    }
    const double h = fabs(sp / k1.dt);
    y.t = x.t + h * k1.dt;
    y.r = x.r + h * k1.dr;
    y.th = x.th + h * k1.dth;
    y.ph = x.ph + h * k1.dph;
    y.pr = x.pr + h * k1.dpr;
    y.pth = x.pth + h * k1.dpth;
    y.pt = x.pt;
    y.pph = x.pph;
    return h;
}

template <int KIND>
__device__ __forceinline__ double step64(const TraceArgs &A, const SpacetimeC &st, const Ray64 &x,
                                         Ray64 &y)
{
    if (A.euler) return euler_step64<KIND>(st, x, A.sp, y);
    return rk4_step64<KIND>(st, x, A.sp, A.w6, y);
}

// ------------------------------------------------------------------ the double-float step
__device__ __forceinline__ void tf_state(const Ray64 &x, RayTF &s)
{
    s.t = tf_from(x.t);
    s.r = tf_from(x.r);
    s.th = tf_from(x.th);
    s.ph = tf_from(x.ph);
    s.pr = tf_from(x.pr);
    s.pth = tf_from(x.pth);
    s.pt = tf_from(x.pt);
    s.pph = tf_from(x.pph);
}

// The evolving coordinates back in FP64 (the constants of motion of x are kept).
__device__ __forceinline__ void tf_unstate(const RayTF &s, Ray64 &x)
{
    x.t = tf_to(s.t);
    x.r = tf_to(s.r);
    x.th = tf_to(s.th);
    x.ph = tf_to(s.ph);
    x.pr = tf_to(s.pr);
    x.pth = tf_to(s.pth);
}

// The tables of pair.cuh, copied by each block into shared memory.
__device__ const PairTables g_pair_tables = make_pair_tables();

// The evolving coordinates of an FP64 state in the words of a three-float one, and back: a ray that
// stays in FP64 for a while needs no registers of its own for it.
__device__ __forceinline__ void hold64(double v, TF &t)
{
    t.a = __int_as_float(__double2loint(v));
    t.b = __int_as_float(__double2hiint(v));
}
__device__ __forceinline__ double held64(TF t)
{
    return __hiloint2double(__float_as_int(t.b), __float_as_int(t.a));
}
__device__ __forceinline__ void hold64(const Ray64 &x, RayTF &s)
{
    hold64(x.t, s.t);
    hold64(x.r, s.r);
    hold64(x.th, s.th);
    hold64(x.ph, s.ph);
    hold64(x.pr, s.pr);
    hold64(x.pth, s.pth);
}
__device__ __forceinline__ void held64(const RayTF &s, Ray64 &x)
{
    x.t = held64(s.t);
    x.r = held64(s.r);
    x.th = held64(s.th);
    x.ph = held64(s.ph);
    x.pr = held64(s.pr);
    x.pth = held64(s.pth);
}

// The same step in FP64, out of line: the double-float kernels keep their registers.
template <int KIND>
__device__ __noinline__ double rk4_step64_call(const SpacetimeC &st, const Ray64 &x, double sp,
                                               double w6, Ray64 &y)
{
    return rk4_step64<KIND>(st, x, sp, w6, y);
}

// A double-float step of an FP64 state, for the FP32 kernel with its zone inline (MODE 1).
template <int KIND>
__device__ __forceinline__ bool pair_step64(const PairSpacetime &c, const PairTables *tab, Ray64 &x,
                                            TF sp, TF w6, double &h)
{
    RayTF T;
    DF hd;
    tf_state(x, T);
    if (!pair_step<KIND>(c, tab, T, sp, w6, 0.0f, hd)) return false;
    h = df_to(hd);
    tf_unstate(T, x);
    return true;
}

template <int KIND>
__device__ __noinline__ bool pair_step64_call(const PairSpacetime &c, const PairTables *tab, Ray64 &x,
                                              TF sp, TF w6, double &h)
{
    return pair_step64<KIND>(c, tab, x, sp, w6, h);
}

// What MODE 1 compiles of it, by its effect on the FP32 steps beside it: Kerr nothing (it has no
// zone by default, MODE 1's only form; a ray at r < 0 takes FP64), cameras of both kinds a call,
// Manko-Novikov the step itself.  gt_trace_batch_noalloc, FP32 steps alone: 40,000 Kerr rays x
// 4,000 steps 5.41 ms (the step inline 9.09, a call 9.43), 16,000 of both kinds x 2,000 4.93 to
// 5.26 (inline 5.23 to 5.36), 40,000 Manko-Novikov x 2,000 8.77 to 9.19 (a call 9.88); in the
// zone, 12,000 Manko-Novikov rays x 1,000 steps 25 ms (a call 21).
template <int KIND>
__device__ __forceinline__ bool inline_zone_step(const PairSpacetime &c, const PairTables *tab, Ray64 &x,
                                                 TF sp, TF w6, double &h)
{
    if constexpr (KIND == KIND_KERR) return false;
    else if constexpr (KIND == KIND_ANY) return pair_step64_call<KIND>(c, tab, x, sp, w6, h);
    else return pair_step64<KIND>(c, tab, x, sp, w6, h);
}

// ------------------------------------------------------------------ ring and redshift
__device__ __forceinline__ bool in_disk(const DiskArgs &dk, double r, double th)
{
    return r >= dk.r_in && r <= dk.r_out && fabs(r * cos(th)) <= dk.half_thickness;
}

// Redshift factor of the ray x at the ring (Sec. 3.3.3): the emitter moves on the
// circular orbit through (r, theta) -- p_r = p_theta = 0, dp_r/dtau = 0 and p_t = -1,
// i.e. A p_phi^2 - 2 B p_phi + C = 0 with (A, B, C) = d_r (g^{phi phi}, g^{t phi}, g^{tt}),
// the root with positive angular velocity, rescaled to g^{mu nu} p_mu p_nu = -1 -- and
// z = (p . u_S) / (p . u_O), u_O the static observer at the camera, p . u_O =
// p_t / sqrt(-g_tt(camera)).  Exact r derivatives by dual numbers (forward differences
// with KIND_FD).  NaN where no timelike circular orbit exists.
template <int KIND>
__device__ double redshift64(const SpacetimeC &st, double gl_tt_cam, const Ray64 &x)
{
    double g[3], A, B, C;
    if (KIND == KIND_FD) {
        double g0[5], gr[5];
        upper_metric(st, x.r, x.th, g0);
        upper_metric(st, x.r + FD_DELTA, x.th, gr);
        A = (gr[2] - g0[2]) / FD_DELTA;
        B = (gr[1] - g0[1]) / FD_DELTA;
        C = (gr[0] - g0[0]) / FD_DELTA;
        g[0] = g0[0];
        g[1] = g0[1];
        g[2] = g0[2];
    } else {
        D3<double> gd[3];
        if (st.kind == KIND_KERR)
            kerr_upper_tphi<double, D3<double>>(st, x.r, x.th, gd);
        else
            mn_upper_tphi<double, D3<double>>(st, x.r, x.th, gd);
        C = gd[0].r;
        B = gd[1].r;
        A = gd[2].r;
        g[0] = gd[0].v;
        g[1] = gd[1].v;
        g[2] = gd[2].v;
    }
    const double disc = B * B - A * C;
    if (!(disc >= 0.0) || A == 0.0) return nan("");
    const double sq = sqrt(disc);
    const double roots[2] = {(B + sq) / A, (B - sq) / A};
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const double pph = roots[k];
        const double ut = -g[0] + g[1] * pph;
        const double uph = -g[1] + g[2] * pph;
        const double norm = g[0] - 2.0 * g[1] * pph + g[2] * pph * pph;
        if (ut > 0.0 && uph / ut > 0.0 && norm < 0.0) {
            const double lam = 1.0 / sqrt(-norm);
            const double num = (x.pt * ut + x.pph * uph) * lam;
            return num / (x.pt / sqrt(-gl_tt_cam));
        }
    }
    return nan("");
}

__device__ __forceinline__ bool finite6(const Ray64 &y)
{
    return isfinite(y.t) && isfinite(y.r) && isfinite(y.th) && isfinite(y.ph) && isfinite(y.pr) &&
           isfinite(y.pth);
}

__device__ __forceinline__ double round_f32(double v) { return (double)(float)v; }

// End position of a ray that did not run (watchdog drain): position outputs only.
__device__ __forceinline__ void store_ray(const TraceArgs &A, int64_t id, double t, double r,
                                          double th, double ph, int status, uint32_t n)
{
    if (A.f32_io) {
        t = round_f32(t);
        r = round_f32(r);
        th = round_f32(th);
        ph = round_f32(ph);
    }
    if (A.t) A.t[id] = t;
    if (A.r) A.r[id] = r;
    if (A.th) A.th[id] = th;
    if (A.ph) A.ph[id] = ph;
    if (A.status) A.status[id] = (uint8_t)status;
    if (A.nsteps) A.nsteps[id] = n;
    if (A.z) A.z[id] = nan("");
}

// End state of a ray: position outputs (float32-rounded with f32_io), the redshift
// factor, and with state arrays the whole state written back.
__device__ __forceinline__ void store_full(const TraceArgs &A, int64_t id, const Ray64 &x,
                                           int status, uint32_t n, double z)
{
    store_ray(A, id, x.t, x.r, x.th, x.ph, status, n);
    if (A.z) A.z[id] = z;
    if (A.states.t) {
        A.states.t[id] = x.t;
        A.states.r[id] = x.r;
        A.states.th[id] = x.th;
        A.states.ph[id] = x.ph;
        A.states.pt[id] = x.pt;
        A.states.pr[id] = x.pr;
        A.states.pth[id] = x.pth;
        A.states.pph[id] = x.pph;
    }
}

// Camera of flat ray id (binary search over the prefix offsets).
__device__ __forceinline__ int find_camera(const CamDesc *__restrict__ cams, int n_cams, int64_t id)
{
    int lo = 0, hi = n_cams - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cams[mid].offset <= id)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Status after a step (listing's order: escape first, then step collapse).
__device__ __forceinline__ int exit_status(double r, double h, double r_esc, double sp, uint32_t n,
                                           int64_t n_steps)
{
    if (r > r_esc) return GT_RAY_ESCAPED;
    if (h < sp * 0.00003) return GT_RAY_HORIZON;
    if ((int64_t)n >= n_steps) return GT_RAY_MAXSTEPS;
    return -1;
}

// ------------------------------------------------------------------ FP32-mixed pieces
struct RayMixed {
    F2 t, r, th, ph, pr, pth;
    double pt, pph; // constants of motion kept in FP64
    float ptf, pphf;
};

__device__ __forceinline__ void mixed_from64(const Ray64 &x, RayMixed &m)
{
    m.t = f2_from(x.t);
    m.r = f2_from(x.r);
    m.th = f2_from(x.th);
    m.ph = f2_from(x.ph);
    m.pr = f2_from(x.pr);
    m.pth = f2_from(x.pth);
    m.pt = x.pt;
    m.pph = x.pph;
    m.ptf = (float)x.pt;
    m.pphf = (float)x.pph;
}

__device__ __forceinline__ void mixed_to64(const RayMixed &m, Ray64 &x)
{
    x.t = f2_to(m.t);
    x.r = f2_to(m.r);
    x.th = f2_to(m.th);
    x.ph = f2_to(m.ph);
    x.pr = f2_to(m.pr);
    x.pth = f2_to(m.pth);
    x.pt = m.pt;
    x.pph = m.pph;
}

template <int KIND, bool PRECISE, bool OWN = false>
__device__ __forceinline__ void rates_f32(const SpacetimeF &st, float r, float s, float cs,
                                          float pr, float pth, float pt, float pph,
                                          Rates<float> &o)
{
    if (KIND == KIND_KERR || (KIND == 2 && st.kind == KIND_KERR))
        kerr_rates_sc<float, OWN>(st, r, s, cs, pr, pth, pt, pph, o);
    else
        mn_rates_sc<float, PRECISE>(st, r, s, cs, pr, pth, pt, pph, o);
}

// One FP32 RK4 step on the compensated state; returns h (as float).
template <int KIND, bool PRECISE = false>
__device__ __forceinline__ float rk4_step32(const SpacetimeF &st, RayMixed &m, float sp, float w6)
{
    Rates<float> k1, k2, k3, k4;
    const float r = m.r.hi, th = m.th.hi, pr = m.pr.hi, pth = m.pth.hi;
    // sin/cos of theta once per step; the later stages rotate them by their small offsets
    float s1, c1, s, c;
    sincosf(th, &s1, &c1);
    rates_f32<KIND, PRECISE>(st, r, s1, c1, pr, pth, m.ptf, m.pphf, k1);
    const float h = fabsf(sp / k1.dt);
    const float hh = 0.5f * h;
    rotate_sc(s1, c1, th, hh * k1.dth, &s, &c);
    rates_f32<KIND, PRECISE>(st, fmaf(hh, k1.dr, r), s, c, fmaf(hh, k1.dpr, pr),
                             fmaf(hh, k1.dpth, pth), m.ptf, m.pphf, k2);
    rotate_sc(s1, c1, th, hh * k2.dth, &s, &c);
    rates_f32<KIND, PRECISE>(st, fmaf(hh, k2.dr, r), s, c, fmaf(hh, k2.dpr, pr),
                             fmaf(hh, k2.dpth, pth), m.ptf, m.pphf, k3);
    rotate_sc(s1, c1, th, h * k3.dth, &s, &c);
    rates_f32<KIND, PRECISE>(st, fmaf(h, k3.dr, r), s, c, fmaf(h, k3.dpr, pr),
                             fmaf(h, k3.dpth, pth), m.ptf, m.pphf, k4);
    const float hw = h * w6;
    f2_add(m.t, hw * (k1.dt + 2.0f * k2.dt + 2.0f * k3.dt + k4.dt));
    f2_add(m.r, hw * (k1.dr + 2.0f * k2.dr + 2.0f * k3.dr + k4.dr));
    f2_add(m.th, hw * (k1.dth + 2.0f * k2.dth + 2.0f * k3.dth + k4.dth));
    f2_add(m.ph, hw * (k1.dph + 2.0f * k2.dph + 2.0f * k3.dph + k4.dph));
    f2_add(m.pr, hw * (k1.dpr + 2.0f * k2.dpr + 2.0f * k3.dpr + k4.dpr));
    f2_add(m.pth, hw * (k1.dpth + 2.0f * k2.dpth + 2.0f * k3.dpth + k4.dpth));
    return h;
}

// The same step out of line, for the rays whose stage angles the fast step below does not take.
template <int KIND, bool PRECISE>
__device__ __noinline__ float rk4_step32_call(const SpacetimeF &st, RayMixed &m, float sp, float w6)
{
    return rk4_step32<KIND, PRECISE>(st, m, sp, w6);
}

// rk4_step32 without a branch between its stages: the rotation of sin/cos by the series alone,
// `turn` receiving the largest stage angle -- beyond 1/4 (not met in practice) the result is
// not rk4_step32's and the caller repeats the step out of line.  The fused multiply-adds of the
// sums are written out as the compiler forms them across rk4_step32's basic blocks, so that
// both give the same bits.
__device__ __forceinline__ void rotate_series(float s, float c, float d, float *s2, float *c2)
{
    const float d2 = d * d;
    const float sd = fmaf(d * d2, fmaf(d2, fmaf(d2, -1.0f / 5040.0f, 1.0f / 120.0f), -1.0f / 6.0f), d);
    const float cd = fmaf(d2, fmaf(d2, fmaf(d2, -1.0f / 720.0f, 1.0f / 24.0f), -0.5f), 1.0f);
    *s2 = fmaf(s, cd, c * sd);
    *c2 = fmaf(c, cd, -(s * sd));
}

// OWN: the bits of a field behind a branch on the ray's own kind of spacetime -- the rates rounded
// before they are summed, except theta's.
template <bool OWN>
__device__ __forceinline__ float stage_sum(float k1, float k2, float k3, float k4)
{
    const float s = __fmaf_rn(2.0f, k3, __fmaf_rn(2.0f, k2, k1));
    return OWN ? __fadd_rn(s, k4) : s + k4;
}

template <int KIND, bool PRECISE = false, bool OWN = false>
__device__ __forceinline__ float rk4_step32_fast(const SpacetimeF &st, RayMixed &m, float sp,
                                                 float w6, float &turn)
{
    Rates<float> k1, k2, k3, k4;
    const float r = m.r.hi, th = m.th.hi, pr = m.pr.hi, pth = m.pth.hi;
    float s1, c1, s, c;
    sincosf(th, &s1, &c1);
    rates_f32<KIND, PRECISE, OWN>(st, r, s1, c1, pr, pth, m.ptf, m.pphf, k1);
    const float h = fabsf(sp / k1.dt);
    const float hh = 0.5f * h;
    const float d1 = __fmul_rn(hh, k1.dth);
    rotate_series(s1, c1, d1, &s, &c);
    rates_f32<KIND, PRECISE, OWN>(st, fmaf(hh, k1.dr, r), s, c, fmaf(hh, k1.dpr, pr),
                             fmaf(hh, k1.dpth, pth), m.ptf, m.pphf, k2);
    const float d2 = __fmul_rn(hh, k2.dth);
    rotate_series(s1, c1, d2, &s, &c);
    rates_f32<KIND, PRECISE, OWN>(st, fmaf(hh, k2.dr, r), s, c, fmaf(hh, k2.dpr, pr),
                             fmaf(hh, k2.dpth, pth), m.ptf, m.pphf, k3);
    const float d3 = __fmul_rn(h, k3.dth);
    rotate_series(s1, c1, d3, &s, &c);
    rates_f32<KIND, PRECISE, OWN>(st, fmaf(h, k3.dr, r), s, c, fmaf(h, k3.dpr, pr),
                             fmaf(h, k3.dpth, pth), m.ptf, m.pphf, k4);
    turn = fmaxf(fmaxf(fabsf(d1), fabsf(d2)), fabsf(d3));
    const float hw = h * w6;
    f2_add(m.t, hw * stage_sum<OWN>(k1.dt, k2.dt, k3.dt, k4.dt));
    f2_add(m.r, hw * stage_sum<OWN>(k1.dr, k2.dr, k3.dr, k4.dr));
    f2_add(m.th, hw * stage_sum<false>(k1.dth, k2.dth, k3.dth, k4.dth));
    f2_add(m.ph, hw * stage_sum<OWN>(k1.dph, k2.dph, k3.dph, k4.dph));
    f2_add(m.pr, hw * stage_sum<OWN>(k1.dpr, k2.dpr, k3.dpr, k4.dpr));
    f2_add(m.pth, hw * stage_sum<OWN>(k1.dpth, k2.dpth, k3.dpth, k4.dpth));
    return h;
}

// H = 0 re-projection in FP64 (mixed mode): solve g^rr p_r^2 = -(rest) for |p_r|,
// keeping the sign of p_r.  Skipped near radial turning points, where the radial
// term is small against the rest and the square root is ill-conditioned.
__device__ __forceinline__ void reproject_pr(const SpacetimeC &st, Ray64 &x)
{
    double g[5];
    upper_metric(st, x.r, x.th, g);
    const double rest = g[0] * x.pt * x.pt + 2.0 * g[1] * x.pt * x.pph + g[2] * x.pph * x.pph +
                        g[4] * x.pth * x.pth;
    const double rad = g[3] * x.pr * x.pr;
    const double scale = fabs(g[0] * x.pt * x.pt) + fabs(g[2] * x.pph * x.pph) + rad +
                         g[4] * x.pth * x.pth;
    if (!(rad > 0.05 * scale)) return;
    const double pr2 = -rest / g[3];
    if (!(pr2 > 0.0) || !isfinite(pr2)) return;
    x.pr = copysign(sqrt(pr2), x.pr);
}

// ------------------------------------------------------------------ the kernel
// MODE 0: FP64 plain.
// MODE 1: FP32-mixed with the FP64 zone inline (used where no park lists exist).
// MODE 2: FP32-mixed, FP32 steps only; a ray entering the FP64 zone (r < r_switch) is
//         parked on the output list; input list items continue in FP32.
// MODE 3: FP64 zone steps for parked rays; a ray leaving the zone (r > 1.25 r_switch)
//         is parked on the output list for the next FP32 launch.
// MODE 4: MODE 3 with the double-float step.
// MODE 5: MODE 0 with the double-float step.
// KIND: 0 Kerr, 1 Manko-Novikov, 2 per-camera, 3 per-camera with forward-difference
// derivatives (MODE 0 only).
// Work of a launch: fresh rays [0, n_fresh) then input-list items [0, *in_count).

__device__ __forceinline__ void park(const TraceArgs &A, int64_t id, uint32_t n, int cam,
                                     const Ray64 &x, bool *ok)
{
    const unsigned long long slot = atomicAdd(A.out_count, 1ull);
    if (slot >= A.out_cap) { // cannot happen with capacity = rays of the launch
        *ok = false;
        return;
    }
    ParkItem &it = A.out_items[slot];
    it.id = id;
    it.n = n;
    it.cam = cam;
    it.t = x.t;
    it.r = x.r;
    it.th = x.th;
    it.ph = x.ph;
    it.pr = x.pr;
    it.pth = x.pth;
    it.pt = x.pt;
    it.pph = x.pph;
    *ok = true;
}

// SINGLE: one camera, its constants in the kernel's parameters (A.pair, A.stf).
template <int MODE, int KIND, bool PRECISE, bool SINGLE>
__device__ __forceinline__ void trace_body(const TraceArgs &A, int one_shot)
{
    constexpr bool ZONE = MODE == 3 || MODE == 4;  // zone rays, parked when they leave
    constexpr bool PAIR = MODE == 4 || MODE == 5;  // three-float state, double-float step
    constexpr bool TABLES = PAIR || (MODE == 1 && KIND != KIND_KERR);
    // per-ray spacetimes come with KIND_ANY only, and never to the double-float MODE 5
    const RayParams *const rays = KIND == KIND_ANY && MODE != 5 ? A.rays : nullptr;
    __shared__ PairTables tab_s[1];
    const PairTables *tab = tab_s;
    if (TABLES) {
        const float *src = reinterpret_cast<const float *>(&g_pair_tables);
        float *dst = reinterpret_cast<float *>(tab_s);
        for (int i = threadIdx.x; i < (int)(sizeof(PairTables) / sizeof(float)); i += blockDim.x)
            dst[i] = src[i];
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    unsigned long long *next = A.scratch + SCR_NEXT_RAY;
    volatile unsigned long long *tflag = A.scratch + SCR_TIMEOUT;
    const uint64_t t_start = A.timeout_ns ? globaltimer_ns() : 0;
    const CamDesc *__restrict__ cams = A.cams;
    const int64_t n_in =
        A.in_count ? (int64_t)(*A.in_count < A.in_cap ? *A.in_count : A.in_cap) : 0;
    const int64_t n_work = A.n_fresh + n_in;

    int64_t id = -1;
    int cam = 0;
    bool active = false;
    bool drained = false;
    uint32_t n = 0;
    uint32_t n_entry = 0;           // step count when the ray entered this launch (zone steps)
    uint32_t n_f64 = 0;             // zone field evaluations of the ray in FP64 (this launch)
    PairSpacetime pr_ray;           // double-float constants of a per-ray spacetime
    RayTF T;                        // state of the double-float kernels
    // A GT_MODE_FP64 ray that stays where pairs are refused -- below 4M, at the axis -- keeps its
    // FP64 state: no conversion of twelve values a step (~72 instructions of the FP64 pipe beside
    // the step's 1,343) and no refused pair step.  48,000 Manko-Novikov rays x 1,000 steps at 3.8M
    // 138.8 -> 130.3 ms (the FP64 kernel: 143.6), 3,000 across 4M 266 -> 251, on the axis 151 ->
    // 148.  Kerr refuses only at the axis (43.7 ms; the FP64 kernel 54.2), and the test in front of
    // every step costs a lone Schwarzschild warp 4 %: left out there.
    constexpr bool KEEP64 = MODE == 5 && KIND != KIND_KERR;
    bool in64 = false; // T holds the FP64 state (hold64)
    uint32_t rp_next = 0xFFFFFFFFu; // next step count that is a multiple of reproject_every
    Ray64 x;
    RayMixed m;
    SpacetimeC st = cams[0].st;
    SpacetimeF stf = to_float(st);
    double r_esc = cams[0].r_escape;
    double r_sw = cams[0].r_switch;
    const float spf = A.sp_f, w6f = A.w6_f;
    const float h_thr_f = A.h_thr_f;
    const uint32_t n_last = (uint32_t)A.n_steps; // n_steps <= 2^32 - 1
    F2 r_esc_f = f2_from(r_esc);
    float r_sw_f = (float)r_sw;
    TF r_esc_t = tf_from(r_esc), r_out_t = tf_from(1.25 * r_sw);

    auto load_camera = [&](int c) {
        cam = c;
        // the FP32-only kernel keeps just the float constants live; the FP64 ones are
        // reloaded for the occasional re-projection
        if (MODE != 2 && !PAIR) st = cams[c].st;
        r_esc = cams[c].r_escape;
        r_sw = cams[c].r_switch;
        if (MODE == 1 || MODE == 2) stf = to_float(cams[c].st);
        if (MODE == 2) {
            r_esc_f = f2_from(r_esc);
            r_sw_f = (float)r_sw;
        }
        if (PAIR) {
            r_esc_t = tf_from(r_esc);
            r_out_t = tf_from(1.25 * r_sw);
        }
    };
    auto load_rayparams = [&](int64_t rid, bool init) {
        CamDesc d;
        d.M = rays->M;
        d.S = rays->spin[rid] * rays->M * rays->M; // spin = a/M
        d.Q = rays->q[rid];
        d.r0 = rays->r0;
        d.th0 = rays->theta0[rid];
        d.fov_deg = 90.0;
        d.res_x = d.res_y = 1;
        d.offset = 0;
        setup_desc(d, A.flags, rays->r_switch);
        if (MODE != 2) st = d.st;
        if (MODE == 1 || MODE == 4) pr_ray = d.pair;
        r_esc = d.r_escape;
        r_sw = d.r_switch;
        if (MODE == 1 || MODE == 2) stf = to_float(d.st);
        if (MODE == 2) {
            r_esc_f = f2_from(r_esc);
            r_sw_f = (float)r_sw;
        }
        if (PAIR) {
            r_esc_t = tf_from(r_esc);
            r_out_t = tf_from(1.25 * r_sw);
        }
        if (init) camera_init_dir(d, rays->alpha[rid], rays->beta[rid], x);
        return d.valid != 0;
    };

    auto picked = [&](int c) {
        return SINGLE || !A.pick_mask || (cams[c].route & A.pick_mask) == A.pick;
    };

    // Start work item `w`; returns false when the ray is already finished and stored, or another
    // launch's.
    auto start = [&](int64_t w) -> bool {
        if (w < A.n_fresh) { // a fresh ray: initial data from the camera
            const int64_t pix = A.fresh_ids ? A.fresh_ids[w] : w;
            id = (A.fresh_ids && A.compact_out) ? w : pix;
            if (rays) {
                const bool valid = load_rayparams(pix, true);
                n = 0;
                if (!valid || A.n_steps <= 0) {
                    store_ray(A, id, x.t, x.r, x.th, x.ph, valid ? GT_RAY_MAXSTEPS : GT_RAY_NONFINITE, 0);
                    return false;
                }
            } else if (A.states.t) { // an arbitrary initial state (gt_trace_states)
                x.t = A.states.t[pix];
                x.r = A.states.r[pix];
                x.th = A.states.th[pix];
                x.ph = A.states.ph[pix];
                x.pt = A.states.pt[pix];
                x.pr = A.states.pr[pix];
                x.pth = A.states.pth[pix];
                x.pph = A.states.pph[pix];
                n = 0;
                if (A.n_steps <= 0) {
                    store_full(A, id, x, GT_RAY_MAXSTEPS, 0, nan(""));
                    return false;
                }
            } else {
                if (KIND >= KIND_ANY || A.n_cams > 1) load_camera(find_camera(cams, A.n_cams, pix));
                if (!picked(cam)) return false;
                camera_init(cams[cam], A.first + pix - cams[cam].offset, x);
                if (A.f32_io) { // the listing's kernels take the initial state as float32
                    x.t = round_f32(x.t);
                    x.r = round_f32(x.r);
                    x.th = round_f32(x.th);
                    x.ph = round_f32(x.ph);
                    x.pt = round_f32(x.pt);
                    x.pr = round_f32(x.pr);
                    x.pth = round_f32(x.pth);
                    x.pph = round_f32(x.pph);
                }
                n = 0;
                if (A.n_steps <= 0) {
                    store_full(A, id, x, GT_RAY_MAXSTEPS, 0, nan(""));
                    return false;
                }
            }
        } else { // a parked ray from the input list
            const ParkItem &it = A.in_items[w - A.n_fresh];
            id = it.id;
            n = it.n;
            if (rays)
                load_rayparams(id, false);
            else if (KIND >= KIND_ANY || A.n_cams > 1)
                load_camera(it.cam);
            if (!picked(cam)) return false;
            x.t = it.t;
            x.r = it.r;
            x.th = it.th;
            x.ph = it.ph;
            x.pr = it.pr;
            x.pth = it.pth;
            x.pt = it.pt;
            x.pph = it.pph;
        }
        n_entry = n;
        n_f64 = 0;
        if (PAIR) tf_state(x, T);
        in64 = false;
        if (MODE == 1 || MODE == 2) {
            mixed_from64(x, m);
            if (A.reproject_every > 0) {
                const uint64_t k = (uint64_t)A.reproject_every;
                const uint64_t nx = ((uint64_t)n / k + 1u) * k;
                rp_next = nx < 0xFFFFFFFFull ? (uint32_t)nx : 0xFFFFFFFFu;
            }
        }
        return true;
    };

    if (one_shot) {
        drained = true;
        const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        if (w < n_work) active = start(w);
    }

    for (uint32_t it = 0;; ++it) {
        // ---- refill finished lanes from the global queue
        if (!drained) {
            const unsigned need = __ballot_sync(FULL_MASK, !active);
            if (need) {
                const int cnt = __popc(need);
                const int leader = __ffs(need) - 1;
                unsigned long long base = 0;
                if (lane == leader) base = atomicAdd(next, (unsigned long long)cnt);
                base = __shfl_sync(FULL_MASK, base, leader);
                if (base + (unsigned long long)cnt >= (unsigned long long)n_work) drained = true;
                if (!active) {
                    const int64_t w = (int64_t)base + __popc(need & lt_mask);
                    if (w < n_work) active = start(w);
                }
            }
        }
        const unsigned live = __ballot_sync(FULL_MASK, active);
        if (!live) {
            if (drained) break;
            continue;
        }
        // ---- watchdog: stop every lane with status TIMEOUT
        if (A.timeout_ns && (MODE == 2 || (it & 127u) == 0u)) {
            int stop = 0;
            if (lane == 0) {
                if (*tflag) {
                    stop = 1;
                } else if (globaltimer_ns() - t_start > A.timeout_ns) {
                    atomicExch(A.scratch + SCR_TIMEOUT, 1ull);
                    stop = 1;
                }
            }
            stop = __shfl_sync(FULL_MASK, stop, 0);
            if (stop) {
                if (active) {
                    if (MODE == 1 || MODE == 2) mixed_to64(m, x);
                    if (PAIR && !in64) tf_unstate(T, x);
                    if (PAIR && in64) held64(T, x);
                    store_full(A, id, x, GT_RAY_TIMEOUT, n, nan(""));
                }
                if (!one_shot) {
                    for (;;) { // drain the queue without integrating
                        unsigned long long base = 0;
                        if (lane == 0) base = atomicAdd(next, 32ull);
                        base = __shfl_sync(FULL_MASK, base, 0);
                        if (base >= (unsigned long long)n_work) break;
                        const int64_t w = (int64_t)base + lane;
                        if (w < n_work) {
                            if (w < A.n_fresh && A.states.t) {
                                if (A.status) A.status[w] = GT_RAY_TIMEOUT; // state untouched
                                if (A.nsteps) A.nsteps[w] = 0;
                            } else if (w < A.n_fresh) {
                                const int64_t pix = A.fresh_ids ? A.fresh_ids[w] : w;
                                const int c = A.n_cams > 1 ? find_camera(cams, A.n_cams, pix) : 0;
                                if (!picked(c)) continue;
                                const double r0 = rays ? rays->r0 : cams[c].r0;
                                const double th0 = rays ? rays->theta0[pix] : cams[c].th0;
                                store_ray(A, (A.fresh_ids && A.compact_out) ? w : pix, 0.0, r0,
                                          th0, 0.0, GT_RAY_TIMEOUT, 0);
                            } else {
                                const ParkItem &p = A.in_items[w - A.n_fresh];
                                if (!picked(p.cam)) continue;
                                Ray64 y;
                                y.t = p.t;
                                y.r = p.r;
                                y.th = p.th;
                                y.ph = p.ph;
                                y.pt = p.pt;
                                y.pr = p.pr;
                                y.pth = p.pth;
                                y.pph = p.pph;
                                store_full(A, p.id, y, GT_RAY_TIMEOUT, p.n, nan(""));
                            }
                        }
                    }
                }
                return;
            }
        }
        if (!active) continue;

        // ---- one RK4 step
        int status = -1;
        if (PAIR) {
            // GT_MODE_FP64 takes Manko-Novikov steps below 4M in FP64: next to the ergosurface
            // 1/A^2 amplifies the rounding of the field, where 48 bits show against 53
            const PairSpacetime &pc = SINGLE ? A.pair : rays ? pr_ray : cams[cam].pair;
            // (the zone's precision is the mixed mode's: steps up to the axis itself)
            const float rho_min = MODE == 5 ? PAIR_RHO_STEPS * A.sp_tf.a : 0.0f;
            const bool hard = KEEP64 && (in64 || T.r.a - pc.r_plus.a < pc.r_hard);
            DF h;
            ++n;
            if (!hard && pair_step<KIND>(pc, tab, T, A.sp_tf, A.w6_tf, rho_min, h)) {
                if (tf_greater(T.r, r_esc_t))
                    status = GT_RAY_ESCAPED;
                else if (h.hi < A.h_thr_df.hi || (h.hi == A.h_thr_df.hi && h.lo < A.h_thr_df.lo))
                    status = GT_RAY_HORIZON;
                else if ((int64_t)n >= A.n_steps)
                    status = GT_RAY_MAXSTEPS;
                // the ring is tested after the escape and before the horizon
                if (MODE == 4 && A.disk.on && status != GT_RAY_ESCAPED &&
                    in_disk(A.disk, tf_to(T.r), tf_to(T.th)))
                    status = GT_RAY_DISK;
                if (status >= 0) tf_unstate(T, x);
            } else {
                Ray64 y;
                if (in64)
                    held64(T, x);
                else
                    tf_unstate(T, x);
                const double h64 = rk4_step64_call<KIND>(rays ? st : cams[cam].st, x, A.sp, A.w6, y);
                n_f64 += 4;
                if (!isfinite(h64) || !finite6(y)) {
                    status = GT_RAY_NONFINITE;
                } else {
                    x = y;
                    status = exit_status(x.r, h64, r_esc, A.sp, n, A.n_steps);
                    if (MODE == 4 && A.disk.on && status != GT_RAY_ESCAPED &&
                        in_disk(A.disk, x.r, x.th))
                        status = GT_RAY_DISK;
                    const float r = (float)x.r;
                    in64 = KEEP64 && (r - pc.r_plus.a < pc.r_hard ||
                                      r * fabsf(__sinf((float)x.th)) < rho_min);
                    if (in64)
                        hold64(x, T);
                    else
                        tf_state(x, T);
                }
            }
            if (ZONE && status < 0 && tf_greater(T.r, r_out_t)) { // leave the zone
                bool ok;
                tf_unstate(T, x);
                park(A, id, n, cam, x, &ok);
                if (ok) {
                    active = false;
                    atomicAdd(A.scratch + SCR_ZONE_STEPS, (unsigned long long)(n - n_entry));
                    if (n_f64) atomicAdd(A.scratch + SCR_ZONE_F64, (unsigned long long)n_f64);
                }
            }
        } else if (MODE == 0 || MODE == 3) {
            Ray64 y;
            const double h = step64<KIND>(A, st, x, y);
            if (MODE == 3) n_f64 += 4;
            ++n;
            if (!isfinite(h) || !finite6(y)) {
                status = GT_RAY_NONFINITE;
            } else {
                x = y;
                status = exit_status(x.r, h, r_esc, A.sp, n, A.n_steps);
                // the ring is tested after the escape and before the horizon
                if (A.disk.on && status != GT_RAY_ESCAPED && in_disk(A.disk, x.r, x.th))
                    status = GT_RAY_DISK;
                if (MODE == 3 && status < 0 && x.r > 1.25 * r_sw) { // leave the FP64 zone
                    bool ok;
                    park(A, id, n, cam, x, &ok);
                    if (ok) {
                        active = false;
                        atomicAdd(A.scratch + SCR_ZONE_STEPS, (unsigned long long)(n - n_entry));
                        if (n_f64) atomicAdd(A.scratch + SCR_ZONE_F64, (unsigned long long)n_f64);
                    }
                }
            }
        } else if (MODE == 1) {
            double h;
            bool ok = true;
            if ((double)m.r.hi < r_sw) { // the zone inline
                mixed_to64(m, x);
                if (A.zone_df && inline_zone_step<KIND>(rays ? pr_ray : cams[cam].pair, tab, x, A.sp_tf,
                                                        A.w6_tf, h)) {
                    mixed_from64(x, m);
                } else {
                    Ray64 y;
                    h = rk4_step64_call<KIND>(st, x, A.sp, A.w6, y);
                    n_f64 += 4;
                    ok = isfinite(h) && finite6(y);
                    if (ok) mixed_from64(y, m);
                }
            } else {
                RayMixed keep = m;
                h = (double)rk4_step32<KIND>(stf, m, spf, w6f);
                ok = isfinite(h) && isfinite(m.t.hi) && isfinite(m.r.hi) && isfinite(m.th.hi) &&
                     isfinite(m.ph.hi) && isfinite(m.pr.hi) && isfinite(m.pth.hi);
                if (!ok) m = keep;
            }
            ++n;
            if (!ok) {
                status = GT_RAY_NONFINITE;
                mixed_to64(m, x);
            } else {
                const double r_now = f2_to(m.r);
                status = exit_status(r_now, h, r_esc, A.sp, n, A.n_steps);
                if (A.disk.on && status != GT_RAY_ESCAPED && in_disk(A.disk, r_now, f2_to(m.th)))
                    status = GT_RAY_DISK;
                if (status >= 0) {
                    mixed_to64(m, x);
                } else if (n == rp_next) {
                    rp_next = rp_next + (uint32_t)A.reproject_every < rp_next
                                  ? 0xFFFFFFFFu
                                  : rp_next + (uint32_t)A.reproject_every;
                    mixed_to64(m, x);
                    reproject_pr(st, x);
                    m.pr = f2_from(x.pr);
                }
            }
        } else { // MODE 2: FP32 steps only, exit tests in FP32
            // What bounds it: issue slots with four warps a scheduler (the FP32 pipe is busy 73 % of
            // the cycles, a slot used in 83 %), the dependent chain of a step with fewer -- and a
            // terminating image ends on its longest rays, 450,000 steps of a lone warp where the
            // mean is 250,000.  Votes, refills and exit tests per step, three branches around the
            // stage rotations and the spacetime's constants in registers cost both.  In the
            // flush-to-zero build a step is 396 instructions (Kerr) and 1,127 (Manko-Novikov), 482
            // and 1,318 with all of these; a lone Kerr warp takes 686 cycles a step (1,284), a full
            // chip 481 a warp (641); Manko-Novikov 1,611 (2,550) and 1,331 (1,676).  Two steps per
            // iteration spare the copy of the state but not the instruction cache: a lone Kerr
            // warp 665 cycles, a full chip 530, Manko-Novikov 2,630 and 1,500.
            // Steps back to back until some lane of the warp has something to do: an exit, the
            // zone, a re-projection, a stage angle the fast step does not take.  One test covers
            // them all (the sum is finite only if every coordinate is; r within [r_switch,
            // r_escape) and h at or above the horizon's step are false for NaN); the exact tests
            // below decide.  128 steps at most, for the watchdog.
            const uint32_t n_event = rp_next < n_last ? rp_next : n_last;
            const SpacetimeF &sf = SINGLE ? A.stf : stf;
            RayMixed keep;
            float h, turn;
            bool event;
            for (int q = 0;;) {
                keep = m;
                if (KIND != KIND_ANY)
                    h = rk4_step32_fast<KIND, PRECISE>(sf, m, spf, w6f, turn);
                // one branch a step, none between its stages: a lone warp of Kerr rays with
                // spacetimes of their own takes 374 ns a step (499 with a branch a stage)
                else if (sf.kind == KIND_KERR)
                    h = rk4_step32_fast<KIND_KERR, PRECISE, true>(sf, m, spf, w6f, turn);
                else
                    h = rk4_step32_fast<KIND_MN, PRECISE, true>(sf, m, spf, w6f, turn);
                ++n;
                const float sum = ((m.t.hi + m.th.hi) + (m.ph.hi + m.pr.hi)) + m.pth.hi;
                event = !(m.r.hi < r_esc_f.hi && m.r.hi >= r_sw_f && h >= h_thr_f &&
                          turn <= 0.25f && fabsf(sum) <= 3.4028234e38f && n != n_event);
                if (__any_sync(live, event || A.disk.on) || ++q == 128) break;
            }
            if (!event && !A.disk.on) continue;
            if (!(turn <= 0.25f)) {
                m = keep;
                h = rk4_step32_call<KIND, PRECISE>(sf, m, spf, w6f);
            }
            const bool ok = isfinite(h) && isfinite(m.t.hi) && isfinite(m.r.hi) &&
                            isfinite(m.th.hi) && isfinite(m.ph.hi) && isfinite(m.pr.hi) &&
                            isfinite(m.pth.hi);
            if (!ok) {
                m = keep;
                status = GT_RAY_NONFINITE;
            } else if (m.r.hi > r_esc_f.hi || (m.r.hi == r_esc_f.hi && m.r.lo > r_esc_f.lo)) {
                status = GT_RAY_ESCAPED;
            } else if (A.disk.on && in_disk(A.disk, f2_to(m.r), f2_to(m.th))) {
                status = GT_RAY_DISK;
            } else if (h < h_thr_f) {
                status = GT_RAY_HORIZON;
            } else if ((int64_t)n >= A.n_steps) {
                status = GT_RAY_MAXSTEPS;
            } else if (m.r.hi < r_sw_f) { // enter the FP64 zone: hand the ray over
                mixed_to64(m, x);
                bool parked;
                park(A, id, n, cam, x, &parked);
                if (parked) active = false;
            } else if (n == rp_next) {
                rp_next = rp_next + (uint32_t)A.reproject_every < rp_next
                              ? 0xFFFFFFFFu
                              : rp_next + (uint32_t)A.reproject_every;
                mixed_to64(m, x);
                SpacetimeC st64;
                if (rays) {
                    CamDesc d;
                    d.M = rays->M;
                    d.S = rays->spin[id] * rays->M * rays->M;
                    d.Q = rays->q[id];
                    d.r0 = rays->r0;
                    d.th0 = rays->theta0[id];
                    d.fov_deg = 90.0;
                    d.res_x = d.res_y = 1;
                    d.offset = 0;
                    setup_desc(d, A.flags, rays->r_switch);
                    st64 = d.st;
                } else {
                    st64 = cams[cam].st;
                }
                reproject_pr(st64, x);
                m.pr = f2_from(x.pr);
            }
            if (status >= 0) mixed_to64(m, x);
        }
        if (status >= 0) {
            if (ZONE) {
                atomicAdd(A.scratch + SCR_ZONE_STEPS, (unsigned long long)(n - n_entry));
                if (n_f64) atomicAdd(A.scratch + SCR_ZONE_F64, (unsigned long long)n_f64);
            }
            double z = nan("");
            if (status == GT_RAY_DISK && A.z) z = redshift64<KIND>(cams[cam].st, cams[cam].gl_tt, x);
            store_full(A, id, x, status, n, z);
            active = false;
        }
    }
}

} // namespace
} // namespace gt
