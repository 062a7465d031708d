// pair_route.cpp -- host check of the double-float step the kernels run (pair_step of
// csrc/pair.cuh) at the limits of what it accepts.  The first argument names the part; each
// prints one JSON line.
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#define GT_HD inline
typedef long double LD;
static inline void sincos_t(double x, double *s, double *c) { *s = sin(x); *c = cos(x); }
static inline double exp_t(double x) { return exp(x); }
static inline double rcp_t(double x) { return 1.0 / x; }
static inline double rsqrt_t(double x) { return 1.0 / sqrt(x); }
static inline double fma_t(double a, double b, double c) { return fma(a, b, c); }
static inline void sincos_t(LD x, LD *s, LD *c) { *s = sinl(x); *c = cosl(x); }
static inline LD exp_t(LD x) { return expl(x); }
static inline LD rcp_t(LD x) { return 1.0L / x; }
static inline LD rsqrt_t(LD x) { return 1.0L / sqrtl(x); }
static inline LD fma_t(LD a, LD b, LD c) { return a * b + c; }
namespace gt {
using ::exp_t;
using ::fma_t;
using ::rcp_t;
using ::rsqrt_t;
using ::sincos_t;
} // namespace gt

#include "../paper_2310_15183_gb300/csrc/pair.cuh"

using namespace gt;

static const PairTables TAB = make_pair_tables();

static uint64_t g_state = 0x15183ull;
static double uni(double lo, double hi)
{ // splitmix64
    uint64_t z = (g_state += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return lo + (hi - lo) * (double)(z >> 11) * (1.0 / 9007199254740992.0);
}
static LD ld(DF a) { return (LD)a.hi + (LD)a.lo; }
static LD ld(TF a) { return (LD)a.a + (LD)a.b + (LD)a.c; }
static DF df(LD v) { const float h = (float)v; return DF(h, (float)(v - h)); }
static TF tf(LD v)
{
    TF t;
    t.a = (float)v;
    const LD r = v - t.a;
    t.b = (float)r;
    t.c = (float)(r - t.b);
    return t;
}
// constants of one spacetime in double (as the set-up kernel forms them), long double, pairs
struct Constants {
    SpacetimeC c = {};
    SpacetimeT<LD> l = {};
    PairSpacetime p = {};
};
static Constants constants(double M, double S, double Q)
{
    Constants k;
    SpacetimeC &c = k.c;
    SpacetimeT<LD> &l = k.l;
    c.M = M;
    l.M = M;
    if (Q != 0) {
        c.kind = KIND_MN;
        const double sm = S / M, al = (-M + sqrt(M * M - sm * sm)) / sm;
        const double kk = M * (1 - al * al) / (1 + al * al), be = Q * M * M * M / (kk * kk * kk);
        c.alpha = al;
        c.k = kk;
        c.ik = 1 / kk;
        c.two_beta = 2 * be;
        c.three_beta2 = 3 * be * be;
        c.c_g = (1 - al * al) * (1 - al * al) / (kk * kk);
        c.w_inf = 4 * kk * al / (1 - al * al);
        c.k2 = kk * kk;
        c.inv_k2 = 1 / (kk * kk);
        c.two_k = 2 * kk;
        c.r_plus = M + kk;
        const LD a = al, q = kk, b = be;
        l.alpha = a;
        l.k = q;
        l.ik = 1 / q;
        l.two_beta = 2 * b;
        l.three_beta2 = 3 * b * b;
        l.c_g = (1 - a * a) * (1 - a * a) / (q * q);
        l.w_inf = 4 * q * a / (1 - a * a);
        l.k2 = q * q;
        l.inv_k2 = 1 / (q * q);
        l.two_k = 2 * q;
        l.r_plus = (LD)M + q;
    } else {
        c.kind = KIND_KERR;
        c.a = S / M;
        c.a2 = c.a * c.a;
        c.r_plus = M + sqrt(M * M - c.a2);
        l.a = c.a;
        l.a2 = l.a * l.a;
        l.r_plus = M + sqrtl((LD)M * M - l.a2);
    }
    l.kind = k.p.kind = c.kind;
    PairSpacetime &p = k.p;
    p.r_plus = tf(l.r_plus);
    p.r_plus2 = df(l.r_plus);
    p.split = df(2 * (l.r_plus - M));
    p.a = df(l.a);
    p.a2 = df(l.a2);
    p.ik = tf(l.ik);
    p.alpha = tf(l.alpha);
    p.two_beta = df(l.two_beta);
    p.three_beta2 = df(l.three_beta2);
    p.c_g = tf(l.c_g);
    p.w_inf = tf(l.w_inf);
    p.k2 = tf(l.k2);
    p.inv_k2 = tf(l.inv_k2);
    p.two_k = tf(l.two_k);
    return k;
}

template <class T>
static void rates_t(const SpacetimeT<T> &c, T r, T th, T pr, T pth, T pt, T pph, Rates<T> &o)
{
    T s, cs;
    sincos_t(th, &s, &cs);
    if (c.kind == KIND_KERR)
        kerr_rates_sc<T>(c, r, s, cs, pr, pth, pt, pph, o);
    else
        mn_rates_sc<T>(c, r, s, cs, pr, pth, pt, pph, o);
}

// ------------------------------------------------------------------ trajectories
template <class T>
struct State {
    T t, r, th, ph, pr, pth, pt, pph;
};
template <class T>
static void rk4(const SpacetimeT<T> &c, State<T> &x, T sp)
{
    Rates<T> k[4];
    rates_t<T>(c, x.r, x.th, x.pr, x.pth, x.pt, x.pph, k[0]);
    const T h = sp / k[0].dt < 0 ? -sp / k[0].dt : sp / k[0].dt;
    for (int i = 1; i < 4; i++) {
        const T d = i < 3 ? h / 2 : h;
        rates_t<T>(c, x.r + d * k[i - 1].dr, x.th + d * k[i - 1].dth, x.pr + d * k[i - 1].dpr,
                   x.pth + d * k[i - 1].dpth, x.pt, x.pph, k[i]);
    }
    const T w = h * (T)(1.0 / 6.0);
    x.t += w * (k[0].dt + 2 * k[1].dt + 2 * k[2].dt + k[3].dt);
    x.r += w * (k[0].dr + 2 * k[1].dr + 2 * k[2].dr + k[3].dr);
    x.th += w * (k[0].dth + 2 * k[1].dth + 2 * k[2].dth + k[3].dth);
    x.ph += w * (k[0].dph + 2 * k[1].dph + 2 * k[2].dph + k[3].dph);
    x.pr += w * (k[0].dpr + 2 * k[1].dpr + 2 * k[2].dpr + k[3].dpr);
    x.pth += w * (k[0].dpth + 2 * k[1].dpth + 2 * k[2].dpth + k[3].dpth);
}

static RayTF ray(const State<double> &x)
{
    RayTF z;
    z.t = tf_from(x.t);
    z.r = tf_from(x.r);
    z.th = tf_from(x.th);
    z.ph = tf_from(x.ph);
    z.pr = tf_from(x.pr);
    z.pth = tf_from(x.pth);
    z.pt = tf_from(x.pt);
    z.pph = tf_from(x.pph);
    return z;
}

// A camera ray's initial state: direction (-1, be, al / sin th0) at r0, p_t from H = 0, scaled
// so that dt/dtau = 1.
static State<double> camera_ray(const Constants &k, double r0, double th0, double al, double be)
{
    State<double> x = {0, r0, th0, 0, -1, be * r0 * r0, -1, al * r0 * r0 * sin(th0)};
    Rates<double> o;
    for (int it = 0; it < 60; it++) {
        rates_t<double>(k.c, x.r, x.th, x.pr, x.pth, x.pt, x.pph, o);
        x.pt -= (o.dt * x.pt + o.dph * x.pph + o.dr * x.pr + o.dth * x.pth) / (2 * o.dt);
    }
    rates_t<double>(k.c, x.r, x.th, x.pr, x.pth, x.pt, x.pph, o);
    const double sc = 1 / fabs(o.dt);
    x.pr *= sc;
    x.pth *= sc;
    x.pt *= sc;
    x.pph *= sc;
    return x;
}

// Steps whose rates are finite and whose new state is not: an RK4 weight of 1e38 in place of 1/6.
static void new_state()
{
    int refused = 0, untouched = 0, taken = 0, n = 0;
    for (double Q : {0.0, 2.0}) {
        const Constants k = constants(0.5, 0.2, Q);
        for (int i = 0; i < 32; i++, n++) {
            const State<double> x = camera_ray(k, uni(6, 20), uni(0.5, 1.5), uni(-.05, .05), uni(-.05, .05));
            RayTF z = ray(x);
            const RayTF z0 = z;
            DF h;
            auto step = [&](double w) {
                return Q == 0 ? pair_step<KIND_KERR>(k.p, &TAB, z, tf_from(1.0), tf_from(w), 0.0f, h)
                              : pair_step<KIND_MN>(k.p, &TAB, z, tf_from(1.0), tf_from(w), 0.0f, h);
            };
            refused += !step(1e38);
            untouched += memcmp(&z, &z0, sizeof z) == 0;
            taken += step(1.0 / 6.0) && isfinite(z.t.a) && memcmp(&z, &z0, sizeof z) != 0;
        }
    }
    printf("{\"n\": %d, \"refused\": %d, \"untouched\": %d, \"taken\": %d}\n", n, refused, untouched, taken);
}

// Kernel's choice for a GT_MODE_FP64 camera ray: the pair step where pair_accurate, above 4M in
// Manko-Novikov and away from the axis, FP64 elsewhere.
static void route_step(const Constants &k, State<double> &x, RayTF &z, double sp)
{
    DF h;
    const TF t = tf_from(sp), w = tf_from(1.0 / 6.0);
    const float rho = PAIR_RHO_STEPS * t.a;
    const bool mn = k.c.kind == KIND_MN;
    if (!(mn && z.r.a < (float)(4 * k.c.M)) &&
        (mn ? pair_step<KIND_MN>(k.p, &TAB, z, t, w, rho, h) : pair_step<KIND_KERR>(k.p, &TAB, z, t, w, rho, h)))
        return;
    x.t = tf_to(z.t);
    x.r = tf_to(z.r);
    x.th = tf_to(z.th);
    x.ph = tf_to(z.ph);
    x.pr = tf_to(z.pr);
    x.pth = tf_to(z.pth);
    rk4<double>(k.c, x, sp);
    z = ray(x);
}

// End positions of `frames` seeded camera frames of both kinds against long double: the 2-norm
// error over a frame's 20 rays relative to the truth's, root mean square over the frames, of t,
// r, theta, phi, for the kernel's choice and for FP64; the geometric mean over the frames of the
// ratio of the two; and how many frames took pairs.
static void accuracy(int argc, char **argv)
{
    if (argc < 9) return;
    const long n = atol(argv[2]);
    const double spM = atof(argv[3]), lo = atof(argv[4]), hi = atof(argv[5]);
    const double th_lo = atof(argv[6]), th_hi = atof(argv[7]);
    const int frames = atoi(argv[8]);
    const double M = 0.5, sp = spM * M;
    double rms[2][4] = {}, lg[4] = {};
    int pairs = 0;
    for (int f = 0; f < frames; f++) {
        const bool mn = f % 2;
        const double spin = mn ? uni(0.1, 0.98) : (f % 4 ? 0.999 : 0.2) * uni(0, 1);
        const Constants k = constants(M, spin * M * M, mn ? (f % 4 == 1 ? 2.0 : -2.0) : 0.0);
        const double r0 = M * exp(uni(log(lo), log(hi))), th0 = exp(uni(log(th_lo), log(th_hi)));
        const double V = tan(uni(10, 60) * M_PI / 180) / r0;
        const bool pair = pair_accurate(M, r0, sp, n);
        pairs += pair;
        LD nn[4] = {}, e[2][4] = {};
        for (int id = 0; id < 20; id++) {
            State<double> x = camera_ray(k, r0, th0, V * (2.0 * (id % 5) - 4) / 4, V * (2.0 * (id / 5) - 3) / 3);
            State<LD> y = {x.t, x.r, x.th, x.ph, x.pr, x.pth, x.pt, x.pph};
            State<double> w = x;
            RayTF z = ray(x);
            long i = 0;
            for (; i < n && y.r <= 1.5 * r0 && y.r > 1.02 * k.c.r_plus; i++) {
                rk4<double>(k.c, x, sp);
                rk4<LD>(k.l, y, (LD)sp);
                if (pair) route_step(k, w, z, sp);
            }
            const LD v[4] = {y.t, y.r, y.th, y.ph};
            const double d[4] = {x.t, x.r, x.th, x.ph};
            const double q[4] = {tf_to(z.t), tf_to(z.r), tf_to(z.th), tf_to(z.ph)};
            for (int j = 0; j < 4; j++) {
                nn[j] += v[j] * v[j];
                const LD a = (pair ? q[j] : d[j]) - v[j], b = d[j] - v[j];
                e[0][j] += a * a;
                e[1][j] += b * b;
            }
        }
        for (int j = 0; j < 4; j++) {
            for (int m = 0; m < 2; m++) rms[m][j] += (double)(e[m][j] / nn[j]) / frames;
            lg[j] += 0.5 * log((double)(e[0][j] / e[1][j])) / frames;
        }
    }
    printf("{\"pairs\": %d, \"route\": [%.3e, %.3e, %.3e, %.3e], \"f64\": [%.3e, %.3e, %.3e, %.3e], \"ratio\": [%.3f, %.3f, %.3f, %.3f]}\n", pairs,
           sqrt(rms[0][0]), sqrt(rms[0][1]), sqrt(rms[0][2]), sqrt(rms[0][3]), sqrt(rms[1][0]),
           sqrt(rms[1][1]), sqrt(rms[1][2]), sqrt(rms[1][3]), exp(lg[0]), exp(lg[1]), exp(lg[2]), exp(lg[3]));
}

// The operations over all that the step gives them: exp to the exponent bounds, in units of
// 2^-45 + |x| 2^-47; sin/cos to the reduction's limit and the rotation by whole pairs, absolute.
static void operations()
{
    LD w[3] = {};
    for (int i = 0; i < 400000; i++) {
        const DF x = df((LD)uni(-48, 48) + uni(-1, 1) * 1e-9L);
        const LD want = expl(ld(x)), unit = ldexpl(1, -45) + fabsl(ld(x)) * ldexpl(1, -47);
        w[0] = fmaxl(w[0], fabsl(ld(p_exp(x, &TAB)) - want) / want / unit);
        const TF th = tf((LD)uni(-128, 128) + uni(-1, 1) * 1e-17L);
        DF s, c, s2, c2;
        p_sincos(tf_pair(th), th.c, &TAB, &s, &c);
        w[1] = fmaxl(w[1], fmaxl(fabsl(ld(s) - sinl(ld(th))), fabsl(ld(c) - cosl(ld(th)))));
        const DF d = df((LD)uni(-1, 1) * ldexpl(1, -9 - (int)uni(0, 30)) * (1 + uni(-1, 1) * 1e-8L));
        p_rotate(s, c, d, &s2, &c2);
        const LD a = atan2l(ld(s), ld(c)) + ld(d);
        w[2] = fmaxl(w[2], fmaxl(fabsl(ld(s2) - sinl(a)), fabsl(ld(c2) - cosl(a))));
    }
    printf("{\"exp\": %.3e, \"sincos\": %.3e, \"rotate\": %.3e}\n", (double)w[0], (double)w[1], (double)w[2]);
}

int main(int argc, char **argv)
{
    const char *part = argc > 1 ? argv[1] : "";
    if (!strcmp(part, "operations")) operations();
    if (!strcmp(part, "accuracy")) accuracy(argc, argv);
    if (!strcmp(part, "rule") && argc > 5)
        printf("%d\n", pair_accurate(atof(argv[2]), atof(argv[3]), atof(argv[4]), atol(argv[5])));
    if (!strcmp(part, "new_state")) new_state();
    return 0;
}
