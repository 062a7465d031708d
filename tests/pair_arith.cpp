// pair_arith.cpp -- host check of the double-float step's arithmetic (csrc/pair.cuh) against
// long double: product, sum, fused forms, reciprocal, inverse square root, exp, sin/cos and
// the three-float coordinate on seeded operands; the Kerr and Manko-Novikov rates at random
// phase-space points (the ergosurface and the neighbourhood of the horizon included), beside
// the same rates in FP64 and in the renormalised double-float of df.cuh; and whole RK4
// trajectories of camera-like rays against long double, beside the FP64 ones.
// Prints one JSON line.
#include <math.h>
#include <stdint.h>
#include <stdio.h>

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
#include "../paper_2310_15183_gb300/csrc/zone_df.cuh"

using namespace gt;

static const PairTables TAB = make_pair_tables();
struct Exp {
    DF operator()(DF a) const { return p_exp(a, &TAB); }
};

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
static DF rnd()
{
    const double m = uni(1, 2) * ldexp(1.0, (int)floor(uni(-30, 30)));
    return DF(uni(0, 1) < 0.5 ? -m : m);
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

static bool rates_pair(const PairSpacetime &c, DF rp, DF s, DF cs, DF pr, DF pth, TF pt, TF pph,
                       Rates<DF> &o)
{
    if (c.kind == KIND_KERR) {
        kerr_rates_pair(c, rp, s, cs, pr, pth, pt, pph, o);
        return true;
    }
    float ex[4];
    mn_rates_pair(c, rp, s, cs, pr, pth, pt, pph, Exp(), o, ex);
    return fmaxf(fabsf(ex[0]), fabsf(ex[1])) <= 24 && fmaxf(fabsf(ex[2]), fabsf(ex[3])) <= 48;
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
struct StateTF {
    TF t, r, th, ph, pr, pth, pt, pph;
};
static void rk4_pair(const PairSpacetime &c, StateTF &x, TF sp, TF w6)
{ // the stages of the kernels' pair_step
    const DF rp0 = tf_diff(x.r, c.r_plus);
    DF rp = rp0, pr = tf_pair(x.pr), pth = tf_pair(x.pth), h(0, 0), s1, c1;
    p_sincos(tf_pair(x.th), x.th.c, &TAB, &s1, &c1);
    DF s = s1, cs = c1;
    Rates<DF> k, acc;
    for (int i = 0; i < 4; i++) {
        rates_pair(c, rp, s, cs, pr, pth, x.pt, x.pph, k);
        if (i == 0) {
            h = p_norm(p_mul3(p_rcp(k.dt), sp));
            if (h.hi < 0) h = p_neg(h);
            acc = k;
        } else {
            const float w = i < 3 ? 2.0f : 1.0f;
            auto add = [&](DF &a, DF b) { a = p_add(a, p_scale(b, w)); };
            add(acc.dt, k.dt);
            add(acc.dr, k.dr);
            add(acc.dth, k.dth);
            add(acc.dph, k.dph);
            add(acc.dpr, k.dpr);
            add(acc.dpth, k.dpth);
        }
        if (i < 3) {
            const DF d = p_scale(h, i < 2 ? 0.5f : 1.0f);
            rp = p_norm(p_fma(d, k.dr, rp0));
            pr = p_fma(d, k.dpr, tf_pair(x.pr));
            pth = p_fma(d, k.dpth, tf_pair(x.pth));
            p_rotate(s1, c1, p_norm(p_mul(d, k.dth)), &s, &cs);
        }
    }
    const DF w = p_norm(p_mul3(h, w6));
    auto upd = [&](TF &a, DF b) { a = tf_add(a, p_norm(p_mul(w, b))); };
    upd(x.t, acc.dt);
    upd(x.r, acc.dr);
    upd(x.th, acc.dth);
    upd(x.ph, acc.dph);
    upd(x.pr, acc.dpr);
    upd(x.pth, acc.dpth);
}

// 2-norm errors, relative to the 2-norm of the truth, of t, r, theta, phi over a small frame
static void frame(double M, double S, double Q, double r0, double th0, int n, const char *name)
{
    const Constants k = constants(M, S, Q);
    const double V = tan(37.5 * M_PI / 180) / r0;
    LD nn[4] = {}, ep[4] = {}, ef[4] = {};
    for (int id = 0; id < 30; id++) {
        const double al = V * (2.0 * (id % 6) - 5) / 5, be = V * (2.0 * (id / 6) - 4) / 4;
        State<double> x = {0, r0, th0, 0, -1, be * r0 * r0, -1, al * r0 * r0 * sin(th0)};
        Rates<double> o;
        for (int it = 0; it < 60; it++) { // p_t from H = 0
            rates_t<double>(k.c, x.r, x.th, x.pr, x.pth, x.pt, x.pph, o);
            x.pt -= (o.dt * x.pt + o.dph * x.pph + o.dr * x.pr + o.dth * x.pth) / (2 * o.dt);
        }
        rates_t<double>(k.c, x.r, x.th, x.pr, x.pth, x.pt, x.pph, o);
        const double sc = 1 / fabs(o.dt);
        x.pr *= sc;
        x.pth *= sc;
        x.pt *= sc;
        x.pph *= sc;
        State<LD> y = {x.t, x.r, x.th, x.ph, x.pr, x.pth, x.pt, x.pph};
        StateTF z = {tf(x.t), tf(x.r), tf(x.th), tf(x.ph), tf(x.pr), tf(x.pth), tf(x.pt), tf(x.pph)};
        for (int i = 0; i < n; i++) {
            rk4<double>(k.c, x, 1.5e-4);
            rk4<LD>(k.l, y, (LD)1.5e-4);
            rk4_pair(k.p, z, tf(1.5e-4), tf(1.0 / 6.0));
        }
        const LD v[4] = {y.t, y.r, y.th, y.ph};
        const double d[4] = {x.t, x.r, x.th, x.ph};
        const TF q[4] = {z.t, z.r, z.th, z.ph};
        for (int j = 0; j < 4; j++) {
            nn[j] += v[j] * v[j];
            ep[j] += (tf_to(q[j]) - v[j]) * (tf_to(q[j]) - v[j]);
            ef[j] += (d[j] - v[j]) * (d[j] - v[j]);
        }
    }
    printf("\"%s\": {\"pair\": [%.2e, %.2e, %.2e, %.2e], \"f64\": [%.2e, %.2e, %.2e, %.2e]}, ", name,
           (double)sqrtl(ep[0] / nn[0]), (double)sqrtl(ep[1] / nn[1]), (double)sqrtl(ep[2] / nn[2]),
           (double)sqrtl(ep[3] / nn[3]), (double)sqrtl(ef[0] / nn[0]), (double)sqrtl(ef[1] / nn[1]),
           (double)sqrtl(ef[2] / nn[2]), (double)sqrtl(ef[3] / nn[3]));
}

static void rates(double M, double S, double Q, double lo, double hi, const char *name)
{
    const Constants k = constants(M, S, Q);
    const SpacetimeT<DF> cd = to_df(k.c);
    std::vector<double> e[3]; // pair, df, f64
    for (int i = 0; i < 10000; i++) {
        const double r = k.c.r_plus + uni(lo, hi), th = uni(1e-3, M_PI - 1e-3);
        const double pr = uni(-2, 2), pth = uni(-3, 3), pt = -1, pph = uni(-4, 4);
        Rates<LD> oL;
        Rates<double> o6;
        Rates<DF> op, od;
        rates_t<LD>(k.l, r, th, pr, pth, pt, pph, oL);
        rates_t<double>(k.c, r, th, pr, pth, pt, pph, o6);
        DF s, cs;
        const TF tt = tf(th);
        p_sincos(tf_pair(tt), tt.c, &TAB, &s, &cs);
        if (!rates_pair(k.p, tf_diff(tf(r), k.p.r_plus), s, cs, DF(pr), DF(pth), tf(pt), tf(pph), op))
            continue;
        const DF S0(sin(th)), C0(cos(th));
        if (Q == 0)
            kerr_rates_sc<DF>(cd, DF(r), S0, C0, DF(pr), DF(pth), DF(pt), DF(pph), od);
        else
            mn_rates_sc<DF>(cd, DF(r), S0, C0, DF(pr), DF(pth), DF(pt), DF(pph), od);
        const LD v[6] = {oL.dt, oL.dr, oL.dth, oL.dph, oL.dpr, oL.dpth};
        const LD w[3][6] = {{ld(op.dt), ld(op.dr), ld(op.dth), ld(op.dph), ld(op.dpr), ld(op.dpth)},
                            {ld(od.dt), ld(od.dr), ld(od.dth), ld(od.dph), ld(od.dpr), ld(od.dpth)},
                            {o6.dt, o6.dr, o6.dth, o6.dph, o6.dpr, o6.dpth}};
        LD scale = 0;
        bool fin = true;
        for (int j = 0; j < 6; j++) {
            scale = fmaxl(scale, fabsl(v[j]));
            fin = fin && isfinite(v[j]) && isfinite(w[0][j]) && isfinite(w[1][j]);
        }
        if (!fin) continue;
        for (int m = 0; m < 3; m++) {
            LD x = 0;
            for (int j = 0; j < 6; j++) x = fmaxl(x, fabsl(w[m][j] - v[j]) / scale);
            e[m].push_back((double)x);
        }
    }
    printf("\"%s\": {\"n\": %zu", name, e[0].size());
    const char *which[3] = {"pair", "df", "f64"};
    for (int m = 0; m < 3; m++) {
        std::sort(e[m].begin(), e[m].end());
        printf(", \"%s\": [%.2e, %.2e]", which[m], e[m][e[m].size() / 2],
               e[m][(size_t)(0.99 * (double)(e[m].size() - 1))]);
    }
    printf("}, ");
}

int main()
{
    LD w[9] = {};
    for (int i = 0; i < 200000; i++) {
        const DF a = rnd(), b = rnd(), c = rnd();
        auto rel = [](LD got, LD want, LD scale) { return fabsl(got - want) / scale; };
        const LD A = ld(a), B = ld(b), C = ld(c);
        w[0] = fmaxl(w[0], rel(ld(p_mul(a, b)), A * B, fabsl(A * B)));
        w[1] = fmaxl(w[1], rel(ld(p_add(a, b)), A + B, fabsl(A) + fabsl(B)));
        w[2] = fmaxl(w[2], rel(ld(p_fma(a, b, c)), A * B + C, fabsl(A * B) + fabsl(C)));
        w[3] = fmaxl(w[3], rel(ld(p_rcp(a)), 1 / A, fabsl(1 / A)));
        const DF q(fabs((double)A));
        w[4] = fmaxl(w[4], rel(ld(p_rsqrt(q)), 1 / sqrtl(ld(q)), 1 / sqrtl(ld(q))));
        const DF x(uni(-8, 8));
        w[5] = fmaxl(w[5], rel(ld(p_exp(x, &TAB)), expl(ld(x)), expl(ld(x))));
        const TF th = tf(uni(-100, 100));
        DF s, cs;
        p_sincos(tf_pair(th), th.c, &TAB, &s, &cs);
        w[6] = fmaxl(w[6], fmaxl(fabsl(ld(s) - sinl(ld(th))), fabsl(ld(cs) - cosl(ld(th)))));
        const double d0 = uni(-1, 1) * ldexp(1.0, -(int)uni(9, 40));
        const LD a0 = atan2l(ld(s), ld(cs)) + (LD)(float)d0; // the angle of the pair, turned
        DF s2, c2;
        p_rotate(s, cs, DF((float)d0, 0.0f), &s2, &c2);
        w[8] = fmaxl(w[8], fmaxl(fabsl(ld(s2) - sinl(a0)), fabsl(ld(c2) - cosl(a0))));
        const TF t = tf((LD)uni(-20, 20) + uni(-1, 1) * 1e-18L);
        const DF d(uni(-1, 1) * ldexp(1.0, -(int)uni(0, 40)));
        if (fabsl(ld(t)) > 1e-3) w[7] = fmaxl(w[7], rel(ld(tf_add(t, d)), ld(t) + ld(d), fabsl(ld(t)) + fabsl(ld(d))));
    }
    printf("{\"mul\": %.2e, \"add\": %.2e, \"fma\": %.2e, \"rcp\": %.2e, \"rsqrt\": %.2e, \"exp\": %.2e, "
           "\"sincos\": %.2e, \"tf_add\": %.2e, \"rotate\": %.2e, ",
           (double)w[0], (double)w[1], (double)w[2], (double)w[3], (double)w[4], (double)w[5],
           (double)w[6], (double)w[7], (double)w[8]);
    printf("\"rates\": {");
    rates(1, 0.9, 0, 1e-4, 0.1, "kerr near r_+");
    rates(1, 0.9, 0, 0.1, 20, "kerr");
    rates(0.5, 0, 0, 0.1, 20, "schwarzschild");
    rates(0.5, 0.24, 2, 0.05, 0.4, "mn inner");
    rates(0.5, 0.24, 2, 0.4, 1.4, "mn zone");
    rates(0.5, 0.24, -2, 0.4, 1.4, "mn zone q < 0");
    rates(0.5, 0.24, 2, 1.4, 20, "mn outside");
    rates(0.5, 0.025, 2, 1.4, 20, "mn low spin outside");
    printf("\"\": 0}, \"frames\": {");
    frame(0.5, 0, 0, 10, 1.26, 2000, "schwarzschild 2000");
    frame(0.5, 0.2, 0, 15, 1.3, 2000, "kerr 2000");
    frame(0.5, 0.24, 2, 15, 1.3, 2000, "mn 2000");
    frame(0.5, 0.24, 2, 15, 1.3, 20000, "mn 20000");
    frame(0.5, 0.24, 2, 1.9, 1.3, 4000, "mn zone 4000");
    printf("\"\": 0}}\n");
    return 0;
}
