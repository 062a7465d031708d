// pair.cuh -- the step of the double-float integrator: field evaluations on pairs of floats
// whose sums are not renormalised, and a ray state held in three floats per coordinate, so
// that a whole RK4 step runs on the FP32 pipes (host and device).
//
// What bounds it: a GB300 SM issues one FP64 warp instruction per ~19 cycles (64 cycles for
// a lone warp, conversions between float and double included) against four FP32 ones per
// cycle, so the arithmetic that replaces one FP64 operation may take up to ~60 FP32
// instructions before it loses.  The double-float operators of df.cuh cost 20 instructions
// for a sum and 7 for a product, most of them renormalisation.  Here a pair (hi, lo) stands
// for hi + lo with |lo| a few ulp(hi), and
//   product  p = fl(a.hi b.hi), its error by one FMA, then three FMAs for the cross terms,
//            lo * lo included: 5 instructions (with lo * lo kept, an un-renormalised operand
//            costs no precision: the error is 2^-24 of |lo| terms, not of their squares);
//   sum      TwoSum of the high parts, low parts added to its error: 8 instructions.
// This is the unnormalised pair arithmetic of Lange and Rump ("Faithfully rounded
// floating-point computations", 2020).  Operands are renormalised (3 instructions) only in
// front of a reciprocal or a square root.  exp and sin/cos take a table entry (Tang's
// table-driven method, 1989: 64 entries of 2^(j/64), 128 of sin and cos of j pi/64) and a
// short polynomial in the remainder.
//
// The state: an RK4 increment is about 1e-5 of the coordinate it moves, so a 53-bit state
// rounds away half an ulp per step and the sum of those roundings is what an FP64 run's
// error is made of.  Three floats (72 bits) take the increment without a conversion and
// without that rounding.
//
// Measured against the FP64 kernel it replaces for GT_MODE_FP64 camera rays (one GB300): 48,000
// Manko-Novikov rays x 2,000 steps 287 -> 38.6 ms (200,000 rays: 2.9e9 steps/s), Kerr 1.06e10
// steps/s; against the renormalised double-float zone step with an FP64 state, 40,000
// in-zone rays x 4,000 steps 242 -> 77.7 ms.  Against long double the end positions of 2,000 to
// 20,000 steps of 3e-4 M are off by 4e-17 to 1.6e-15 (t, r, theta, phi; relative 2-norm over a
// frame) where FP64's are off by 1.1e-15 to 7e-15 (tests/pair_arith.cpp).  That holds for many
// small steps away from the axis: pair_accurate and PAIR_RHO_STEPS below draw the line.
#pragma once

#include <stdint.h>

#include "df.cuh"
#include "spacetime.cuh"

namespace gt {

#ifdef __CUDA_ARCH__
#define GT_P_ADD(a, b) __fadd_rn((a), (b))
#define GT_P_MUL(a, b) __fmul_rn((a), (b))
#else
#define GT_P_ADD(a, b) ((a) + (b))
#define GT_P_MUL(a, b) ((a) * (b))
#endif

// ------------------------------------------------------------------ three floats
struct TF {
    float a, b, c; // a + b + c, |b| <= ulp(a)/2, |c| <= ulp(b)/2
};

GT_HD TF tf_from(double v)
{
    TF t;
    t.a = (float)v;
    const double r = v - (double)t.a;
    t.b = (float)r;
    t.c = (float)(r - (double)t.b);
    return t;
}

GT_HD double tf_to(TF t) { return (double)t.a + ((double)t.b + (double)t.c); }

// ------------------------------------------------------------------ pair arithmetic
GT_HD DF p_mul(DF a, DF b)
{
    const float p = GT_P_MUL(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.lo, b.lo, e);
    e = fmaf(a.hi, b.lo, e);
    return DF(p, fmaf(a.lo, b.hi, e));
}

GT_HD DF p_sq(DF a)
{
    const float p = GT_P_MUL(a.hi, a.hi);
    float e = fmaf(a.hi, a.hi, -p);
    e = fmaf(a.lo, a.lo, e);
    return DF(p, fmaf(GT_P_ADD(a.hi, a.hi), a.lo, e));
}

GT_HD DF p_add(DF a, DF b)
{
    const DF s = df_two_sum(a.hi, b.hi);
    return DF(s.hi, GT_P_ADD(s.lo, GT_P_ADD(a.lo, b.lo)));
}

GT_HD DF p_sub(DF a, DF b) { return p_add(a, DF(-b.hi, -b.lo)); }
GT_HD DF p_neg(DF a) { return DF(-a.hi, -a.lo); }

// a b + c
GT_HD DF p_fma(DF a, DF b, DF c)
{
    const float p = GT_P_MUL(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.lo, b.lo, e);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    const DF s = df_two_sum(p, c.hi);
    return DF(s.hi, GT_P_ADD(s.lo, GT_P_ADD(e, c.lo)));
}

// a c and a c + d with a constant of three floats.  A constant rounded to a pair would bias
// every step the same way (2^-49 of the increment, the size of an FP64 run's error); its third
// float enters the error term before that is rounded, so the bias averages out.
GT_HD DF p_mul3(DF a, TF c)
{
    const float p = GT_P_MUL(a.hi, c.a);
    float e = fmaf(a.hi, c.a, -p);
    e = fmaf(a.hi, c.c, fmaf(a.lo, c.b, e));
    e = fmaf(a.hi, c.b, e);
    return DF(p, fmaf(a.lo, c.a, e));
}
GT_HD DF p_fma3(DF a, TF c, DF d)
{
    const DF m = p_mul3(a, c);
    const DF s = df_two_sum(m.hi, d.hi);
    return DF(s.hi, GT_P_ADD(s.lo, GT_P_ADD(m.lo, d.lo)));
}

GT_HD DF p_add3(DF a, TF c)
{
    const DF s = df_two_sum(a.hi, c.a);
    return DF(s.hi, GT_P_ADD(s.lo, GT_P_ADD(c.b, GT_P_ADD(a.lo, c.c))));
}
GT_HD DF p_sub3(DF a, TF c)
{
    const TF m = {-c.a, -c.b, -c.c};
    return p_add3(a, m);
}

// c - a b
GT_HD DF p_fnma(DF a, DF b, DF c) { return p_fma(DF(-a.hi, -a.lo), b, c); }

// a + f and a f with a float; times a power of two
GT_HD DF p_addf(DF a, float f)
{
    const DF s = df_two_sum(a.hi, f);
    return DF(s.hi, GT_P_ADD(s.lo, a.lo));
}
GT_HD DF p_mulf(DF a, float f)
{
    const float p = GT_P_MUL(a.hi, f);
    return DF(p, fmaf(a.lo, f, fmaf(a.hi, f, -p)));
}
GT_HD DF p_scale(DF a, float pow2) { return DF(GT_P_MUL(a.hi, pow2), GT_P_MUL(a.lo, pow2)); }

// |lo| <= ulp(hi)/2 again: of a pair with |lo| below |hi|, and of any pair (after a
// cancellation lo may be as large as hi, and a product of such a pair is only a float's)
GT_HD DF p_norm(DF a) { return df_fast_two_sum(a.hi, a.lo); }
GT_HD DF p_renorm(DF a) { return df_two_sum(a.hi, a.lo); }

// 1/a: y an estimate of 1/hi to a few ulp, r = 1 - a y, 1/a = y (1 + r + r^2 + ...)
GT_HD DF p_rcp(DF v)
{
    const DF a = p_norm(v);
#ifdef __CUDA_ARCH__
    const float y = __fdividef(1.0f, a.hi);
#else
    const float y = 1.0f / a.hi;
#endif
    float r = fmaf(-a.hi, y, 1.0f);
    r = fmaf(-a.lo, y, r);
    return df_fast_two_sum(y, GT_P_MUL(y, fmaf(r, r, r)));
}

// 1/sqrt(a), as rsqrt_t of df.cuh with the residual formed from the pair product
GT_HD DF p_rsqrt(DF v)
{
    const DF a = p_norm(v);
#ifdef __CUDA_ARCH__
    const float y = rsqrtf(a.hi);
#else
    const float y = 1.0f / sqrtf(a.hi);
#endif
    const DF ay2 = p_mul(a, df_two_prod(y, y));
    const float r = GT_P_ADD(GT_P_ADD(1.0f, -ay2.hi), -ay2.lo); // 1 - hi exact (Sterbenz)
    return df_fast_two_sum(y, GT_P_MUL(y, GT_P_MUL(r, fmaf(0.375f, r, 0.5f))));
}

// ------------------------------------------------------------------ tables
constexpr int EXP_TAB = 64;  // 2^(j/64)
constexpr int TRIG_TAB = 128; // sin, cos of j pi/64

struct PairTables {
    TF ex[EXP_TAB];
    TF sc[TRIG_TAB][2]; // sin, cos
};

// Entries by their Taylor series in double (arguments below 0.7 and pi/4), as three floats: an
// entry serves thousands of steps, so its rounding would bias them all the same way.
constexpr TF table_entry(double v)
{
    const float a = (float)v;
    const float b = (float)(v - (double)a);
    return TF{a, b, (float)(v - (double)a - (double)b)};
}

constexpr PairTables make_pair_tables()
{
    PairTables t = {};
    for (int j = 0; j < EXP_TAB; j++) {
        const double x = 0.693147180559945309417 * (double)j / EXP_TAB;
        double sum = 1.0;
        for (int k = 24; k >= 1; k--) sum = 1.0 + sum * x / (double)k;
        t.ex[j] = table_entry(sum);
    }
    for (int j = 0; j < TRIG_TAB; j++) {
        const int q = ((j + 16) / 32) % 4, i = j - 32 * ((j + 16) / 32); // nearest quarter turn
        const double x = 3.14159265358979323846 * (double)i / 64.0, x2 = x * x;
        double s = 1.0, c = 1.0;
        for (int k = 12; k >= 1; k--) {
            s = 1.0 - s * x2 / (double)(2 * k * (2 * k + 1));
            c = 1.0 - c * x2 / (double)((2 * k - 1) * 2 * k);
        }
        s = s * x;
        const double sn = q == 0 ? s : q == 1 ? c : q == 2 ? -s : -c;
        const double cn = q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s;
        t.sc[j][0] = table_entry(sn);
        t.sc[j][1] = table_entry(cn);
    }
    return t;
}

// exp(a) for |a| <= 87: n = rint(64 a / ln 2), r = a - n ln2/64 (|r| < 0.0055), table times
// 1 + r + r^2/2 + ... + r^5/120 with r + r^2/2 in pairs and the rest (below 2^-24) in float.
// ln2/64 = L0 + L1 + L2: n L0 exact (11 bits by 13), n L1 a product pair, n L2 rounded.
GT_HD DF p_exp(DF a, const PairTables *__restrict__ tab)
{
    const float L0 = 0.010833740234375f;       // 11 bits of ln2/64
    const float L1 = -3.31553815158e-06f;      // float nearest ln2/64 - L0
    const float L2 = 2.57280464023e-14f;       // float nearest the rest
    const float nf = rintf(GT_P_MUL(a.hi, 92.3324826168937f));
    const int n = (int)nf;
    const float t0 = fmaf(-nf, L0, a.hi);
    const DF p = df_two_prod(nf, L1);
    const DF s = df_two_sum(t0, -p.hi);
    const DF r = df_two_sum(s.hi, GT_P_ADD(s.lo, fmaf(-nf, L2, GT_P_ADD(a.lo, -p.lo))));
    const float rh = r.hi, rl = r.lo;
    const DF q = df_two_prod(rh, rh);
    const float u = fmaf(rh, fmaf(rh, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f);
    const float c = GT_P_MUL(GT_P_MUL(q.hi, rh), u);
    const DF m = df_fast_two_sum(rh, GT_P_MUL(0.5f, q.hi));
    const DF em1(m.hi, GT_P_ADD(m.lo, GT_P_ADD(rl, fmaf(0.5f, q.lo, fmaf(rl, rh, c)))));
    const TF t = tab->ex[n & (EXP_TAB - 1)];
    const DF e = p_mul(DF(t.a, t.b), em1);
    const DF f = df_fast_two_sum(t.a, e.hi);
    const DF g(f.hi, GT_P_ADD(f.lo, GT_P_ADD(t.b, GT_P_ADD(t.c, e.lo))));
    const int k = (n >> 6) + 127; // 2^(n >> 6): |n >> 6| <= 126
#ifdef __CUDA_ARCH__
    const float sc = __int_as_float(k << 23);
#else
    const float sc = ldexpf(1.0f, k - 127);
#endif
    return p_scale(g, sc);
}

// sin and cos of the angle th (+ th2, a third part): k = rint(64 th / pi), the remainder
// d = th - k pi/64 (|d| < 0.025) rotates the table entry.  sin d = d + d^3 q, q = -1/6 +
// d^2/120 - d^4/5040; cos d - 1 = -d^2/2 + d^4 (1/24 - d^2/720), pairs where a term exceeds
// 2^-24 of one.  pi/64 = P0 + P1 + P2 with k P0, k P1 exact for |k| < 2^12 (|th| < 200).
GT_HD void p_sincos(DF th, float th2, const PairTables *__restrict__ tab, DF *so, DF *co)
{
    const float P0 = 0.0490875244140625f;         // 12 bits of pi/64
    const float P1 = -1.3917451724410057e-07f;    // the next 12 bits
    const float P2 = -2.72047367272e-11f;         // float nearest the rest
    const float kf = rintf(GT_P_MUL(th.hi, 20.3718327157626f));
    const int k = (int)kf;
    const float t0 = fmaf(-kf, P0, th.hi);
    const DF s = df_two_sum(t0, -GT_P_MUL(kf, P1));
    const DF p = df_two_prod(kf, P2);
    const DF w = df_two_sum(th.lo, -p.hi);
    const DF s2 = df_two_sum(s.hi, w.hi);
    const DF d(s2.hi, GT_P_ADD(GT_P_ADD(s2.lo, s.lo), GT_P_ADD(GT_P_ADD(th2, w.lo), -p.lo)));
    const DF d2 = p_sq(d);
    const float t = d2.hi;
    const float qf = GT_P_MUL(t, fmaf(t, -1.0f / 5040.0f, 1.0f / 120.0f));
    const float t2 = fmaf(GT_P_ADD(t, t), d2.lo, GT_P_MUL(t, t));
    // the float nearest 1/24 is 1.24e-9 above it
    const float pf = fmaf(t2, fmaf(t, -1.0f / 720.0f, 1.0f / 24.0f), GT_P_MUL(t2, -1.2417635e-09f));
    const DF q = p_addf(DF(-0.16666667163372039794921875f, 4.967053879312289e-09f), qf);
    const DF sd = p_fma(p_mul(d, d2), q, d);
    const DF cd(GT_P_MUL(-0.5f, d2.hi), fmaf(-0.5f, d2.lo, pf));
    const int j = k & (TRIG_TAB - 1);
    const TF S3 = tab->sc[j][0], C3 = tab->sc[j][1];
    const DF S(S3.a, S3.b), C(C3.a, C3.b);
    *so = p_add3(p_fma(S, cd, p_mul(C, sd)), S3);
    *co = p_add3(p_fma(C, cd, p_neg(p_mul(S, sd))), C3);
}

// sin and cos of th + d from s = sin th, c = cos th for the small angle of an RK4 stage,
// |d| <= 2^-9: sin d = d - d^3/6 and cos d - 1 = -d^2/2 + d^4/24, each beyond d itself below
// 2^-18 of the result, so in float; a third of p_sincos's instructions.  One table look-up a
// step instead of four: the 256 x 256 Manko-Novikov FP64 frame 39.8 -> 38.6 ms, the 64 x 64
// Schwarzschild one 4.26 -> 4.14 ms; frames of the zone as before (77.9 ms).
GT_HD void p_rotate(DF s, DF c, DF d, DF *so, DF *co)
{
    const float t = GT_P_MUL(d.hi, d.hi);
    const float s3 = GT_P_MUL(GT_P_MUL(t, d.hi), -1.0f / 6.0f);
    // -(d.hi + d.lo)^2 / 2 with the product's error: t is 2^-18, its rounding 2^-43
    const float te = fmaf(GT_P_ADD(d.hi, d.hi), d.lo, fmaf(d.hi, d.hi, -t));
    const DF sd(d.hi, GT_P_ADD(d.lo, s3));
    const DF cd(GT_P_MUL(-0.5f, t), fmaf(GT_P_MUL(t, t), 1.0f / 24.0f, GT_P_MUL(-0.5f, te)));
    *so = p_add(p_fma(s, cd, p_mul(c, sd)), s);
    *co = p_add(p_fma(c, cd, p_neg(p_mul(s, sd))), c);
}

// ------------------------------------------------------------------ coordinates
// the leading pair, and the sum with a pair as a pair
GT_HD DF tf_pair(TF t) { return DF(t.a, t.b); }

GT_HD TF tf_add(TF x, DF d)
{
    const DF s0 = df_two_sum(x.a, d.hi);
    const DF s1 = df_two_sum(x.b, d.lo);
    const DF s2 = df_two_sum(s0.lo, s1.hi);
    const float c = GT_P_ADD(x.c, GT_P_ADD(s1.lo, s2.lo));
    const DF u = df_fast_two_sum(s0.hi, s2.hi);
    const DF v = df_fast_two_sum(u.lo, c);
    const DF w = df_fast_two_sum(u.hi, v.hi);
    TF o;
    o.a = w.hi;
    const DF z = df_fast_two_sum(w.lo, v.lo);
    o.b = z.hi;
    o.c = z.lo;
    return o;
}

// x - y of two coordinates as a pair: exact but for the last rounding of the low part
GT_HD DF tf_diff(TF x, TF y)
{
    const DF s0 = df_two_sum(x.a, -y.a);
    const DF s1 = df_two_sum(x.b, -y.b);
    const DF s2 = df_two_sum(s0.lo, s1.hi);
    const DF u = df_fast_two_sum(s0.hi, s2.hi);
    return df_fast_two_sum(u.hi, GT_P_ADD(u.lo, GT_P_ADD(s2.lo, GT_P_ADD(s1.lo, GT_P_ADD(x.c, -y.c)))));
}

// ------------------------------------------------------------------ fields
// Spacetime constants of the pair step.  The horizon distance r - r_+ is formed from the
// three-float r and r_+, so Kerr's Delta = (r - r_+)(r - r_-) and Manko-Novikov's x - 1 keep
// their relative precision next to the horizon.
struct PairSpacetime {
    int kind;
    float r_hard; // r - r_+ below which GT_MODE_FP64 steps in FP64 (Manko-Novikov)
    TF r_plus;
    DF r_plus2;  // r_+ as a pair
    DF split;    // Kerr r_+ - r_-
    DF a, a2;    // Kerr
    DF two_beta, three_beta2;                        // Manko-Novikov
    TF ik, alpha, c_g, w_inf, k2, inv_k2, two_k;
};

// Kerr rates at r = r_+ + rp (kerr_rates_sc of spacetime.cuh, Delta from its roots).
GT_HD void kerr_rates_pair(const PairSpacetime &c, DF rp, DF s, DF cs, DF pr, DF pth, TF pt,
                           TF pph, Rates<DF> &o)
{
    const DF r = p_add(rp, c.r_plus2);
    const DF ra2 = p_fma(r, r, c.a2);
    const DF ac = p_mul(c.a, cs);
    const DF Sigma = p_fma(ac, ac, p_sq(r));
    const DF Delta = p_mul(rp, p_add(rp, c.split));
    const DF iSigma = p_rcp(Sigma), iDelta = p_rcp(Delta), is = p_rcp(s);
    const DF apt = p_mul3(c.a, pt), aph = p_mul3(c.a, pph);
    const DF W = p_fma3(ra2, pt, aph);
    const DF Vp = p_mul3(is, pph);
    const DF V = p_fma(apt, s, Vp);
    const DF WiD = p_mul(W, iDelta);
    const DF Dpr = p_mul(Delta, pr);
    // K = 2 Sigma H
    DF K = p_fnma(W, WiD, p_sq(V));
    K = p_fma(pth, pth, K);
    K = p_fma(Dpr, pr, K);
    o.dr = p_mul(Dpr, iSigma);
    o.dth = p_mul(pth, iSigma);
    o.dt = p_mul(p_fnma(ra2, WiD, p_mul(c.a, p_mul(V, s))), iSigma);
    o.dph = p_mul(p_fnma(c.a, WiD, p_mul(V, is)), iSigma);
    const DF KiS = p_mul(K, iSigma);
    // -K_r/2 = -(r - M)(pr^2 + WiD^2) + 2 r pt WiD + r KiS
    const DF rM = p_fma(DF(0.5f, 0.0f), c.split, rp);
    const DF g = p_fma(WiD, WiD, p_sq(pr));
    const DF rk = p_mul(r, p_fma3(p_scale(WiD, 2.0f), pt, KiS));
    o.dpr = p_mul(p_fnma(rM, g, rk), iSigma);
    // -K_th/2 = cos (V (pph/sin^2 - a pt) - a^2 sin KiS)
    const DF h = p_mul(V, p_fma(Vp, is, p_neg(apt)));
    o.dpth = p_mul(p_mul(p_fnma(p_mul(c.a2, s), KiS, h), cs), iSigma);
}

// Manko-Novikov rates at r = r_+ + rp by the reverse sweep of mn_rates_sc, the adjoints of
// the products at the end of the forward sweep taken through their logarithms:
//   2H = -pt^2 / f + F pw^2 + G Q,  f = e A / B, F = f / (xs k^2), G = exp(2psi - 2gamma'') c_g / B
// gives, with T1 = pt^2 / f, T2 = F pw^2, T3 = 4 k F pw pt, T4 = G Q and S = T1 + T2 - T3 om0,
//   B_b = -(T1 + T2 + T4)/B, A_b = S/A, C_b = T3/(e A), xs_b = -T2/xs, (2psi)_b = T4 + S,
//   (2gamma'')_b = -T4,
// and Eg = Ea - Eb replaces the third multipole sum (an identity of the truncated sums too).
// EXP(a) evaluates the exponential; ex receives the high parts of the four exponents.
template <class EXP>
GT_HD void mn_rates_pair(const PairSpacetime &c, DF rp, DF s, DF cs, DF pr, DF pth, TF pt, TF pph,
                         const EXP &EXPF, Rates<DF> &o, float ex[4])
{
    const DF tb = c.two_beta;
    const DF xm1 = p_mul3(rp, c.ik);
    const DF x = p_addf(xm1, 1.0f), xp1 = p_addf(xm1, 2.0f);
    const DF y = cs, s2 = p_sq(s);
    const DF x2m1 = p_mul(xm1, xp1);
    const DF iR = p_rsqrt(p_fma(y, y, x2m1));
    // Multipole tails.  With w = 1/R^2, v = x y w and p = P2(x y/R) w the closed forms of
    // mn_rates_sc (t = 1/R, u = x y/R) have no Legendre polynomial left in them:
    //   Ea = (En - On) / (1 + sa (1 + p + v)), Eb = -(En + On) / (1 + sb (1 + p - v)),
    //   On = v (2 hq + 3 p (v^2 - w)),  hq = 2.5 v^2 - 1.5 w  (v hq = P3 t^3),
    //   En = w (v^2 + p^2) - p hq,
    // sa = (x - y) t, sb = (x + y) t.
    const DF w = p_sq(iR);
    const DF xy = p_mul(x, y);
    const DF v = p_mul(xy, w);
    const DF v2 = p_sq(v);
    const DF p = p_sub(p_mulf(v2, 1.5f), p_scale(w, 0.5f));
    const DF hq = p_sub(p_mulf(v2, 2.5f), p_mulf(w, 1.5f));
    const DF vw = p_sub(v2, w);
    const DF xmy = p_sub(x, y), xpy = p_add(x, y);
    const DF sa = p_mul(xmy, iR), sb = p_mul(xpy, iR);
    const DF Qe = p_addf(p, 1.0f);
    const DF Qa = p_add(Qe, v), Qb = p_sub(Qe, v);
    const DF ia = p_rcp(p_addf(p_mul(sa, Qa), 1.0f)), ib = p_rcp(p_addf(p_mul(sb, Qb), 1.0f));
    const DF p3 = p_mulf(p, 3.0f), p2 = p_sq(p);
    const DF Oq = p_fma(p3, vw, p_scale(hq, 2.0f));
    const DF On = p_mul(v, Oq);
    const DF vp = p_add(v2, p2);
    const DF En = p_fnma(p, hq, p_mul(w, vp));
    const DF Ea = p_mul(p_sub(En, On), ia), Eb = p_neg(p_mul(p_add(En, On), ib));
    const DF xa = p_neg(p_mul(Ea, tb)), xb = p_mul(Eb, tb);
    const DF fa = p_neg(p_mul3(EXPF(xa), c.alpha));
    const DF fb = p_mul3(EXPF(xb), c.alpha);
    const DF ab = p_mul(fa, fb);
    const DF opab = p_addf(ab, 1.0f);
    const DF bma = p_sub(fb, fa);
    const DF op2 = p_sq(opab), bm2 = p_sq(bma);
    const DF A = p_renorm(p_fnma(s2, bm2, p_mul(x2m1, op2))); // zero on the ergosurface
    const DF yp1 = p_addf(y, 1.0f), omy = p_neg(p_addf(y, -1.0f));
    const DF Bq1 = p_fma(xm1, ab, xp1);
    const DF Bq2 = p_fma(omy, fb, p_mul(yp1, fa));
    const DF B = p_fma(Bq1, Bq1, p_sq(Bq2));
    const DF fsum = p_add(fa, fb), omab = p_neg(p_addf(ab, -1.0f));
    const DF C1 = p_fnma(y, fsum, bma);
    const DF C2 = p_fma(x, omab, opab);
    const DF c1 = p_mul(x2m1, opab), c2 = p_mul(s2, bma);
    const DF C = p_fma(c1, C1, p_mul(c2, C2));
    const DF tp = p_mul(tb, p);
    const DF psi2 = p_mul(tp, iR);
    const DF h = p_mul(v, hq);
    const DF p2w = p_mul(p2, w);
    const DF g2 = p_fma(p_sub(Ea, Eb), tb, p_mul(c.three_beta2, p_fma(h, h, p_neg(p2w))));
    const DF xg = p_sub(psi2, g2);
    ex[0] = xa.hi;
    ex[1] = xb.hi;
    ex[2] = psi2.hi;
    ex[3] = xg.hi;
    const DF e = EXPF(psi2);
    const DF eA = p_mul(e, A);
    const DF ieA = p_rcp(eA), iB = p_rcp(B), ixs = p_rcp(p_mul(x2m1, s2));
    const DF invf = p_mul(B, ieA);
    const DF F = p_mul3(p_mul(p_mul(eA, iB), ixs), c.inv_k2);
    const DF om0 = p_mul(C, ieA);
    const DF om = p_sub3(p_mul3(om0, c.two_k), c.w_inf);
    const DF G = p_mul3(p_mul(EXPF(xg), iB), c.c_g);
    const DF Delta = p_mul3(x2m1, c.k2);
    const DF pw = p_add3(p_mul3(om, pt), pph);
    const DF Fpw = p_mul(F, pw);
    const DF Dpr = p_mul(Delta, pr);
    const DF Q = p_fma(Dpr, pr, p_sq(pth));
    const DF ptf = p_mul3(invf, pt);
    o.dt = p_sub(p_mul(Fpw, om), ptf);
    o.dph = Fpw;
    o.dr = p_mul(G, Dpr);
    o.dth = p_mul(G, pth);

    // ---- backward sweep
    const DF T1 = p_mul3(ptf, pt), T2 = p_mul(Fpw, pw), T4 = p_mul(G, Q);
    const DF T3 = p_mul3(p_scale(p_mul3(Fpw, pt), 2.0f), c.two_k);
    const DF T12 = p_add(T1, T2);
    const DF S = p_fnma(T3, om0, T12);
    const DF A_b = p_mul(S, p_mul(ieA, e));
    const DF B_b = p_neg(p_mul(p_add(T12, T4), iB));
    const DF C_b = p_mul(T3, ieA);
    const DF psi2_b = p_add(T4, S);
    const DF xsb = p_neg(p_mul(T2, ixs)); // adjoint of xs = x2m1 s2
    DF x2m1_b = p_fma3(p_mul(p_mul(G, pr), pr), c.k2, p_mul(xsb, s2));
    DF s2_b = p_mul(xsb, x2m1);
    // C = c1 C1 + c2 C2
    const DF C1_b = p_mul(C_b, c1), C2_b = p_mul(C_b, c2);
    const DF c1_b = p_mul(C_b, C1), c2_b = p_mul(C_b, C2);
    x2m1_b = p_fma(c1_b, opab, x2m1_b);
    DF opab_b = p_fma(c1_b, x2m1, C2_b);
    s2_b = p_fma(c2_b, bma, s2_b);
    DF bma_b = p_fma(c2_b, s2, C1_b);
    DF x_b = p_mul(C2_b, omab);
    DF ab_b = p_neg(p_mul(C2_b, x));
    DF y_b = p_neg(p_mul(C1_b, fsum));
    DF fa_b = p_neg(p_mul(C1_b, y));
    DF fb_b = fa_b;
    // B = Bq1^2 + Bq2^2
    const DF B2 = p_scale(B_b, 2.0f);
    const DF Bq1_b = p_mul(Bq1, B2), Bq2_b = p_mul(Bq2, B2);
    y_b = p_fnma(Bq2_b, bma, y_b);
    fa_b = p_fma(Bq2_b, yp1, fa_b);
    fb_b = p_fma(Bq2_b, omy, fb_b);
    DF xm1_b = p_fma(Bq1_b, ab, Bq1_b); // through xm1, and xp1 = xm1 + 2
    ab_b = p_fma(Bq1_b, xm1, ab_b);
    // A = x2m1 opab^2 - s2 bma^2
    x2m1_b = p_fma(A_b, op2, x2m1_b);
    s2_b = p_fnma(A_b, bm2, s2_b);
    const DF A2 = p_scale(A_b, 2.0f);
    opab_b = p_fma(A2, c1, opab_b);
    bma_b = p_fnma(A2, c2, bma_b);
    // bma = fb - fa, opab = ab + 1, ab = fa fb; fa = -alpha exp(-tb Ea), fb = alpha exp(tb Eb)
    ab_b = p_mul(p_add(ab_b, opab_b), ab);
    const DF la_b = p_fma(p_sub(fa_b, bma_b), fa, ab_b);
    const DF lb_b = p_fma(p_add(fb_b, bma_b), fb, ab_b);
    // 2 gamma'' = tb (Ea - Eb) + 3 beta^2 (h^2 - p^2 w), its adjoint -T4
    const DF Ga = p_mul(p_mul(p_neg(p_add(la_b, T4)), tb), ia);
    const DF Gb = p_mul(p_mul(p_add(lb_b, T4), tb), ib);
    // Ea = (En - On) ia, Eb = -(En + On) ib
    const DF En_b = p_sub(Ga, Gb), On_m = p_add(Ga, Gb); // On_m = -On_b
    const DF da_m = p_mul(Ea, Ga), db_m = p_mul(Eb, Gb); // minus the adjoints of 1/ia, 1/ib
    const DF sa_m = p_mul(da_m, Qa), sb_m = p_mul(db_m, Qb);
    const DF Qa_m = p_mul(da_m, sa), Qb_m = p_mul(db_m, sb);
    x_b = p_fnma(iR, p_add(sa_m, sb_m), x_b);
    y_b = p_fma(iR, p_sub(sa_m, sb_m), y_b);
    // psi2 = tb p iR
    DF iR_b = p_fma(tp, psi2_b, p_neg(p_fma(xmy, sa_m, p_mul(xpy, sb_m))));
    DF p_b = p_fma(p_mul(tb, psi2_b), iR, p_neg(p_add(Qa_m, Qb_m)));
    DF v_b = p_sub(Qb_m, Qa_m);
    // On = v (2 hq + 3 p (v^2 - w))
    v_b = p_fnma(On_m, Oq, v_b);
    const DF qm = p_mul(On_m, v);
    p_b = p_fnma(p_mulf(qm, 3.0f), vw, p_b);
    const DF vw_m = p_mul(qm, p3);
    // 3 beta^2 (h^2 - p^2 w), h = v hq
    const DF km = p_mul(T4, c.three_beta2);
    const DF hm = p_scale(p_mul(h, km), 2.0f);
    v_b = p_fnma(hm, hq, v_b);
    p_b = p_fma(p_scale(p_mul(p, w), 2.0f), km, p_b);
    // En = w (v^2 + p^2) - p hq
    p_b = p_fnma(En_b, hq, p_b);
    const DF z = p_mul(En_b, w);
    p_b = p_fma(p_scale(p, 2.0f), z, p_b);
    const DF hq_m = p_fma(hm, v, p_fma(En_b, p, p_scale(qm, 2.0f))); // -hq_b
    // p = 1.5 v^2 - w/2, hq = 2.5 v^2 - 1.5 w, v = x y w, w = iR^2
    DF v2_b = p_sub(p_add(p_mulf(p_b, 1.5f), z), p_add(p_mulf(hq_m, 2.5f), vw_m));
    DF w_b = p_fma(En_b, vp, p_fma(p2, km, vw_m));
    w_b = p_add(w_b, p_sub(p_mulf(hq_m, 1.5f), p_scale(p_b, 0.5f)));
    v_b = p_fma(p_scale(v, 2.0f), v2_b, v_b);
    w_b = p_fma(v_b, xy, w_b);
    const DF xy_b = p_mul(v_b, w);
    iR_b = p_fma(p_scale(iR, 2.0f), w_b, iR_b);
    x_b = p_fma(xy_b, y, x_b);
    y_b = p_fma(xy_b, x, y_b);
    // iR = R2^(-1/2), R2 = x2m1 + y^2
    const DF R2h = p_mul(iR_b, p_mul(iR, w)); // -2 R2_b
    x2m1_b = p_fma(DF(-0.5f, 0.0f), R2h, x2m1_b);
    y_b = p_fnma(y, R2h, y_b);
    // x2m1 = xm1 xp1: d x2m1 = 2 x dx; x, xm1, xp1 move together
    const DF dx = p_add(p_fma(p_scale(x, 2.0f), x2m1_b, xm1_b), x_b);
    o.dpr = p_mul3(p_scale(dx, -0.5f), c.ik);
    o.dpth = p_mul(s, p_fma(DF(0.5f, 0.0f), y_b, p_neg(p_mul(cs, s2_b))));
}

// ------------------------------------------------------------------ the step
// Ray state of the double-float kernels: three floats per coordinate.
struct RayTF {
    TF t, r, th, ph, pr, pth, pt, pph;
};

// Largest |exponent| of a Manko-Novikov evaluation taken in double-float: |2 beta Ea|,
// |2 beta Eb| <= 24 and |2 psi|, |2 psi - 2 gamma''| <= 48.  Beyond, products of the metric
// functions overflow the float range (an infinite high part turns the low part into NaN, so
// the rates come out non-finite) or, silently, low parts fall below the normal floats.
constexpr float PAIR_MAX_EF = 24.0f;
constexpr float PAIR_MAX_EPSI = 48.0f;

// Where a trace of double-float steps ends at least as close to the exact flow as one of FP64
// steps.  A pair rate is off by 2^-47 (FP64's by 2^-52), an FP64 coordinate by half an ulp a
// step.  So the pairs need increments that are small against the scale on which the rates
// change, and steps enough to average: t and phi start at zero, and after ten steps of any size
// they are off by 6e-15 where FP64's are off by 1e-16.  Root-mean-square error over camera
// frames of both kinds, spins 0 to 0.999, pair / FP64, worst of t, r, theta, phi:
//   steps of 3e-4 M, r0 15-50 M:  500 steps 1.40, 700 1.15, 900 0.99, 1000 0.87, 2000 0.62;
//   1000 steps, r0 8.5-60 M: of 1e-3 M 0.81, of 1e-4 M 1.17 (1500 of them: 0.79);
//   2000 steps of 1e-4 M, r0 30-60 M: 0.55, 60-100 M: 1.17 (5000, 80-100 M: 0.50);
//   2000 steps of 3e-4 M, r0 60-100 M: 0.77;  8000 of 2.5e-4 M, 200-400 M: 0.38;
//   whole paths, r0 8.5-30 M: steps of 2e-3 M 0.43, of 5e-3 M 1.34, of 0.2 M up to 25.
inline bool pair_accurate(double M, double r0, double sp, int64_t n_steps)
{
    const double n = (double)n_steps, path = sp * n;
    return n_steps >= 1000 && sp <= 2e-3 * M && path >= 0.15 * M && path >= 0.005 * r0 &&
           r0 <= 0.05 * M * n && r0 <= 1000.0 * M;
}

// The same at the axis, where theta and phi change on the scale rho = r sin theta: steps from
// rho below 1000 times their length are FP64's.  Frames with theta0 of 1e-3 to 0.3, worst ratio
// as above: 0.5 to 1.2 (no such line: 1.5 to 108; at 300 times: 0.5 to 2.9).
constexpr float PAIR_RHO_STEPS = 1000.0f;

struct PairExp {
    const PairTables *tab;
    GT_HD DF operator()(DF a) const { return p_exp(a, tab); }
};

// One RK4 step of x in double-float: the stages of rk4_step64 (stage points x + h/2 k1,
// x + h/2 k2, x + h k3; weights 1, 2, 2, 1 times h w6; h = |sp / k1.dt|) in a rolled loop, so
// one copy of the field is compiled.  Returns false, x untouched, where an evaluation leaves
// the double-float range (exponents, the axis, |theta| beyond the table reduction, a rate or a
// new coordinate that is not finite): the caller repeats the step in FP64.
// A step that starts closer to the axis than rho_min is refused too.
template <int KIND>
GT_HD bool pair_step(const PairSpacetime &c, const PairTables *tab, RayTF &x, TF sp, TF w6,
                     float rho_min, DF &h_out)
{
    const DF rp0 = tf_diff(x.r, c.r_plus);
    DF rp = rp0, pr = tf_pair(x.pr), pth = tf_pair(x.pth), s1, c1;
    p_sincos(tf_pair(x.th), x.th.c, tab, &s1, &c1);
    DF s = s1, cs = c1;
    Rates<DF> k, acc;
    DF h(0.0f, 0.0f);
    bool ok = fabsf(x.th.a) <= 128.0f && fabsf(s1.hi) >= 1e-6f && x.r.a * fabsf(s1.hi) >= rho_min;
#pragma unroll 1
    for (int stage = 0; stage < 4; stage++) {
        if (KIND == KIND_MN || (KIND != KIND_KERR && c.kind == KIND_MN)) {
            float ex[4];
            mn_rates_pair(c, rp, s, cs, pr, pth, x.pt, x.pph, PairExp{tab}, k, ex);
            ok = ok && fmaxf(fabsf(ex[0]), fabsf(ex[1])) <= PAIR_MAX_EF &&
                 fmaxf(fabsf(ex[2]), fabsf(ex[3])) <= PAIR_MAX_EPSI;
        } else {
            kerr_rates_pair(c, rp, s, cs, pr, pth, x.pt, x.pph, k);
        }
        if (stage == 0) {
            h = p_norm(p_mul3(p_rcp(k.dt), sp));
            if (h.hi < 0.0f) h = p_neg(h);
            acc = k;
        } else {
            const float w = stage < 3 ? 2.0f : 1.0f;
            acc.dt = p_add(acc.dt, p_scale(k.dt, w));
            acc.dr = p_add(acc.dr, p_scale(k.dr, w));
            acc.dth = p_add(acc.dth, p_scale(k.dth, w));
            acc.dph = p_add(acc.dph, p_scale(k.dph, w));
            acc.dpr = p_add(acc.dpr, p_scale(k.dpr, w));
            acc.dpth = p_add(acc.dpth, p_scale(k.dpth, w));
        }
        if (stage < 3) {
            const DF d = p_scale(h, stage < 2 ? 0.5f : 1.0f);
            rp = p_norm(p_fma(d, k.dr, rp0));
            pr = p_fma(d, k.dpr, tf_pair(x.pr));
            pth = p_fma(d, k.dpth, tf_pair(x.pth));
            const DF dth = p_norm(p_mul(d, k.dth));
            if (fabsf(dth.hi) <= 0.001953125f) {
                p_rotate(s1, c1, dth, &s, &cs);
            } else { // a step of a radian's order
                const DF th = p_norm(p_add(tf_pair(x.th), dth));
                ok = ok && fabsf(th.hi) <= 128.0f;
                p_sincos(th, x.th.c, tab, &s, &cs);
            }
            ok = ok && fabsf(s.hi) >= 1e-6f;
        }
    }
    const DF hw = p_norm(p_mul3(h, w6));
    const DF dt = p_norm(p_mul(hw, acc.dt)), dr = p_norm(p_mul(hw, acc.dr));
    const DF dth = p_norm(p_mul(hw, acc.dth)), dph = p_norm(p_mul(hw, acc.dph));
    const DF dpr = p_norm(p_mul(hw, acc.dpr)), dpth = p_norm(p_mul(hw, acc.dpth));
    // one test of the new state: an increment is finite only if h and every stage's rate were,
    // and a bound on the sum of all magnitudes holds for each new coordinate
    const float m = ((fabsf(x.t.a) + fabsf(dt.hi)) + (fabsf(x.r.a) + fabsf(dr.hi))) +
                    ((fabsf(x.th.a) + fabsf(dth.hi)) + (fabsf(x.ph.a) + fabsf(dph.hi))) +
                    ((fabsf(x.pr.a) + fabsf(dpr.hi)) + (fabsf(x.pth.a) + fabsf(dpth.hi)));
    if (!ok || !(m <= 1e38f)) return false;
    x.t = tf_add(x.t, dt);
    x.r = tf_add(x.r, dr);
    x.th = tf_add(x.th, dth);
    x.ph = tf_add(x.ph, dph);
    x.pr = tf_add(x.pr, dpr);
    x.pth = tf_add(x.pth, dpth);
    h_out = h;
    return true;
}

GT_HD bool tf_greater(TF x, TF y)
{
    return x.a > y.a || (x.a == y.a && (x.b > y.b || (x.b == y.b && x.c > y.c)));
}

#undef GT_P_ADD
#undef GT_P_MUL

} // namespace gt
