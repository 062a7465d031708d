// features.cuh -- the surrogate network's input columns (device, inline).
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "internal.cuh"
#include "surrogate.cuh"

namespace gt {
namespace sg {

// Tables of the sin/cos below (pair.cuh).
static __device__ const PairTables g_trig = make_pair_tables();

// sin and cos of an FP64 angle, and the unit vector of two, as the floats nearest the FP64
// results (to 2^-46, so but for about one in 2^21 they are the same).  FP64 instructions take 64
// cycles of a lone warp each, ~60 of them for a sincos: the pairs take the angle apart with
// five of them and do the rest in FP32.  Angles beyond the table reduction go to FP64.
static __device__ __noinline__ void sincos64(double th, DF *s, DF *c)
{
    double s64, c64;
    sincos(th, &s64, &c64);
    *s = DF(s64);
    *c = DF(c64);
}

__device__ __forceinline__ void sincos_pair(double th, DF *s, DF *c)
{
    const TF t = tf_from(th);
    if (fabsf(t.a) <= 128.0f)
        p_sincos(tf_pair(t), t.c, &g_trig, s, c);
    else
        sincos64(th, s, c);
}

__device__ __forceinline__ void unit_vector(double th, double ph, float d[3])
{
    DF st, ct, sp, cp;
    sincos_pair(th, &st, &ct);
    sincos_pair(ph, &sp, &cp);
    d[0] = p_norm(p_mul(st, cp)).hi;
    d[1] = p_norm(p_mul(st, sp)).hi;
    d[2] = p_norm(ct).hi;
}

// rho = |(a, b)| and (a, b) / max(rho, 1e-3) in FP64
static __device__ __noinline__ void polar64(double a, double b, float f[3])
{
    const double rho = sqrt(a * a + b * b);
    const double irho = 1.0 / fmax(rho, 1e-3);
    f[0] = (float)rho;
    f[1] = (float)(a * irho);
    f[2] = (float)(b * irho);
}

// The network's 16 input columns from the 5 inputs (alpha, beta, a/M, q, theta0):
// 0-4 the inputs scaled to about [-1, 1]; 5-7 the pixel direction in polar form
// (rho, cos psi, sin psi) of the scaled (alpha, beta); 8-9 cos and sin of theta0; the
// rest zero.  The derived columns are fixed functions of the inputs, formed in pairs as above
// (in FP64 where rho leaves [1e-3, 1e6]): a 128-row tile has them after 3,200 cycles, 7,000 in
// FP64 (8 training steps of 8,192 rows, labels likewise: 912 -> 880 us).
__device__ __forceinline__ void make_features(double al, double bt, double spin, double q,
                                              double th0, const Norm &nm, float f[16])
{
    const double a = al * nm.inv_h, b = bt * nm.inv_v;
    f[2] = (float)(spin * nm.spin_scale + nm.spin_shift);
    f[3] = (float)(q * nm.q_scale);
    f[4] = (float)(th0 * nm.th_scale + nm.th_shift);
    const DF A(a), B(b);
    f[0] = A.hi;
    f[1] = B.hi;
    const DF r2 = p_fma(A, A, p_sq(B));
    if (r2.hi > 1.001e-6f && r2.hi < 1e12f) {
        const DF ir = p_rsqrt(r2);
        f[5] = p_norm(p_mul(r2, ir)).hi;
        f[6] = p_norm(p_mul(A, ir)).hi;
        f[7] = p_norm(p_mul(B, ir)).hi;
    } else {
        polar64(a, b, f + 5);
    }
    DF s, c;
    sincos_pair(th0, &s, &c);
    f[8] = p_norm(c).hi;
    f[9] = p_norm(s).hi;
#pragma unroll
    for (int j = 10; j < 16; j++) f[j] = 0.0f;
}

// bf16 pair of v: hi = bf16(v), lo = bf16(v - hi)
__device__ __forceinline__ void split_pair(float v, __nv_bfloat16 *hi, __nv_bfloat16 *lo)
{
    *hi = __float2bfloat16(v);
    *lo = __float2bfloat16(v - __bfloat162float(*hi));
}

// The inputs of a camera pixel (flat j * res_x + i).
__device__ __forceinline__ void pixel_features(const CamDesc &c, int64_t pix, const Norm &nm,
                                               float f[16])
{
    const int i = (int)(pix % c.res_x), j = (int)(pix / c.res_x);
    const double al = c.res_x > 1 ? c.H * (double)(2 * i - (c.res_x - 1)) / (double)(c.res_x - 1) : 0.0;
    const double bt = c.res_y > 1 ? c.V * (double)(2 * j - (c.res_y - 1)) / (double)(c.res_y - 1) : 0.0;
    make_features(al, bt, (c.S / c.M) / c.M, c.Q, c.th0, nm, f);
}

} // namespace sg
} // namespace gt
