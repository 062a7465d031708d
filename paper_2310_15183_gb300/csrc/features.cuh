// features.cuh -- the surrogate network's input columns (device, inline).
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "internal.cuh"
#include "surrogate.cuh"

namespace gt {
namespace sg {

// The network's 16 input columns from the 5 inputs (alpha, beta, a/M, q, theta0):
// 0-4 the inputs scaled to about [-1, 1]; 5-7 the pixel direction in polar form
// (rho, cos psi, sin psi) of the scaled (alpha, beta); 8-9 cos and sin of theta0; the
// rest zero.  The derived columns are fixed functions of the inputs.
__device__ __forceinline__ void make_features(double al, double bt, double spin, double q,
                                              double th0, const Norm &nm, float f[16])
{
    const double a = al * nm.inv_h, b = bt * nm.inv_v;
    const double rho = sqrt(a * a + b * b);
    const double irho = 1.0 / fmax(rho, 1e-3);
    f[0] = (float)a;
    f[1] = (float)b;
    f[2] = (float)(spin * nm.spin_scale + nm.spin_shift);
    f[3] = (float)(q * nm.q_scale);
    f[4] = (float)(th0 * nm.th_scale + nm.th_shift);
    f[5] = (float)rho;
    f[6] = (float)(a * irho);
    f[7] = (float)(b * irho);
    f[8] = (float)cos(th0);
    f[9] = (float)sin(th0);
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
