// surrogate.cu -- the MLP surrogate of the ray tracer: per-pixel (alpha, beta, spin,
// q, theta0) -> (escape logit, end direction), trained on rays the integrator itself
// produces, evaluated and trained by the fused tcgen05 kernels of mlp_fused.cu, and backed
// by the integrator for low-confidence and photon-ring pixels.
//
// Network: 16 (5 inputs and 5 columns derived from them, zero padded) -> 256 -> 256 ->
// 256 -> 256 -> 16 (4 used: logit and the unit vector of the end direction, which unlike
// (theta, phi) has no jump at phi = +-pi), SiLU between layers.  FP32 master weights and
// AdamW state.  The forward products are split-precision BF16: each layer input x and
// weight w is carried as a bf16 pair (hi, lo), hi = bf16(v), lo = bf16(v - hi), and the
// product is x_hi w_hi + x_lo w_hi + x_hi w_lo in one accumulator, which carries
// the layer to about 2^-16 relative instead of bf16's 2^-8 (the dropped x_lo w_lo term is
// 2^-16 of the product); the end direction is read from the last layer, and a single
// 16-bit product leaves a rounding floor of 5e-4 (FP16) to 2e-3 rad (BF16) under it.  The
// backward products take plain BF16, whose range holds gradients scaled by 1/batch.
// Accumulation is FP32 throughout.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <new>
#include <vector>

#include "../../include/geotrace.h"
#include "internal.cuh"
#include "mlp_fused.cuh"
#include "camera.cuh"
#include "features.cuh"
#include "surrogate.cuh"

namespace gt {
namespace sg {

// ------------------------------------------------------------------ kernels
// counter-based normal deviates: splitmix64 -> two uniforms -> Box-Muller
__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

__global__ void init_params_kernel(float *p, int64_t n, const int64_t *offs, const float *scales,
                                   int n_seg, uint64_t seed)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int s = 0;
    while (s + 1 < n_seg && offs[s + 1] <= i) ++s;
    const float sc = scales[s];
    if (sc == 0.0f) {
        p[i] = 0.0f;
        return;
    }
    const uint64_t a = splitmix64(seed ^ (uint64_t)(2 * i));
    const uint64_t b = splitmix64(seed ^ (uint64_t)(2 * i + 1));
    const double u1 = ((a >> 11) + 1) * (1.0 / 9007199254740993.0);
    const double u2 = (b >> 11) * (1.0 / 9007199254740992.0);
    p[i] = sc * (float)(sqrt(-2.0 * log(u1)) * cos(2.0 * M_PI * u2));
}

// Offsets of the layers in the flat parameter vector and in the split weights.
struct Offsets {
    int64_t w[N_LAYERS], b[N_LAYERS], w3[N_LAYERS];
};

// One parameter a thread: with UPDATE an AdamW step, then -- for a weight -- its copies for the
// tensor-core products: the split row [w_hi | w_hi | w_lo] of w3 ([out][3 in]) and the transposed
// bf16 weight of wt ([in][out]).
template <bool UPDATE>
__global__ void update_kernel(int64_t n, const __grid_constant__ Offsets off, float *p, const float *g, float *m, float *v,
                              float lr, float b1, float b2, float eps, float wd, float bc1,
                              float bc2, __nv_bfloat16 *w3, __nv_bfloat16 *wt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int l = 0;
#pragma unroll
    for (int k = 1; k < N_LAYERS; k++) l += i >= off.w[k] ? 1 : 0;
    const bool weight = i < off.b[l];
    float pi = p[i];
    if (UPDATE) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        if (weight) pi -= lr * wd * pi; // decoupled decay, weights only
        pi -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
        p[i] = pi;
    }
    if (!weight) return;
    const int in_dim = l == 0 ? 16 : 256, out_dim = l == N_LAYERS - 1 ? 16 : 256;
    const int k = (int)(i - off.w[l]), o = k / in_dim, c = k % in_dim;
    __nv_bfloat16 hi, lo;
    split_pair(pi, &hi, &lo);
    __nv_bfloat16 *row = w3 + off.w3[l] + (int64_t)o * 3 * in_dim;
    row[c] = hi;
    row[in_dim + c] = hi;
    row[2 * in_dim + c] = lo;
    wt[off.w[l] + (int64_t)c * out_dim + o] = hi;
}

// Constants of motion of a camera ray in the Kerr picture: E = -p_t, L = p_phi and the
// Carter constant K = p_theta^2 + cos^2 theta0 (-a^2 E^2 + L^2/sin^2 theta0), with a = S/M
// (Manko-Novikov rays take the Kerr values of their M and S: an estimate there).
__device__ __forceinline__ void kerr_constants(const CamDesc &c, const Ray64 &p, double *a,
                                               double *E, double *L, double *K)
{
    *a = c.S / c.M;
    *E = -p.pt;
    *L = p.pph;
    const double ct = cos(c.th0), st = sin(c.th0);
    *K = p.pth * p.pth + ct * ct * (-(*a) * (*a) * (*E) * (*E) + (*L) * (*L) / (st * st));
}

// Photon-ring test for a Kerr pixel: the radial potential of its constants of motion,
//   R(r) = (E (r^2 + a^2) - a L)^2 - Delta ((L - a E)^2 + K),
// has a (near) double root for rays near the critical curve.  Returns
// min over r in (r_+, r0] of R(r) / (E^2 r^4) on a geometric grid.
__device__ double kerr_rmin(const CamDesc &c, const Ray64 &p)
{
    double a, E, L, K;
    kerr_constants(c, p, &a, &E, &L, &K);
    const double M = c.M;
    const double rp = c.st.kind == KIND_KERR ? c.st.r_plus : M + sqrt(fmax(M * M - a * a, 0.0));
    const double lo = log(rp * 1.0001), hi = log(c.r0);
    double best = 1e300;
    for (int k = 0; k <= 96; k++) {
        const double r = exp(lo + (hi - lo) * k / 96.0);
        const double W = E * (r * r + a * a) - a * L;
        const double D = r * r - 2.0 * M * r + a * a;
        const double R = W * W - D * ((L - a * E) * (L - a * E) + K);
        const double v = R / (E * E * r * r * r * r);
        best = v < best ? v : best;
    }
    return best;
}

// Smallest sin^2 theta a Kerr ray can reach: the theta potential
// Theta = K + a^2 E^2 cos^2 - L^2 cot^2 vanishes at u = cos^2 theta solving
// -a^2 E^2 u^2 + (a^2 E^2 - K - L^2) u + K = 0; returns 1 - u for its root in [0, 1].
// Rays that pass close to the axis sweep phi fast and end in directions that change
// abruptly from pixel to pixel.
__device__ double kerr_min_sin2(const CamDesc &c, const Ray64 &p)
{
    double a, E, L, K;
    kerr_constants(c, p, &a, &E, &L, &K);
    const double A = -a * a * E * E, B = a * a * E * E - K - L * L, C = K;
    double u;
    if (fabs(A) < 1e-300) {
        u = (K + L * L) > 0.0 ? K / (K + L * L) : 0.0;
    } else {
        const double disc = sqrt(fmax(B * B - 4.0 * A * C, 0.0));
        const double u1 = (-B + disc) / (2.0 * A), u2 = (-B - disc) / (2.0 * A);
        u = 0.0;
        if (u1 >= 0.0 && u1 <= 1.0) u = fmax(u, u1);
        if (u2 >= 0.0 && u2 <= 1.0) u = fmax(u, u2);
    }
    return 1.0 - u;
}

// Probe pixel columns: k stride for k < n - 1, and the last column (res - 1).
__device__ __forceinline__ int probe_coord(int k, int stride, int n, int res)
{
    return k < n - 1 ? k * stride : res - 1;
}

__device__ __forceinline__ bool is_probe(int i, int j, const ProbeGrid &pg, int res_x, int res_y)
{
    return (i % pg.stride == 0 || i == res_x - 1) && (j % pg.stride == 0 || j == res_y - 1);
}

// Gates that send a pixel to the integrator whatever the probes say: an unsure logit, the
// Kerr photon-ring band, the axis, an unsettled direction length.
__device__ __forceinline__ bool pixel_gates(const CamDesc &cam, int64_t pix, float4 z, float tau,
                                            double band, double axis, float dir_tol)
{
    if (fabsf(z.x) < tau) return true;
    if ((band > 0.0 && cam.st.kind == KIND_KERR) || axis > 0.0) {
        Ray64 p;
        camera_init(cam, pix, p);
        if (band > 0.0 && cam.st.kind == KIND_KERR && fabs(kerr_rmin(cam, p)) < band) return true;
        if (axis > 0.0 && kerr_min_sin2(cam, p) < axis * axis) return true;
    }
    if (dir_tol > 0.0f && z.x > 0.0f) {
        const float nn = sqrtf(z.y * z.y + z.z * z.z + z.w * z.w);
        if (!(fabsf(nn - 1.0f) <= dir_tol)) return true;
    }
    return false;
}

// The probe cell holding pixel (i, j): corner columns x0 < x1 and rows y0 < y1, and the
// index (kx, ky) of its upper-left probe.
struct Cell {
    int kx, ky, x0, x1, y0, y1;
};

__device__ __forceinline__ Cell cell_of(int i, int j, const ProbeGrid &pg, int res_x, int res_y)
{
    Cell c;
    c.kx = min(i / pg.stride, pg.nx - 2);
    c.ky = min(j / pg.stride, pg.ny - 2);
    c.x0 = probe_coord(c.kx, pg.stride, pg.nx, res_x);
    c.x1 = probe_coord(c.kx + 1, pg.stride, pg.nx, res_x);
    c.y0 = probe_coord(c.ky, pg.stride, pg.ny, res_y);
    c.y1 = probe_coord(c.ky + 1, pg.stride, pg.ny, res_y);
    return c;
}

// First integrator list: the probes, every pixel a gate sends to the integrator, and --
// with probes -- every pixel whose predicted escape differs from the network's prediction
// at one of its cell's corners (such a pixel fails the cell test whatever the integrator
// finds at the corners).  Tracing them in the probes' launch leaves one tail of long rays
// where two passes would leave two.
__device__ __forceinline__ bool first_pass_pixel(const CamDesc &cam, const float4 *net, int64_t pix,
                                                 const ProbeGrid &pg, float tau, double band,
                                                 double axis, float dir_tol)
{
    const int res_x = cam.res_x, res_y = cam.res_y;
    const int i = (int)(pix % res_x), j = (int)(pix / res_x);
    const float4 z = net[pix];
    if (pg.stride > 0) {
        if (is_probe(i, j, pg, res_x, res_y)) return true;
        const Cell c = cell_of(i, j, pg, res_x, res_y);
        const bool esc = z.x > 0.0f;
        const int64_t r0 = (int64_t)c.y0 * res_x, r1 = (int64_t)c.y1 * res_x;
        if ((net[r0 + c.x0].x > 0.0f) != esc || (net[r0 + c.x1].x > 0.0f) != esc ||
            (net[r1 + c.x0].x > 0.0f) != esc || (net[r1 + c.x1].x > 0.0f) != esc)
            return true;
    }
    return pixel_gates(cam, pix, z, tau, band, axis, dir_tol);
}

// warp-aggregated append of the flagged pixels to a list
__device__ __forceinline__ void append_flagged(bool flag, int64_t pix, int64_t *list,
                                               unsigned long long *count)
{
    const unsigned mask = __ballot_sync(0xffffffffu, flag);
    if (mask) {
        const int lane = threadIdx.x & 31;
        const int leader = __ffs(mask) - 1;
        unsigned long long base = 0;
        if (lane == leader) base = atomicAdd(count, (unsigned long long)__popc(mask));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (flag) list[base + __popc(mask & ((1u << lane) - 1u))] = pix;
    }
}

__global__ void select_kernel(int64_t n_pix, const CamDesc *cam, const float4 *net, ProbeGrid pg,
                              float tau, double band, double axis, float dir_tol, int64_t *list,
                              unsigned long long *count)
{
    const int64_t pix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool flag = pix < n_pix && first_pass_pixel(*cam, net, pix, pg, tau, band, axis, dir_tol);
    append_flagged(flag, pix, list, count);
}

// Probe records from the integrator's results (already in the image) and the network's
// answers at the probes.
__global__ void probe_record_kernel(const CamDesc *cam, ProbeGrid pg, const float4 *net,
                                    const uint8_t *status, const double *th, const double *ph,
                                    ProbeRec *rec)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= pg.nx * pg.ny) return;
    const int kx = k % pg.nx, ky = k / pg.nx;
    const int64_t pix = (int64_t)probe_coord(ky, pg.stride, pg.ny, cam->res_y) * cam->res_x +
                        probe_coord(kx, pg.stride, pg.nx, cam->res_x);
    const float4 z = net[pix];
    ProbeRec o;
    o.exact = status[pix];
    o.net_esc = z.x > 0.0f ? 1 : 0;
    o.pad[0] = o.pad[1] = 0;
    if (o.exact == GT_RAY_ESCAPED) {
        const double s = sin(th[pix]);
        o.err[0] = (float)(s * cos(ph[pix])) - z.y;
        o.err[1] = (float)(s * sin(ph[pix])) - z.z;
        o.err[2] = (float)cos(th[pix]) - z.w;
    } else {
        o.err[0] = o.err[1] = o.err[2] = 0.0f;
    }
    rec[k] = o;
}

// Every pixel the first pass did not trace: with probes, taken from the network only
// inside a probe cell whose four corners the integrator and the network classify alike --
// all escaped, or all not escaping with one common end (all HORIZON, or all MAXSTEPS:
// trapped; the pixel takes that status) -- and, for escaped ones, whose corner error
// vectors differ by less than pg.tol; its end direction is the network's plus the bilinear
// interpolation of the corners' error vectors (the integrator correcting the network
// where it measured it).  The rest go to the second integrator list.
__global__ void gate_kernel(int64_t n_pix, const CamDesc *cam, const float4 *net, ProbeGrid pg,
                            float tau, double band, double axis, float dir_tol, double *t,
                            double *r, double *th, double *ph, uint8_t *status, uint32_t *nsteps,
                            int64_t *fallback, unsigned long long *n_fallback)
{
    const int64_t pix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool fb = false;
    if (pix < n_pix && !first_pass_pixel(*cam, net, pix, pg, tau, band, axis, dir_tol)) {
        const int res_x = cam->res_x, res_y = cam->res_y;
        const int i = (int)(pix % res_x), j = (int)(pix / res_x);
        const float4 z = net[pix];
        float nx = z.y, ny = z.z, nz = z.w;
        int cap_status = GT_RAY_HORIZON; // status given to a captured network pixel
        if (pg.stride > 0) {
            const Cell cl = cell_of(i, j, pg, res_x, res_y);
            const int kx = cl.kx, ky = cl.ky, x0 = cl.x0, x1 = cl.x1, y0 = cl.y0, y1 = cl.y1;
            const ProbeRec &c00 = pg.rec[ky * pg.nx + kx], &c01 = pg.rec[ky * pg.nx + kx + 1];
            const ProbeRec &c10 = pg.rec[(ky + 1) * pg.nx + kx];
            const ProbeRec &c11 = pg.rec[(ky + 1) * pg.nx + kx + 1];
            const bool esc4 = c00.exact == GT_RAY_ESCAPED && c01.exact == GT_RAY_ESCAPED &&
                              c10.exact == GT_RAY_ESCAPED && c11.exact == GT_RAY_ESCAPED &&
                              c00.net_esc && c01.net_esc && c10.net_esc && c11.net_esc;
            const bool cap4 = (c00.exact == GT_RAY_HORIZON || c00.exact == GT_RAY_MAXSTEPS) &&
                              c01.exact == c00.exact && c10.exact == c00.exact &&
                              c11.exact == c00.exact && !c00.net_esc && !c01.net_esc &&
                              !c10.net_esc && !c11.net_esc;
            cap_status = c00.exact;
            if (z.x > 0.0f) {
                float sp = 0.0f, sq = 0.0f;
#pragma unroll
                for (int m = 0; m < 3; m++) {
                    const float a = c00.err[m] - c11.err[m], b = c01.err[m] - c10.err[m];
                    sp = fmaf(a, a, sp);
                    sq = fmaf(b, b, sq);
                }
                if (!esc4 || !(fmaxf(sp, sq) < pg.tol * pg.tol)) {
                    fb = true;
                } else {
                    const float tx = (float)(i - x0) / (float)(x1 - x0);
                    const float ty = (float)(j - y0) / (float)(y1 - y0);
                    const float w00 = (1.0f - tx) * (1.0f - ty), w01 = tx * (1.0f - ty);
                    const float w10 = (1.0f - tx) * ty, w11 = tx * ty;
                    nx += w00 * c00.err[0] + w01 * c01.err[0] + w10 * c10.err[0] + w11 * c11.err[0];
                    ny += w00 * c00.err[1] + w01 * c01.err[1] + w10 * c10.err[1] + w11 * c11.err[1];
                    nz += w00 * c00.err[2] + w01 * c01.err[2] + w10 * c10.err[2] + w11 * c11.err[2];
                }
            } else if (!cap4) {
                fb = true;
            }
        }
        if (!fb) {
            if (z.x > 0.0f) {
                const float nc = sqrtf(nx * nx + ny * ny + nz * nz);
                th[pix] = acos(fminf(fmaxf(nz / nc, -1.0f), 1.0f));
                ph[pix] = atan2(ny, nx);
                status[pix] = GT_RAY_ESCAPED;
            } else {
                th[pix] = nan("");
                ph[pix] = nan("");
                status[pix] = (uint8_t)cap_status;
            }
            t[pix] = nan("");
            r[pix] = nan("");
            nsteps[pix] = 0;
        }
    }
    append_flagged(fb, pix, fallback, n_fallback);
}

} // namespace sg
} // namespace gt

// ====================================================================== host side
namespace {

using namespace gt;
using namespace gt::sg;

inline unsigned blocks_for(int64_t n, int b = 256) { return (unsigned)((n + b - 1) / b); }

} // namespace

struct gt_surrogate {
    int device = 0;
    Norm norm = {};
    Offsets off = {};
    int64_t n_params = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr; // fp32 params, grads, Adam
    __nv_bfloat16 *w3 = nullptr; // split bf16 weights of the forward products, [out][3 in] per layer
    __nv_bfloat16 *wt = nullptr; // transposed bf16 weights of the backward products, [in][out]
    FusedMaps maps;              // both as the kernels read them
    int sm_count = 0;
    int64_t step = 0;
    // training workspace: the buffers of `tr` for up to `cap` rows, laid out for tr.ld of them
    int64_t cap = 0;
    TrainArgs tr = {};
    WGradMaps wmaps;
    float *loss = nullptr;
    // set to 1 by a kernel whose mbarrier wait ran out: host memory the device writes, so that
    // a call reads it after its synchronisation without a copy of its own
    int *err = nullptr, *err_host = nullptr;
};

namespace {

void free_ws(gt_surrogate *s)
{
    for (int l = 0; l < N_LAYERS; l++) {
        cudaFree(s->tr.xt[l]);
        cudaFree(s->tr.dzt[l]);
    }
    cudaFree(s->tr.z);
    s->tr = TrainArgs();
    s->cap = 0;
}

// Buffers for batches of `rows` rows, laid out for exactly that many (padded to whole tiles).
int ensure_ws(gt_surrogate *s, int64_t rows, cudaStream_t st)
{
    const int64_t ld = (rows + FUSED_TILE - 1) / FUSED_TILE * FUSED_TILE;
    if (s->cap < ld) {
        free_ws(s);
        cudaError_t e = cudaSuccess;
        for (int l = 0; l < N_LAYERS && e == cudaSuccess; l++) {
            e = cudaMalloc(&s->tr.xt[l], ld * IN_DIM[l] * sizeof(__nv_bfloat16));
            if (e == cudaSuccess)
                e = cudaMalloc(&s->tr.dzt[l], ld * OUT_DIM[l] * sizeof(__nv_bfloat16));
        }
        if (e == cudaSuccess)
            e = cudaMalloc(&s->tr.z, (int64_t)fused_grid(ld, s->sm_count) * 4 * 256 * FUSED_TILE *
                                         sizeof(float));
        if (e != cudaSuccess) {
            (void)cudaGetLastError(); // a failed allocation is not sticky: no later check reports it
            free_ws(s);
            return e == cudaErrorMemoryAllocation ? GT_ERR_OOM : GT_ERR_CUDA;
        }
        s->cap = ld;
    }
    if (s->tr.ld != ld) {
        s->tr.ld = ld;
        for (int l = 0; l < N_LAYERS; l++) s->tr.db[l] = s->g + s->off.b[l];
        s->tr.loss = s->loss;
        // the network uses 4 of the last layer's 16 outputs: the other rows of its gradient stay zero
        if (cudaMemsetAsync(s->tr.dzt[N_LAYERS - 1], 0, ld * 16 * sizeof(__nv_bfloat16), st) !=
                cudaSuccess ||
            !wgrad_prepare(&s->wmaps, s->tr)) {
            s->tr.ld = 0;
            return GT_ERR_CUDA;
        }
    }
    return GT_OK;
}

struct Dev {
    int prev = -1;
    bool ok = false;
    explicit Dev(int d)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        ok = cudaSetDevice(d) == cudaSuccess;
    }
    ~Dev()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

FusedArgs net_args(gt_surrogate *s, int64_t n)
{
    FusedArgs a = {};
    a.n = n;
    a.norm = s->norm;
    for (int l = 0; l < N_LAYERS; l++) a.bias[l] = s->p + s->off.b[l];
    a.err = s->err;
    return a;
}

struct Batch {
    const double *alpha, *beta, *spin, *q, *theta0;
    const uint8_t *status;
    const double *th_end, *ph_end;
};

// Gradients of the mean loss of rows [row0, row0 + n) into s->g, the loss sum added to s->loss.
cudaError_t gradients(gt_surrogate *s, const Batch &b, int64_t row0, int64_t n, float w_dir,
                      cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(s->g, 0, s->n_params * sizeof(float), st);
    if (e != cudaSuccess) return e;
    FusedArgs a = net_args(s, n);
    a.alpha = b.alpha + row0;
    a.beta = b.beta + row0;
    a.spin = b.spin + row0;
    a.q = b.q + row0;
    a.theta0 = b.theta0 + row0;
    a.tr = s->tr;
    a.tr.status = b.status + row0;
    a.tr.th_end = b.th_end + row0;
    a.tr.ph_end = b.ph_end + row0;
    a.tr.w_dir = w_dir;
    a.tr.inv_b = 1.0f / (float)n;
    e = launch_fused_train(s->maps, a, s->sm_count, st);
    float *gw[N_LAYERS];
    for (int l = 0; l < N_LAYERS; l++) gw[l] = s->g + s->off.w[l];
    if (e == cudaSuccess) e = launch_wgrad(s->wmaps, gw, s->tr.ld, s->err, s->sm_count, st);
    return e;
}

int check_err(gt_surrogate *s, cudaStream_t st)
{
    if (cudaStreamSynchronize(st) != cudaSuccess) return GT_ERR_CUDA;
    const int h = *(volatile int *)s->err_host;
    return h ? GT_ERR_TIMEOUT : GT_OK;
}

// split and transposed bf16 weights from the parameters
cudaError_t refresh_copies(gt_surrogate *s, cudaStream_t st)
{
    update_kernel<false><<<blocks_for(s->n_params), 256, 0, st>>>(
        s->n_params, s->off, s->p, nullptr, nullptr, nullptr, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 1.0f,
        1.0f, s->w3, s->wt);
    return cudaGetLastError();
}

} // namespace

extern "C" {

int gt_surrogate_num_params(int64_t *out)
{
    if (!out) return GT_ERR_INVALID_ARG;
    int64_t n = 0;
    for (int l = 0; l < N_LAYERS; l++) n += (int64_t)OUT_DIM[l] * IN_DIM[l] + OUT_DIM[l];
    *out = n;
    return GT_OK;
}

int gt_surrogate_create(int device, const gt_surrogate_norm *nrm, uint64_t seed, gt_surrogate **out)
{
    if (!out || !nrm) return GT_ERR_INVALID_ARG;
    if (!(nrm->r0 > 0) || !(nrm->fov_deg > 0 && nrm->fov_deg < 180) || !(nrm->spin_max > 0) ||
        !(nrm->theta0_max > nrm->theta0_min) || !(nrm->q_max > 0))
        return GT_ERR_INVALID_ARG;
    *out = nullptr;
    Dev d(device);
    if (!d.ok) return GT_ERR_CUDA;
    gt_surrogate *s = new (std::nothrow) gt_surrogate();
    if (!s) return GT_ERR_OOM;
    s->device = device;
    const double V = tan(0.5 * nrm->fov_deg / 180.0 * M_PI) / nrm->r0;
    const double H = atan(tan(V));
    s->norm.inv_h = 1.0 / H;
    s->norm.inv_v = 1.0 / V;
    s->norm.spin_scale = 2.0 / nrm->spin_max;
    s->norm.spin_shift = -1.0;
    s->norm.q_scale = 1.0 / nrm->q_max;
    s->norm.th_scale = 2.0 / (nrm->theta0_max - nrm->theta0_min);
    s->norm.th_shift = -(nrm->theta0_max + nrm->theta0_min) / (nrm->theta0_max - nrm->theta0_min);
    int64_t off = 0;
    std::vector<int64_t> offs;
    std::vector<float> scales;
    for (int l = 0; l < N_LAYERS; l++) {
        s->off.w[l] = off;
        offs.push_back(off);
        // LeCun-normal weights (the 6 zero-padded input columns do not count)
        const int fan_in = l == 0 ? 10 : IN_DIM[l];
        scales.push_back((float)(1.0 / sqrt((double)fan_in)));
        off += (int64_t)OUT_DIM[l] * IN_DIM[l];
        s->off.b[l] = off;
        offs.push_back(off);
        scales.push_back(0.0f);
        off += OUT_DIM[l];
    }
    s->n_params = off;
    int64_t *d_offs = nullptr;
    float *d_scales = nullptr;
    cudaError_t e = cudaMalloc(&s->p, off * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&s->g, off * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&s->m, off * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&s->v, off * sizeof(float));
    int64_t off3 = 0;
    for (int l = 0; l < N_LAYERS; l++) {
        s->off.w3[l] = off3;
        off3 += (int64_t)OUT_DIM[l] * 3 * IN_DIM[l];
    }
    if (e == cudaSuccess) e = cudaMalloc(&s->w3, off3 * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMalloc(&s->wt, off * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMalloc(&s->loss, sizeof(float));
    if (e == cudaSuccess)
        e = cudaHostAlloc(&s->err_host, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable);
    if (e == cudaSuccess) {
        *s->err_host = 0;
        e = cudaHostGetDevicePointer(&s->err, s->err_host, 0);
    }
    if (e == cudaSuccess) e = cudaMalloc(&d_offs, offs.size() * sizeof(int64_t));
    if (e == cudaSuccess) e = cudaMalloc(&d_scales, scales.size() * sizeof(float));
    if (e == cudaSuccess)
        e = cudaMemcpy(d_offs, offs.data(), offs.size() * sizeof(int64_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(d_scales, scales.data(), scales.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(s->m, 0, off * sizeof(float));
    if (e == cudaSuccess) e = cudaMemset(s->v, 0, off * sizeof(float));
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&s->sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) {
        const void *w[N_LAYERS], *t[N_LAYERS];
        for (int l = 0; l < N_LAYERS; l++) {
            w[l] = s->w3 + s->off.w3[l];
            t[l] = s->wt + s->off.w[l];
        }
        if (!fused_prepare(&s->maps, w, t)) e = cudaErrorUnknown;
    }
    if (e == cudaSuccess) {
        init_params_kernel<<<blocks_for(off), 256>>>(s->p, off, d_offs, d_scales, (int)offs.size(), seed);
        e = refresh_copies(s, 0);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    cudaFree(d_offs);
    cudaFree(d_scales);
    if (e != cudaSuccess) {
        gt_surrogate_destroy(s);
        return e == cudaErrorMemoryAllocation ? GT_ERR_OOM : GT_ERR_CUDA;
    }
    *out = s;
    return GT_OK;
}

int gt_surrogate_destroy(gt_surrogate *s)
{
    if (!s) return GT_ERR_INVALID_ARG;
    Dev d(s->device);
    cudaDeviceSynchronize();
    free_ws(s);
    cudaFree(s->p);
    cudaFree(s->g);
    cudaFree(s->m);
    cudaFree(s->v);
    cudaFree(s->w3);
    cudaFree(s->wt);
    cudaFree(s->loss);
    cudaFreeHost(s->err_host);
    delete s;
    return GT_OK;
}

int gt_surrogate_get_params(gt_surrogate *s, float *host, int64_t n)
{
    if (!s || !host || n != s->n_params) return GT_ERR_INVALID_ARG;
    Dev d(s->device);
    return cudaMemcpy(host, s->p, n * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? GT_OK
                                                                                           : GT_ERR_CUDA;
}

int gt_surrogate_get_grads(gt_surrogate *s, float *host, int64_t n)
{
    if (!s || !host || n != s->n_params) return GT_ERR_INVALID_ARG;
    Dev d(s->device);
    return cudaMemcpy(host, s->g, n * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? GT_OK
                                                                                           : GT_ERR_CUDA;
}

int gt_surrogate_set_params(gt_surrogate *s, const float *host, int64_t n)
{
    if (!s || !host || n != s->n_params) return GT_ERR_INVALID_ARG;
    Dev d(s->device);
    cudaError_t e = cudaMemcpy(s->p, host, n * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = refresh_copies(s, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    return e == cudaSuccess ? GT_OK : GT_ERR_CUDA;
}

int gt_surrogate_eval(gt_ctx *ctx, gt_surrogate *s, int64_t n, const double *alpha,
                      const double *beta, const double *spin, const double *q,
                      const double *theta0, float *out)
{
    if (!ctx || !s || n < 0 || !alpha || !beta || !spin || !q || !theta0 || !out)
        return GT_ERR_INVALID_ARG;
    Dev d(s->device);
    cudaStream_t st = gt_internal_stream(ctx);
    FusedArgs a = net_args(s, n);
    a.alpha = alpha;
    a.beta = beta;
    a.spin = spin;
    a.q = q;
    a.theta0 = theta0;
    a.out = out;
    if (launch_fused(s->maps, a, s->sm_count, st) != cudaSuccess) return GT_ERR_CUDA;
    return check_err(s, st);
}

int gt_surrogate_grad(gt_ctx *ctx, gt_surrogate *s, int64_t n, const double *alpha,
                      const double *beta, const double *spin, const double *q,
                      const double *theta0, const uint8_t *status, const double *th_end,
                      const double *ph_end, float dir_weight, float *grads_host, float *loss_host)
{
    if (!ctx || !s || n < 1 || n > (1 << 20) || !grads_host || !loss_host) return GT_ERR_INVALID_ARG;
    Dev d(s->device);
    cudaStream_t st = gt_internal_stream(ctx);
    int rc = ensure_ws(s, n, st);
    if (rc != GT_OK) return rc;
    const Batch all = {alpha, beta, spin, q, theta0, status, th_end, ph_end};
    cudaError_t e = cudaMemsetAsync(s->loss, 0, sizeof(float), st);
    if (e == cudaSuccess) e = gradients(s, all, 0, n, dir_weight, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(grads_host, s->g, s->n_params * sizeof(float), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(loss_host, s->loss, sizeof(float), cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return GT_ERR_CUDA;
    rc = check_err(s, st);
    if (rc == GT_OK) *loss_host /= (float)n;
    return rc;
}

int gt_surrogate_train(gt_ctx *ctx, gt_surrogate *s, const gt_train_cfg *cfg, int64_t n,
                       const double *alpha, const double *beta, const double *spin,
                       const double *q, const double *theta0, const uint8_t *status,
                       const double *th_end, const double *ph_end, float *loss_per_epoch)
{
    if (!ctx || !s || !cfg || n < 1 || cfg->epochs < 1 || cfg->batch < 128 || cfg->batch % 128 ||
        cfg->batch > (1 << 20) || !(cfg->lr > 0))
        return GT_ERR_INVALID_ARG;
    Dev d(s->device);
    cudaStream_t st = gt_internal_stream(ctx);
    const int B = cfg->batch;
    int rc = ensure_ws(s, B, st);
    if (rc != GT_OK) return rc;
    const Batch all = {alpha, beta, spin, q, theta0, status, th_end, ph_end};
    const int64_t nb = n / B; // full batches only
    if (nb < 1) return GT_ERR_INVALID_ARG;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int ep = 0; ep < cfg->epochs; ep++) {
        cudaError_t e = cudaMemsetAsync(s->loss, 0, sizeof(float), st);
        // cosine learning-rate schedule over the whole run
        for (int64_t b = 0; b < nb && e == cudaSuccess; b++) {
            const double prog = ((double)ep * nb + b) / ((double)cfg->epochs * nb);
            const float lr = (float)(cfg->lr * 0.5 * (1.0 + cos(M_PI * prog)));
            e = gradients(s, all, b * B, B, (float)cfg->dir_weight, st);
            if (e != cudaSuccess) break;
            s->step++;
            const float bc1 = 1.0f - powf(b1, (float)s->step), bc2 = 1.0f - powf(b2, (float)s->step);
            update_kernel<true><<<blocks_for(s->n_params), 256, 0, st>>>(
                s->n_params, s->off, s->p, s->g, s->m, s->v, lr, b1, b2, eps,
                (float)cfg->weight_decay, bc1, bc2, s->w3, s->wt);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return GT_ERR_CUDA;
        if (loss_per_epoch) {
            float l = 0;
            e = cudaMemcpyAsync(&l, s->loss, sizeof l, cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) return GT_ERR_CUDA;
            loss_per_epoch[ep] = l / (float)(nb * B);
        }
    }
    return check_err(s, st);
}

} // extern "C"

// Inference with gating (declared in geotrace.h); needs the context's camera, so it is
// implemented next to the context in capi.cu through these helpers.
namespace gt {
namespace sg {

// The network on every pixel of the camera; its answers to `net` (float4 per pixel).
int net_pass(gt_surrogate *s, const CamDesc *d_cam, int64_t n_pix, float4 *net, cudaStream_t st)
{
    FusedArgs a = net_args(s, n_pix);
    a.cam = d_cam;
    a.out = (float *)net;
    if (launch_fused(s->maps, a, s->sm_count, st) != cudaSuccess) return GT_ERR_CUDA;
    return check_err(s, st);
}

int select_first(const CamDesc *d_cam, int64_t n_pix, const float4 *net, const ProbeGrid &pg,
                 float tau, double band, double axis, float dir_tol, int64_t *list,
                 unsigned long long *count, cudaStream_t st)
{
    select_kernel<<<blocks_for(n_pix), 256, 0, st>>>(n_pix, d_cam, net, pg, tau, band, axis,
                                                     dir_tol, list, count);
    return cudaGetLastError() == cudaSuccess ? GT_OK : GT_ERR_CUDA;
}

int probe_records(const CamDesc *d_cam, const ProbeGrid &pg, const float4 *net,
                  const uint8_t *status, const double *th, const double *ph, ProbeRec *rec,
                  cudaStream_t st)
{
    const int n = pg.nx * pg.ny;
    probe_record_kernel<<<blocks_for(n), 256, 0, st>>>(d_cam, pg, net, status, th, ph, rec);
    return cudaGetLastError() == cudaSuccess ? GT_OK : GT_ERR_CUDA;
}

int gate_rest(const CamDesc *d_cam, int64_t n_pix, const float4 *net, const ProbeGrid &pg,
              float tau, double band, double axis, float dir_tol, double *t, double *r, double *th,
              double *ph, uint8_t *status, uint32_t *nsteps, int64_t *list,
              unsigned long long *count, cudaStream_t st)
{
    gate_kernel<<<blocks_for(n_pix), 256, 0, st>>>(n_pix, d_cam, net, pg, tau, band, axis, dir_tol,
                                                   t, r, th, ph, status, nsteps, list, count);
    return cudaGetLastError() == cudaSuccess ? GT_OK : GT_ERR_CUDA;
}

} // namespace sg
} // namespace gt
