// mlp_fused.cuh -- the surrogate's passes as single kernels: forward (inference),
// forward + loss + backward (training), and the weight gradients of all layers.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.cuh"
#include "surrogate.cuh"

namespace gt {
namespace sg {

// Tensor maps of the weights, encoded once per network: the split weights [w_hi | w_hi | w_lo] of
// each layer's forward product (64 x 256 boxes; 64 x 16 for the last) and the transposed bf16
// weights of each layer's backward product (64 x 256).
struct FusedMaps {
    CUtensorMap w[N_LAYERS];
    CUtensorMap wt[N_LAYERS]; // wt[0] unused
};

// Training outputs of a batch of `rows` rows, padded to `ld` = a multiple of 128.
struct TrainArgs {
    const uint8_t *status;      // labels: integrator status and end direction
    const double *th_end, *ph_end;
    float w_dir, inv_b;
    int64_t ld;
    __nv_bfloat16 *xt[N_LAYERS];  // each layer's input, transposed: [IN_DIM][ld]
    __nv_bfloat16 *dzt[N_LAYERS]; // each layer's output gradient, transposed: [OUT_DIM][ld]
    float *z;                   // pre-activations of the tile in flight: [grid][4][256][128]
    float *db[N_LAYERS];        // bias gradients, added to
    float *loss;                // loss sum, added to
};

struct FusedArgs {
    int64_t n;
    // inputs: the pixels of a camera, or five arrays of n samples
    const CamDesc *cam;
    const double *alpha, *beta, *spin, *q, *theta0;
    Norm norm;
    const float *bias[N_LAYERS];
    float *out; // n x 4: logit and end direction (inference)
    int *err;   // set to 1 when an mbarrier wait ran out
    TrainArgs tr;
};

// Rows a CTA takes at a time, and the number of CTAs of a launch over n rows.
constexpr int FUSED_TILE = 128;
int fused_grid(int64_t n, int sm_count);

// w3, wt: device weights of each layer; false when the driver cannot encode the maps
bool fused_prepare(FusedMaps *maps, const void *const w3[N_LAYERS], const void *const wt[N_LAYERS]);
cudaError_t launch_fused(const FusedMaps &maps, const FusedArgs &a, int sm_count, cudaStream_t s);
// forward, loss and backward of the rows of `a` (a.tr set)
cudaError_t launch_fused_train(const FusedMaps &maps, const FusedArgs &a, int sm_count,
                               cudaStream_t s);

// Weight gradients g[w_off[l]][n, k] += sum_b dzt[l][n, b] xt[l][k, b] of all layers in one launch.
struct WGradMaps {
    CUtensorMap a[N_LAYERS], b[N_LAYERS];
};
bool wgrad_prepare(WGradMaps *maps, const TrainArgs &t);
cudaError_t launch_wgrad(const WGradMaps &maps, float *const g[N_LAYERS], int64_t ld, int *err,
                         int sm_count, cudaStream_t s);

} // namespace sg
} // namespace gt
