// mlp_fused.cuh -- the surrogate's forward pass in one kernel (inference).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.cuh"
#include "surrogate.cuh"

namespace gt {
namespace sg {

// Tensor maps of the split weights [w_hi | w_hi | w_lo] of each layer (64 x 128 boxes; 64 x 16
// for the last), encoded once per network.
struct FusedMaps {
    CUtensorMap w[N_LAYERS];
};

struct FusedArgs {
    int64_t n;
    // inputs: the pixels of a camera, or five arrays of n samples
    const CamDesc *cam;
    const double *alpha, *beta, *spin, *q, *theta0;
    Norm norm;
    const float *bias[N_LAYERS];
    float *out; // n x 4: logit and end direction
    int *err;   // set to 1 when an mbarrier wait ran out
};

// false when the driver cannot encode the maps
bool fused_prepare(FusedMaps *maps, const void *const w3[N_LAYERS]);
cudaError_t launch_fused(const FusedMaps &maps, const FusedArgs &a, int sm_count, cudaStream_t s);

} // namespace sg
} // namespace gt
