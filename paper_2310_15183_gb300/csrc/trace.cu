// trace.cu -- the ray-queue kernels (trace_body.cuh) but the FP32 one, and their launches.
#include "trace_body.cuh"

namespace gt {
namespace {

template <int MODE, int KIND, bool PRECISE = false>
__global__ void __launch_bounds__(256, MODE == 2 ? 2 : 1)
    trace_kernel(const __grid_constant__ TraceArgs A, int one_shot)
{
    trace_body<MODE, KIND, PRECISE, false>(A, one_shot);
}

// The double-float kernels: 168 registers, 12 warps an SM.  The Manko-Novikov sweep spills
// ~250 bytes a thread at that, which costs less than the third warp per scheduler gives:
// 200,000 Manko-Novikov rays x 1,000 steps take 67.9 ms against 69.5 ms with 252 registers
// and 8 warps (208: 69.9 ms), 48,000 rays 40.5 against 46.3 ms; Kerr (160) is the same either
// way.  A per-ray spacetime lives in registers and local memory already: it keeps 255.
template <int MODE, int KIND, bool SINGLE>
__global__ void __maxnreg__(KIND == KIND_ANY ? 255 : 168)
    pair_kernel(const __grid_constant__ TraceArgs A, int one_shot)
{
    trace_body<MODE, KIND, false, SINGLE>(A, one_shot);
}

__global__ void camera_setup_kernel(CamDesc *cams, int n, int flags, double r_switch)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    CamDesc d = cams[c];
    setup_desc(d, flags, r_switch);
    cams[c] = d;
}

} // namespace

cudaError_t launch_camera_setup(CamDesc *d_cams, int n_cams, int flags, double r_switch,
                                cudaStream_t s)
{
    const int block = 64;
    camera_setup_kernel<<<(n_cams + block - 1) / block, block, 0, s>>>(d_cams, n_cams, flags,
                                                                       r_switch);
    return cudaGetLastError();
}

// Loop condition of the graph-resident FP32-mixed rounds: continue while rays are parked.
static __global__ void set_loop_condition_kernel(cudaGraphConditionalHandle h,
                                          const unsigned long long *count)
{
    cudaGraphSetConditional(h, *count != 0ull ? 1u : 0u);
}

cudaError_t launch_set_condition(cudaGraphConditionalHandle h, const unsigned long long *count,
                                 cudaStream_t s)
{
    set_loop_condition_kernel<<<1, 1, 0, s>>>(h, count);
    return cudaGetLastError();
}

template <int MODE, int KIND>
static cudaError_t launch_one(const TraceArgs &a, int block, int grid, bool one_shot, cudaStream_t s)
{
    const int once = one_shot ? 1 : 0;
    if constexpr (MODE >= 4) {
        if (KIND < KIND_ANY && a.single)
            pair_kernel<MODE, KIND, (KIND < KIND_ANY)><<<grid, block, 0, s>>>(a, once);
        else
            pair_kernel<MODE, KIND, false><<<grid, block, 0, s>>>(a, once);
    } else if constexpr (MODE == 2) {
        if (KIND != KIND_KERR && (a.flags & GT_FLAG_PRECISE_MN))
            trace_kernel<MODE, KIND, KIND != KIND_KERR><<<grid, block, 0, s>>>(a, once);
        else
            trace_kernel<MODE, KIND><<<grid, block, 0, s>>>(a, once);
    } else {
        trace_kernel<MODE, KIND><<<grid, block, 0, s>>>(a, once);
    }
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_mode(const TraceArgs &a, int kind_hint, int block, int grid,
                               bool one_shot, cudaStream_t s)
{
    if (kind_hint == KIND_KERR) return launch_one<MODE, KIND_KERR>(a, block, grid, one_shot, s);
    if (kind_hint == KIND_MN) return launch_one<MODE, KIND_MN>(a, block, grid, one_shot, s);
    if (kind_hint == KIND_FD) {
        if constexpr (MODE == 0) return launch_one<0, KIND_FD>(a, block, grid, one_shot, s);
        return cudaErrorInvalidValue; // the listing's numerics run in FP64 only
    }
    return launch_one<MODE, KIND_ANY>(a, block, grid, one_shot, s);
}

cudaError_t launch_trace(const TraceArgs &args, int kmode, int kind_hint, int block, int grid,
                         bool one_shot, cudaStream_t s)
{
    TraceArgs a = args;
    a.sp_f = (float)a.sp;
    a.w6_f = (float)a.w6;
    a.h_thr_f = (float)(a.sp * 0.00003);
    a.sp_tf = tf_from(a.sp);
    a.w6_tf = tf_from(a.w6);
    a.h_thr_df = DF(a.sp * 0.00003);
    switch (kmode) {
    case KMODE_FP64: return launch_mode<0>(a, kind_hint, block, grid, one_shot, s);
    case KMODE_MIXED_INLINE: return launch_mode<1>(a, kind_hint, block, grid, one_shot, s);
    case KMODE_MIXED_FP32:
        // for other scales and steps (ROUTE_FTZ), and for caller states, the build that keeps denormals
        return a.ftz ? launch_trace_fp32(a, kind_hint, block, grid, one_shot, s)
                     : launch_mode<2>(a, kind_hint, block, grid, one_shot, s);
    case KMODE_ZONE_FP64: return launch_mode<3>(a, kind_hint, block, grid, one_shot, s);
    case KMODE_ZONE_PAIR: return launch_mode<4>(a, kind_hint, block, grid, one_shot, s);
    case KMODE_FP64_PAIR: return launch_mode<5>(a, kind_hint, block, grid, one_shot, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int MODE, int KIND>
static int occupancy_one(int block)
{
    int n = 0;
    cudaError_t e;
    if constexpr (MODE >= 4)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, pair_kernel<MODE, KIND, (KIND < KIND_ANY)>, block, 0);
    else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, trace_kernel<MODE, KIND>, block, 0);
    if (e != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

template <int MODE>
static int occupancy_mode(int kind_hint, int block)
{
    if (kind_hint == KIND_KERR) return occupancy_one<MODE, KIND_KERR>(block);
    if (kind_hint == KIND_MN) return occupancy_one<MODE, KIND_MN>(block);
    if (kind_hint == KIND_FD) {
        if constexpr (MODE == 0) return occupancy_one<0, KIND_FD>(block);
        return 1;
    }
    return occupancy_one<MODE, KIND_ANY>(block);
}

int max_blocks_per_sm(int kmode, int kind_hint, int block)
{
    switch (kmode) {
    case KMODE_FP64: return occupancy_mode<0>(kind_hint, block);
    case KMODE_MIXED_INLINE: return occupancy_mode<1>(kind_hint, block);
    case KMODE_MIXED_FP32: return max_blocks_per_sm_fp32(kind_hint, block);
    case KMODE_ZONE_FP64: return occupancy_mode<3>(kind_hint, block);
    case KMODE_ZONE_PAIR: return occupancy_mode<4>(kind_hint, block);
    case KMODE_FP64_PAIR: return occupancy_mode<5>(kind_hint, block);
    default: return 1;
    }
}

} // namespace gt
