// trace_fp32.cu -- the FP32 kernels of the FP32-mixed mode, compiled with -ftz=true.
//
// With denormals a reciprocal, an exponential and an inverse square root each carry two to four
// instructions of scaling around the hardware's approximation and an IEEE division its slow
// path: 100 of a Manko-Novikov step's 1,261 instructions and a tenth of a lone Kerr warp's
// step latency.  In spacetimes and cameras of ordinary scale (pair_range, steps of 1e-9 and
// more) the two compilations give the same bits: Manko-Novikov's sixth power of k / r does leave
// the normal floats far out (1e-49 at r = 1e8 M), in terms that are then below the last bit of
// the sums they enter -- except for spins within 1e-6 of extremal, where the FP32 field is wrong
// by hundreds of times itself either way.  Other scales and steps run
// trace.cu's kernel.  One GB300: 500x400
// Manko-Novikov frame of 20,000 steps 157 -> 142 ms, 301x211 Kerr shadow 306 -> 294 ms
// (264 on some views), 24 Kerr cameras 332 -> 310, labels 281 -> 267, gated image 460 -> 424; a lone
// Kerr warp 764 -> 686 cycles a step, Manko-Novikov on a full chip 1,470 -> 1,333.
#include "trace_body.cuh"

namespace gt {
namespace {

// The FP32 rounds kernel (MODE 2) is held to 128 registers: four resident blocks of 128
// threads per SM, also with PRECISE (GT_FLAG_PRECISE_MN), which needs a few more.
template <int MODE, int KIND, bool PRECISE, bool SINGLE>
__global__ void __launch_bounds__(256, 2)
    trace_kernel(const __grid_constant__ TraceArgs A, int one_shot)
{
    trace_body<MODE, KIND, PRECISE, SINGLE>(A, one_shot);
}

// ------------------------------------------------------------------ two rays per thread
// The FP32 rounds kernel (MODE 2) with two independent ray slots per thread: both slots'
// RK4 steps are issued back to back in one basic block, so the scheduler can interleave
// two dependency chains (instruction-level parallelism at half the resident threads).
// Same arithmetic per ray as trace_kernel<2, KIND>, so results are bitwise equal; for one
// camera of a fixed spacetime kind, without the watchdog, per-ray parameters, state
// arrays or the ring (the launcher falls back to one ray per thread otherwise).
struct Slot32 {
    bool active;
    int64_t id;
    uint32_t n, rp_next;
    RayMixed m;
};

template <int KIND, bool PRECISE>
__global__ void __launch_bounds__(256, 1) trace2_kernel(TraceArgs A)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    unsigned long long *next = A.scratch + SCR_NEXT_RAY;
    const CamDesc &cam = A.cams[0];
    const SpacetimeF stf = to_float(cam.st);
    const F2 r_esc_f = f2_from(cam.r_escape);
    const float r_sw_f = (float)cam.r_switch;
    const float spf = A.sp_f, w6f = A.w6_f, h_thr_f = A.h_thr_f;
    const int64_t n_in = A.in_count ? (int64_t)(*A.in_count < A.in_cap ? *A.in_count : A.in_cap) : 0;
    const int64_t n_work = A.n_fresh + n_in;
    Slot32 sl[2];
    sl[0].active = sl[1].active = false;
    bool drained = false;
    Ray64 x;

    auto start = [&](Slot32 &q, int64_t w) {
        if (w < A.n_fresh) {
            const int64_t pix = A.fresh_ids ? A.fresh_ids[w] : w;
            q.id = (A.fresh_ids && A.compact_out) ? w : pix;
            camera_init(cam, A.first + pix, x);
            q.n = 0;
            if (A.n_steps <= 0) {
                store_full(A, q.id, x, GT_RAY_MAXSTEPS, 0, nan(""));
                return false;
            }
        } else {
            const ParkItem &it = A.in_items[w - A.n_fresh];
            q.id = it.id;
            q.n = it.n;
            x.t = it.t;
            x.r = it.r;
            x.th = it.th;
            x.ph = it.ph;
            x.pr = it.pr;
            x.pth = it.pth;
            x.pt = it.pt;
            x.pph = it.pph;
        }
        mixed_from64(x, q.m);
        q.rp_next = 0xFFFFFFFFu;
        if (A.reproject_every > 0) {
            const uint64_t k = (uint64_t)A.reproject_every;
            const uint64_t nx = ((uint64_t)q.n / k + 1u) * k;
            q.rp_next = nx < 0xFFFFFFFFull ? (uint32_t)nx : 0xFFFFFFFFu;
        }
        return true;
    };

    // exit tests, zone hand-over and re-projection of one slot after its step
    auto finish = [&](Slot32 &q, float h, const RayMixed &keep) {
        ++q.n;
        int status = -1;
        const bool ok = isfinite(h) && isfinite(q.m.t.hi) && isfinite(q.m.r.hi) &&
                        isfinite(q.m.th.hi) && isfinite(q.m.ph.hi) && isfinite(q.m.pr.hi) &&
                        isfinite(q.m.pth.hi);
        if (!ok) {
            q.m = keep;
            status = GT_RAY_NONFINITE;
        } else if (q.m.r.hi > r_esc_f.hi || (q.m.r.hi == r_esc_f.hi && q.m.r.lo > r_esc_f.lo)) {
            status = GT_RAY_ESCAPED;
        } else if (h < h_thr_f) {
            status = GT_RAY_HORIZON;
        } else if ((int64_t)q.n >= A.n_steps) {
            status = GT_RAY_MAXSTEPS;
        } else if (q.m.r.hi < r_sw_f) { // enter the FP64 zone: hand the ray over
            mixed_to64(q.m, x);
            bool parked;
            park(A, q.id, q.n, 0, x, &parked);
            if (parked) q.active = false;
        } else if (q.n == q.rp_next) {
            q.rp_next = q.rp_next + (uint32_t)A.reproject_every < q.rp_next
                            ? 0xFFFFFFFFu
                            : q.rp_next + (uint32_t)A.reproject_every;
            mixed_to64(q.m, x);
            reproject_pr(cam.st, x);
            q.m.pr = f2_from(x.pr);
        }
        if (status >= 0) {
            mixed_to64(q.m, x);
            store_full(A, q.id, x, status, q.n, nan(""));
            q.active = false;
        }
    };

    for (;;) {
#pragma unroll
        for (int k = 0; k < 2; k++) { // refill each slot from the global queue
            if (drained) break;
            const unsigned need = __ballot_sync(FULL_MASK, !sl[k].active);
            if (need) {
                const int cnt = __popc(need);
                const int leader = __ffs(need) - 1;
                unsigned long long base = 0;
                if (lane == leader) base = atomicAdd(next, (unsigned long long)cnt);
                base = __shfl_sync(FULL_MASK, base, leader);
                if (base + (unsigned long long)cnt >= (unsigned long long)n_work) drained = true;
                if (!sl[k].active) {
                    const int64_t w = (int64_t)base + __popc(need & lt_mask);
                    if (w < n_work) sl[k].active = start(sl[k], w);
                }
            }
        }
        if (!__any_sync(FULL_MASK, sl[0].active || sl[1].active)) {
            if (drained) break;
            continue;
        }
        // both steps back to back (a lane's idle slot steps its last state and drops the
        // result); a slot idle in the whole warp -- the queue's tail, or more slots than
        // rays -- is skipped, a warp-uniform branch
        const bool any0 = __any_sync(FULL_MASK, sl[0].active);
        const bool any1 = __any_sync(FULL_MASK, sl[1].active);
        if (any0 && any1) {
            const RayMixed keep0 = sl[0].m, keep1 = sl[1].m;
            const float h0 = rk4_step32<KIND, PRECISE>(stf, sl[0].m, spf, w6f);
            const float h1 = rk4_step32<KIND, PRECISE>(stf, sl[1].m, spf, w6f);
            if (sl[0].active) finish(sl[0], h0, keep0);
            if (sl[1].active) finish(sl[1], h1, keep1);
        } else if (any0) { // static slot indices keep the slots in registers
            const RayMixed keep = sl[0].m;
            const float h = rk4_step32<KIND, PRECISE>(stf, sl[0].m, spf, w6f);
            if (sl[0].active) finish(sl[0], h, keep);
        } else {
            const RayMixed keep = sl[1].m;
            const float h = rk4_step32<KIND, PRECISE>(stf, sl[1].m, spf, w6f);
            if (sl[1].active) finish(sl[1], h, keep);
        }
    }
}

} // namespace

template <int KIND>
static cudaError_t launch_two(const TraceArgs &a, int block, int grid, cudaStream_t s)
{
    if constexpr (KIND == KIND_MN) {
        if (a.flags & GT_FLAG_PRECISE_MN) {
            trace2_kernel<KIND, true><<<grid, block, 0, s>>>(a);
            return cudaGetLastError();
        }
    }
    trace2_kernel<KIND, false><<<grid, block, 0, s>>>(a);
    return cudaGetLastError();
}

bool two_rays_supported(const TraceArgs &a, int kmode, int kind_hint)
{
    return kmode == KMODE_MIXED_FP32 && (kind_hint == KIND_KERR || kind_hint == KIND_MN) &&
           a.ftz && a.n_cams == 1 && !a.rays && !a.states.t && !a.disk.on && a.timeout_ns == 0;
}

cudaError_t launch_trace_two(const TraceArgs &args, int kind_hint, int block, int grid,
                             cudaStream_t s)
{
    TraceArgs a = args;
    a.sp_f = (float)a.sp;
    a.w6_f = (float)a.w6;
    a.h_thr_f = (float)(a.sp * 0.00003);
    a.sp_tf = tf_from(a.sp);
    a.w6_tf = tf_from(a.w6);
    a.h_thr_df = DF(a.sp * 0.00003);
    return kind_hint == KIND_KERR ? launch_two<KIND_KERR>(a, block, grid, s)
                                  : launch_two<KIND_MN>(a, block, grid, s);
}

int max_blocks_per_sm_two(int kind_hint, int block)
{
    int n = 0;
    const cudaError_t e = kind_hint == KIND_KERR
        ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, trace2_kernel<KIND_KERR, false>, block, 0)
        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, trace2_kernel<KIND_MN, false>, block, 0);
    return (e == cudaSuccess && n > 0) ? n : 1;
}

template <int KIND>
static cudaError_t launch_fp32(const TraceArgs &a, int block, int grid, int once, cudaStream_t s)
{
    // Manko-Novikov's thirteen constants as kernel parameters: no spills, 3 % faster.  (Kerr
    // gains nothing from it, and compiles to other fused multiply-adds.)
    constexpr bool CAN_SINGLE = KIND == KIND_MN;
    constexpr bool CAN_PRECISE = KIND != KIND_KERR;
    const bool precise = CAN_PRECISE && (a.flags & GT_FLAG_PRECISE_MN);
    if (CAN_SINGLE && a.single) {
        if (precise)
            trace_kernel<2, KIND, CAN_PRECISE, CAN_SINGLE><<<grid, block, 0, s>>>(a, once);
        else
            trace_kernel<2, KIND, false, CAN_SINGLE><<<grid, block, 0, s>>>(a, once);
    } else if (precise) {
        trace_kernel<2, KIND, CAN_PRECISE, false><<<grid, block, 0, s>>>(a, once);
    } else {
        trace_kernel<2, KIND, false, false><<<grid, block, 0, s>>>(a, once);
    }
    return cudaGetLastError();
}

cudaError_t launch_trace_fp32(const TraceArgs &a, int kind_hint, int block, int grid, bool one_shot,
                              cudaStream_t s)
{
    const int once = one_shot ? 1 : 0;
    if (kind_hint == KIND_KERR) return launch_fp32<KIND_KERR>(a, block, grid, once, s);
    if (kind_hint == KIND_MN) return launch_fp32<KIND_MN>(a, block, grid, once, s);
    if (kind_hint == KIND_ANY) return launch_fp32<KIND_ANY>(a, block, grid, once, s);
    return cudaErrorInvalidValue; // the listing's numerics run in FP64 only
}

int max_blocks_per_sm_fp32(int kind_hint, int block)
{
    int n = 0;
    cudaError_t e;
    if (kind_hint == KIND_KERR)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, trace_kernel<2, KIND_KERR, false, false>, block, 0);
    else if (kind_hint == KIND_MN)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, trace_kernel<2, KIND_MN, false, false>, block, 0);
    else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, trace_kernel<2, KIND_ANY, false, false>, block, 0);
    return e == cudaSuccess && n > 0 ? n : 1;
}

} // namespace gt
