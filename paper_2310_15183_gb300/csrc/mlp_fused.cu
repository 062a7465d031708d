// mlp_fused.cu -- features and all five layers of the surrogate for 128 rows at a time, the
// activations never leaving the SM; with TRAIN also the loss and the input gradients of the
// same rows, followed by one launch for the weight gradients of all layers.
//
// Inference.  What bounds it: the split-precision products cost 48 MMAs (128 x 256 x 16, ~135
// cycles each) per hidden layer and tile, and SiLU two MUFU operations per element, 4,100 cycles of an SM's
// 16 a clock; layer-by-layer GEMMs added 3 KB of activations per row and layer through HBM and
// L2, a pass for the features and one for the outputs.  Here a persistent CTA per SM keeps the
// activations of its 128 rows in shared memory as the two bf16 halves (128 KB, the K-major
// 128-byte-swizzled operand layout) and streams the weights from L2 in 64 x 256 boxes through
// a ring of three (96 KB; the last layer's 24 KB in one slot).  Two accumulators in TMEM
// alternate, and the epilogue hands over its output in K-chunks of 64 columns, which the next
// layer's MMAs follow: all three products of a chunk at once, so that only the last chunk's
// 12 MMAs remain when the epilogue is done, and w_hi is fetched once (256 KB a layer).
// Training, whose parameters after many steps carry any change of rounding, and images, whose
// end angles are stored in FP64 and whose gates are decided by the logits' last bits, keep the
// order of the split GEMM, x_hi w_hi (K = 0..255), x_lo w_hi, x_hi w_lo: its first third follows
// the chunks and 32 MMAs remain.
//
// Measured on one GB300: 2^20 rows 3.19 ms with a GEMM per layer (0.9 ms of MMAs at 0.47 of
// the bf16 peak, the rest traffic and SiLU passes), 1.37 in one kernel, 1.13 with a chunk's
// products together; 300 rows 103 us, 49 and 43.  Error against FP64 over 128 to 4,096 rows:
// 4.9e-7 rms (5.1e-7 in the order of the split GEMM).  Tried and not kept: two halves of 128 columns per layer with
// w_hi held for both passes (1.87 ms: an MMA takes ~105 cycles at N = 128 against ~135 at
// N = 256); the accumulator handed over whole (1.60 ms); the TMEM load of the next chunk
// started before this one's SiLU (1.23 against 1.13 ms: spills at 80 registers).
//
// Training.  A step of 8,192 rows was 37 launches and 467 us on the device: four SiLU-backward
// passes that read row-major FP32 matrices down their columns (46 us each), five column sums
// (13), ten GEMMs of 7 to 14 us with one or two waves' worth of latency each, ten copies of the
// weights.  In the fused kernel the gradient of a tile goes back through the operand buffer the
// way the activations came, the epilogue forming dZ = dX SiLU'(Z) from pre-activations the same
// thread stored (512 KB per CTA, in L2), the transposed bf16 copies for the weight gradients
// and the column sums; MMA order and elementwise formulas are those of the separate kernels.  A
// step is four launches: clear, fused, weight gradients, AdamW with both weight copies.
// A step of 8,192 rows is one tile a CTA, run once: four copies of the epilogue's chunk loop
// cost 15,000 of the kernel's 155,000 cycles in instruction fetches, so training rolls it.
// Measured: 8 steps of 8,192 rows 3.88 -> 0.77 ms; loss and gradients of 16,384 rows with
// their copy to the host 743 -> 133 us.
//
// Warps: 0 loads, 1 issues the MMAs, 2-5 compute the next tile's features (and labels) while
// the current one runs, 6-21 drain the accumulator: bias, SiLU, split, back into the operand
// buffer.  All hand-offs are mbarriers with bounded waits; a wait that runs out sets the
// error flag and every role leaves its loop.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include "features.cuh"
#include "mlp_fused.cuh"
#include "tc_gemm.cuh"
#include "tma_map.cuh"
#include "../../include/geotrace.h"

namespace gt {
namespace sg {

namespace {

constexpr int TILE = FUSED_TILE;
constexpr int RING = 3;
constexpr int FEAT_WARPS = 4, EPI_WARPS = 16;
constexpr int THREADS = 32 * (2 + FEAT_WARPS + EPI_WARPS);
constexpr uint32_t BOX = 64 * 128 * 2;       // one K-chunk of activations
constexpr uint32_t WBOX = 64 * 256 * 2;      // one K-chunk of a layer's weights
constexpr uint32_t OBOX = 64 * 16 * 2;       // one K-chunk of the last layer's
constexpr uint32_t A_BYTES = 8 * BOX;        // hi: 4 K-chunks, lo: 4 K-chunks
constexpr uint32_t BAR_OFF = A_BYTES + RING * WBOX;
constexpr uint32_t N_BAR = 2 * RING + 9;
constexpr uint32_t LAB_OFF = BAR_OFF + 8 * N_BAR + 16;      // labels of the tile (training)
constexpr uint32_t SMEM = LAB_OFF + TILE * 12 + 1024;       // + alignment to the swizzle period
constexpr uint32_t WAIT_LIMIT = 1u << 24;
static_assert(SMEM <= 227 * 1024, "shared memory per CTA");

// 1 / (1 + exp(-z)): the hardware's reciprocal and one Newton step (error 2^-46 and one rounding;
// the denominator is at least 1 and held below 2^125, where the reciprocal leaves the normal
// floats).  An IEEE division has a slow path, and its branch kept the 16 elements of a chunk from
// overlapping: 8 training steps of 8,192 rows 850 against 765 us.
__device__ __forceinline__ float sigmoidf(float z)
{
    const float e = __expf(-z), x = 1.0f + (e > 0x1p125f ? 0x1p125f : e); // NaN stays NaN
    const float y = __fdividef(1.0f, x);
    return fmaf(y, fmaf(-x, y, 1.0f), y);
}
__device__ __forceinline__ float silu(float z) { return __fdividef(z, 1.0f + __expf(-z)); }

// One kind::f16 MMA from the low words of two SW128 K-major descriptors (address >> 4 and the
// fixed leading offset; the high word is a constant): the issuing thread adds 2 per K-slice
// and 1024 per box instead of building 64-bit descriptors.
constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return (saddr >> 4) | (1u << 16); }
template <bool ACCUMULATE>
__device__ __forceinline__ void mma_lo(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .b64 da, db;\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %4};\n\tmov.b64 db, {%2, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}\n" ::"r"(d),
        "r"(a), "r"(b), "r"(idesc), "r"(DESC_HI), "n"(ACCUMULATE ? 1 : 0));
}

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 a, __nv_bfloat16 b)
{
    const __nv_bfloat162 h = __halves2bfloat162(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// eight consecutive values as their bf16 halves: hi = bf16(v), lo = bf16(v - hi)
__device__ __forceinline__ void split8(const float *v, uint4 &hi, uint4 &lo)
{
    uint32_t *h = &hi.x, *l = &lo.x;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const __nv_bfloat16 a = __float2bfloat16(v[2 * j]), b = __float2bfloat16(v[2 * j + 1]);
        h[j] = pack2(a, b);
        l[j] = pack2(__float2bfloat16(v[2 * j] - __bfloat162float(a)),
                     __float2bfloat16(v[2 * j + 1] - __bfloat162float(b)));
    }
}

// Sums of the warp's 32 rows for 16 columns held one row a lane: each step halves the columns a
// lane keeps, and after four of them lanes c and c + 16 (bit-reversed pairs) hold halves of one
// column; lanes 0..15 end with the sum of column `lane`.
__device__ __forceinline__ float column_sums(const float (&v)[16], int lane)
{
    float a[8], b[4], c[2];
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const float keep = lane & 8 ? v[j + 8] : v[j], send = lane & 8 ? v[j] : v[j + 8];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const float keep = lane & 4 ? a[j + 4] : a[j], send = lane & 4 ? a[j] : a[j + 4];
        b[j] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
#pragma unroll
    for (int j = 0; j < 2; j++) {
        const float keep = lane & 2 ? b[j + 2] : b[j], send = lane & 2 ? b[j] : b[j + 2];
        c[j] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    const float keep = lane & 1 ? c[1] : c[0], send = lane & 1 ? c[0] : c[1];
    float s = keep + __shfl_xor_sync(0xffffffffu, send, 1);
    return s + __shfl_xor_sync(0xffffffffu, s, 16);
}

template <bool TRAIN>
__global__ void __launch_bounds__(THREADS, 1)
    fused_kernel(const __grid_constant__ FusedMaps maps, const __grid_constant__ FusedArgs g)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t act = tc::smem_u32(smem), ring = act + A_BYTES, bar = act + BAR_OFF;
    auto FULL = [&](uint32_t s) { return bar + 8u * s; };
    auto EMPTY = [&](uint32_t s) { return bar + 8u * (RING + s); };
    auto ACC = [&](uint32_t b) { return bar + 8u * (2 * RING + b); };     // accumulator complete
    auto ACT = [&](uint32_t k) { return bar + 8u * (2 * RING + 2 + k); }; // K-chunk k written
    const uint32_t TAIL = bar + 8u * (2 * RING + 6); // last layer's MMAs complete (per tile)
    const uint32_t FEAT = TAIL + 8u;                 // features of a tile in the operand buffer
    const uint32_t DONE = TAIL + 16u;
    float *labels = reinterpret_cast<float *>(smem + LAB_OFF); // 128 x 3
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + BAR_OFF + 8 * N_BAR);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t tiles = (g.n + TILE - 1) / TILE;

    if (warp == 1) tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);
    if (threadIdx.x == 0) {
        for (int s = 0; s < RING; s++) {
            tc::mbar_init(FULL(s), 1);
            tc::mbar_init(EMPTY(s), 1);
        }
        for (int b = 0; b < 2; b++) tc::mbar_init(ACC(b), 1);
        for (int k = 0; k < 4; k++) tc::mbar_init(ACT(k), EPI_WARPS);
        tc::mbar_init(TAIL, 1);
        tc::mbar_init(FEAT, FEAT_WARPS);
        tc::mbar_init(DONE, 1);
        tc::fence_mbarrier_init();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    const bool by_chunk = !TRAIN && g.cam == nullptr; // order of a hidden layer's MMAs
    bool ok = true;

    if (warp == 0) {
        if (lane == 0) { // ---- weights
            uint32_t q = 0;
            // n boxes of `bytes` each (K-chunks k0, k0 + 1, ...) into the next slot; l < 0: the
            // transposed weights of layer -l
            auto load = [&](int l, int k0, int n, uint32_t bytes) {
                const uint32_t s = q % RING;
                if (q >= RING && !tc::mbar_wait(EMPTY(s), (q / RING - 1) & 1, WAIT_LIMIT)) ok = false;
                if (!ok) return;
                tc::mbar_expect_tx(FULL(s), n * bytes);
                for (int i = 0; i < n; i++)
                    tc::tma_load_2d(ring + s * WBOX + i * bytes, l < 0 ? &maps.wt[-l] : &maps.w[l],
                                    64 * (k0 + i), 0, FULL(s));
                ++q;
            };
            for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
                load(0, 0, 1, WBOX);
                for (int l = 1; l < N_LAYERS - 1; l++) {
                    if (by_chunk) {
                        for (int k = 0; k < 4; k++) {
                            load(l, k, 1, WBOX);     // w_hi
                            load(l, 8 + k, 1, WBOX); // w_lo
                        }
                    } else {
                        for (int k = 0; k < 12; k++) load(l, k, 1, WBOX); // w_hi, w_hi, w_lo
                    }
                }
                load(N_LAYERS - 1, 0, 12, OBOX); // the last layer's 24 KB in one slot
                if (TRAIN) {
                    load(-(N_LAYERS - 1), 0, 1, WBOX);
                    for (int l = N_LAYERS - 2; l >= 1; l--)
                        for (int k = 0; k < 4; k++) load(-l, k, 1, WBOX);
                }
            }
            // copies still in flight (only after a failed wait) land before the CTA exits
            for (uint32_t j = q > RING ? q - RING : 0; j < q; ++j)
                if (!tc::mbar_wait(FULL(j % RING), (j / RING) & 1, WAIT_LIMIT)) ok = false;
        }
    } else if (warp == 1) {
        if (lane == 0) { // ---- MMA
            const uint32_t id_h = tc::idesc_bf16_f32(TILE, 256);
            const uint32_t id_o = tc::idesc_bf16_f32(TILE, 16);
            uint32_t q = 0, hid = 0, acc = 0, tl = 0;
            auto full = [&](uint32_t j) {
                if (ok) ok = tc::mbar_wait(FULL(j % RING), (j / RING) & 1, WAIT_LIMIT);
                tc::fence_after_sync();
                return ok;
            };
            const uint32_t a_lo = desc_lo(act), b_lo = desc_lo(ring);
            // four K-slices of activation chunk c (0-3 hi, 4-7 lo) with the weights at b
            auto mma4 = [&](uint32_t d, uint32_t c, uint32_t b, uint32_t idesc, bool first) {
                const uint32_t a = a_lo + c * (BOX >> 4);
                if (first)
                    mma_lo<false>(d, a, b, idesc);
                else
                    mma_lo<true>(d, a, b, idesc);
#pragma unroll
                for (int kk = 1; kk < 4; kk++) mma_lo<true>(d, a + 2 * kk, b + 2 * kk, idesc);
            };
            auto slot = [&](uint32_t j) { return b_lo + (j % RING) * (WBOX >> 4); };
            // K-chunk k of the hidden layer's input has been written (and every earlier read of
            // the accumulator about to be overwritten is done: the same warps did it before)
            auto input = [&](uint32_t k) {
                if (ok) ok = tc::mbar_wait(ACT(k), hid & 1, WAIT_LIMIT);
                tc::fence_after_sync();
                return ok;
            };
            for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++tl) {
                // first layer: K' = 48 in one chunk
                ok = tc::mbar_wait(FEAT, tl & 1, WAIT_LIMIT);
                tc::fence_after_sync();
                if (!full(q)) break;
                mma4(tmem + 256 * (acc & 1), 0, slot(q), id_h, true);
                tc::mma_commit(EMPTY(q % RING));
                tc::mma_commit(ACC(acc & 1));
                ++q;
                ++acc;
                for (int l = 1; l < N_LAYERS - 1 && ok; l++, hid++, acc++) {
                    const uint32_t d = tmem + 256 * (acc & 1);
                    for (uint32_t k = 0; k < 4 && ok && by_chunk; k++, q += 2) {
                        if (!input(k) || !full(q)) break;
                        mma4(d, k, slot(q), id_h, k == 0); // x_hi w_hi
                        mma4(d, 4 + k, slot(q), id_h, false); // x_lo w_hi
                        tc::mma_commit(EMPTY(q % RING));
                        if (!full(q + 1)) break;
                        mma4(d, k, slot(q + 1), id_h, false); // x_hi w_lo
                        tc::mma_commit(EMPTY((q + 1) % RING));
                    }
                    for (uint32_t k = 0; k < 12 && ok && !by_chunk; k++, q++) { // x_hi w_hi, x_lo w_hi, x_hi w_lo
                        if (k < 4 && !input(k)) break;
                        if (!full(q)) break;
                        mma4(d, k < 8 ? k : k - 8, slot(q), id_h, k == 0);
                        tc::mma_commit(EMPTY(q % RING));
                    }
                    if (ok) tc::mma_commit(ACC(acc & 1));
                }
                if (!ok || !full(q)) break;
                const uint32_t d = tmem + 256 * (acc & 1);
                for (uint32_t k = 0; k < 12 && ok; k++)
                    if (k >= 4 || input(k))
                        mma4(d, k < 8 ? k : k - 8, slot(q) + k * (OBOX >> 4), id_o, k == 0);
                if (!ok) break;
                tc::mma_commit(EMPTY(q % RING));
                if (!TRAIN) tc::mma_commit(TAIL);
                tc::mma_commit(ACC(acc & 1));
                ++q;
                ++hid;
                ++acc;
                if (!TRAIN) continue;
                // input gradients: the last layer's 16 columns in one K-slice, then 256
                if (!input(0) || !full(q)) break;
                mma_lo<false>(tmem + 256 * (acc & 1), a_lo, slot(q), id_h);
                tc::mma_commit(EMPTY(q % RING));
                tc::mma_commit(ACC(acc & 1));
                ++q;
                ++hid;
                ++acc;
                for (int l = N_LAYERS - 2; l >= 1 && ok; l--, hid++, acc++) {
                    for (uint32_t k = 0; k < 4 && ok; k++, q++) {
                        if (!input(k) || !full(q)) break;
                        mma4(tmem + 256 * (acc & 1), k, slot(q), id_h, k == 0);
                        tc::mma_commit(EMPTY(q % RING));
                    }
                    if (!ok) break;
                    if (l == 1) tc::mma_commit(TAIL);
                    tc::mma_commit(ACC(acc & 1));
                }
            }
            // every issued MMA completes before the accumulator is freed
            tc::mma_commit(DONE);
            if (!tc::mbar_wait(DONE, 0, WAIT_LIMIT)) ok = false;
        }
    } else if (warp < 2 + FEAT_WARPS) { // ---- features, one row a thread
        const int row = (warp - 2) * 32 + lane;
        uint32_t tl = 0;
        for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++tl) {
            const int64_t r = t * TILE + row;
            float f[16];
            if (r >= g.n) {
#pragma unroll
                for (int j = 0; j < 16; j++) f[j] = 0.0f;
            } else if (g.cam) {
                pixel_features(*g.cam, r, g.norm, f);
            } else {
                make_features(g.alpha[r], g.beta[r], g.spin[r], g.q[r], g.theta0[r], g.norm, f);
            }
            float lab[3] = {0.0f, 0.0f, 0.0f}; // end direction; zero when the ray did not escape
            if (TRAIN && r < g.n && g.tr.status[r] == GT_RAY_ESCAPED)
                unit_vector(g.tr.th_end[r], g.tr.ph_end[r], lab);
            if (TRAIN) {
#pragma unroll
                for (int j = 0; j < 16; j++) g.tr.xt[0][j * g.tr.ld + r] = __float2bfloat16(f[j]);
            }
            uint4 hi[2], lo[2];
            split8(f, hi[0], lo[0]);
            split8(f + 8, hi[1], lo[1]);
            // the previous tile's last layer has read the operand buffer
            if (tl > 0) ok = tc::mbar_wait_warp(TAIL, (tl - 1) & 1, WAIT_LIMIT);
            if (!ok) break;
            // row [hi 0..15 | lo 0..15 | hi 0..15 | 0] of one 64-wide chunk
            uint8_t *base = smem + row * 128;
            const uint4 zero = make_uint4(0, 0, 0, 0);
            const uint4 v[8] = {hi[0], hi[1], lo[0], lo[1], hi[0], hi[1], zero, zero};
#pragma unroll
            for (int c = 0; c < 8; c++)
                *reinterpret_cast<uint4 *>(base + ((c ^ (row & 7)) << 4)) = v[c];
            if (TRAIN) {
#pragma unroll
                for (int j = 0; j < 3; j++) labels[3 * row + j] = lab[j];
            }
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(FEAT);
        }
    } else { // ---- epilogue: TMEM lanes 32 (warp % 4), 16 columns of each K-chunk of 64
        const int quarter = warp & 3, group = (warp - 2 - FEAT_WARPS) >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16);
        // this row's 16-byte pieces 2 group, 2 group + 1 of a chunk, 128-byte swizzled
        uint8_t *const p0 = smem + row * 128 + (((2 * group) ^ (row & 7)) << 4);
        uint8_t *const p1 = smem + row * 128 + (((2 * group + 1) ^ (row & 7)) << 4);
        // training: this thread's pre-activations, [layer][column][row]
        float *const zrow = TRAIN ? g.tr.z + (int64_t)blockIdx.x * 4 * 256 * TILE + 16 * group * TILE + row
                                  : nullptr;
        uint32_t acc = 0, tl = 0;
        for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++tl) {
            const int64_t r = t * TILE + row;
            for (int l = 0; l < N_LAYERS - 1 && ok; l++, acc++) {
                // two barriers in turn: one flips again only after every warp has passed it
                ok = tc::mbar_wait_warp(ACC(acc & 1), (acc >> 1) & 1, WAIT_LIMIT);
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t src = t_row + 256 * (acc & 1) + 16 * group;
                const float4 *b4 = reinterpret_cast<const float4 *>(g.bias[l] + 16 * group);
#pragma unroll (TRAIN ? 1 : 4)
                for (int k = 0; k < 4; k++) {
                    float v[16];
                    tc::tmem_ld16(src + 64 * k, v);
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const float4 b = __ldg(b4 + 16 * k + j);
                        v[4 * j] += b.x;
                        v[4 * j + 1] += b.y;
                        v[4 * j + 2] += b.z;
                        v[4 * j + 3] += b.w;
                    }
                    if (TRAIN) {
#pragma unroll
                        for (int j = 0; j < 16; j++) zrow[((l * 4 + k) * 64 + j) * TILE] = v[j];
                    }
#pragma unroll
                    for (int j = 0; j < 16; j++) v[j] = silu(v[j]);
                    if (TRAIN) {
                        __nv_bfloat16 *xt = g.tr.xt[l + 1] + (64 * k + 16 * group) * g.tr.ld + r;
#pragma unroll
                        for (int j = 0; j < 16; j++) xt[j * g.tr.ld] = __float2bfloat16(v[j]);
                    }
                    uint4 hi, lo;
                    split8(v, hi, lo);
                    *reinterpret_cast<uint4 *>(p0 + k * BOX) = hi;
                    *reinterpret_cast<uint4 *>(p0 + (4 + k) * BOX) = lo;
                    split8(v + 8, hi, lo);
                    *reinterpret_cast<uint4 *>(p1 + k * BOX) = hi;
                    *reinterpret_cast<uint4 *>(p1 + (4 + k) * BOX) = lo;
                    tc::fence_proxy_async();
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(ACT(k));
                }
            }
            if (!ok) break;
            ok = tc::mbar_wait_warp(ACC(acc & 1), (acc >> 1) & 1, WAIT_LIMIT);
            if (!ok) break;
            if (!TRAIN && group == 0) {
                tc::fence_after_sync();
                float v[16];
                tc::tmem_ld16(t_row + 256 * (acc & 1), v);
                tc::fence_before_sync();
                if (r < g.n) {
                    const float *b = g.bias[N_LAYERS - 1];
                    float *o = g.out + 4 * r;
                    const float4 z = make_float4(v[0] + __ldg(b), v[1] + __ldg(b + 1),
                                                 v[2] + __ldg(b + 2), v[3] + __ldg(b + 3));
                    if (((uintptr_t)g.out & 15u) == 0) {
                        *reinterpret_cast<float4 *>(o) = z;
                    } else {
                        o[0] = z.x;
                        o[1] = z.y;
                        o[2] = z.z;
                        o[3] = z.w;
                    }
                }
            }
            if (TRAIN && group == 0) { // ---- loss and its gradient, one row a thread
                ok = tc::mbar_wait_warp(FEAT, tl & 1, WAIT_LIMIT); // the labels, written with the features
                if (!ok) break;
                tc::fence_after_sync();
                float v[16];
                tc::tmem_ld16(t_row + 256 * (acc & 1), v);
                const float *b = g.bias[N_LAYERS - 1], *lab = labels + 3 * row;
                float loss = 0.0f, gz[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (r < g.n) {
                    // BCE(logit, y) + w_dir y |d_pred - d|^2, BCE in its stable form
                    const float y = g.tr.status[r] == GT_RAY_ESCAPED ? 1.0f : 0.0f;
                    const float zl = v[0] + __ldg(b);
                    loss = fmaxf(zl, 0.0f) - zl * y + log1pf(__expf(-fabsf(zl)));
                    gz[0] = (sigmoidf(zl) - y) * g.tr.inv_b;
#pragma unroll
                    for (int j = 1; j < 4; j++) {
                        const float d = v[j] + __ldg(b + j) - lab[j - 1];
                        loss += g.tr.w_dir * y * d * d;
                        gz[j] = 2.0f * g.tr.w_dir * y * d * g.tr.inv_b;
                    }
                }
                float sum[5] = {gz[0], gz[1], gz[2], gz[3], loss};
#pragma unroll
                for (int j = 0; j < 5; j++) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], o);
                }
                if (lane == 0) {
#pragma unroll
                    for (int j = 0; j < 4; j++) atomicAdd(g.tr.db[N_LAYERS - 1] + j, sum[j]);
                    atomicAdd(g.tr.loss, sum[4]);
                }
                // columns 4..15 of the gradient are zero (their rows of dzt stay as cleared)
                __nv_bfloat16 hz[4];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    hz[j] = __float2bfloat16(gz[j]);
                    g.tr.dzt[N_LAYERS - 1][j * g.tr.ld + r] = hz[j];
                }
                uint8_t *base = smem + row * 128;
                *reinterpret_cast<uint4 *>(base + ((row & 7) << 4)) =
                    make_uint4(pack2(hz[0], hz[1]), pack2(hz[2], hz[3]), 0, 0);
                *reinterpret_cast<uint4 *>(base + ((1 ^ (row & 7)) << 4)) = make_uint4(0, 0, 0, 0);
                tc::fence_proxy_async();
                tc::fence_before_sync();
            }
            ++acc;
            if (!TRAIN) continue;
            // every warp arrives on every chunk's barrier, written or not: their phases stay equal
            __syncwarp();
            if (lane == 0)
                for (int k = 0; k < 4; k++) tc::mbar_arrive(ACT(k));
            for (int l = N_LAYERS - 2; l >= 0 && ok; l--, acc++) { // dZ_l = dX_(l+1) SiLU'(Z_l)
                float z[16];
                const float *zl = zrow + (int64_t)l * 256 * TILE;
#pragma unroll
                for (int j = 0; j < 16; j++) z[j] = zl[j * TILE];
                ok = tc::mbar_wait_warp(ACC(acc & 1), (acc >> 1) & 1, WAIT_LIMIT);
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t src = t_row + 256 * (acc & 1) + 16 * group;
#pragma unroll 1
                for (int k = 0; k < 4; k++) {
                    float v[16];
                    tc::tmem_ld16(src + 64 * k, v);
#pragma unroll
                    for (int j = 0; j < 16; j++) {
                        const float s = sigmoidf(z[j]);
                        v[j] = v[j] * s * (1.0f + z[j] * (1.0f - s));
                    }
                    if (k < 3) {
#pragma unroll
                        for (int j = 0; j < 16; j++) z[j] = zl[((k + 1) * 64 + j) * TILE];
                    }
                    uint32_t h[8];
                    __nv_bfloat16 *dzt = g.tr.dzt[l] + (64 * k + 16 * group) * g.tr.ld + r;
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const __nv_bfloat16 a = __float2bfloat16(v[2 * j]), b = __float2bfloat16(v[2 * j + 1]);
                        dzt[2 * j * g.tr.ld] = a;
                        dzt[(2 * j + 1) * g.tr.ld] = b;
                        h[j] = pack2(a, b);
                    }
                    if (l > 0) {
                        *reinterpret_cast<uint4 *>(p0 + k * BOX) = make_uint4(h[0], h[1], h[2], h[3]);
                        *reinterpret_cast<uint4 *>(p1 + k * BOX) = make_uint4(h[4], h[5], h[6], h[7]);
                        tc::fence_proxy_async();
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(ACT(k));
                    }
                    const float s = column_sums(v, lane);
                    if (lane < 16) atomicAdd(g.tr.db[l] + 64 * k + 16 * group + lane, s);
                }
                if (l == 0) {
                    tc::fence_before_sync();
                    __syncwarp();
                }
            }
        }
    }
    if (!ok && g.err) atomicExch(g.err, 1);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ weight gradients
// dW_l[n, k] = sum_b dzt_l[n, b] xt_l[k, b]: nine 128 x (256 | 16) output tiles over the five
// layers, each split over the batch so that one wave of CTAs covers the chip; a CTA runs one
// tile and one range of the batch through a ring of four 64-wide chunks and adds its 128 x 256
// partial sums to the gradient with 16-byte reductions.  Bound by latency at a batch of 8,192
// (a CTA has 8 chunks) and by the reads of both operands for large batches.
constexpr int WG_RING = 4, WG_EPI = 8;
constexpr uint32_t WG_STAGE = BOX + WBOX;
constexpr uint32_t WG_BAR = WG_RING * WG_STAGE;
constexpr uint32_t WG_SMEM = WG_BAR + 8 * (2 * WG_RING + 1) + 16 + 1024;
constexpr int WG_TILES = 9; // layers 0..3: two 128-row halves of dW; layer 4: one

struct WGradArgs {
    float *g[N_LAYERS];
    int chunks; // 64-wide chunks of the batch
    int *err;
};

__global__ void __launch_bounds__(64 + 32 * WG_EPI, 1)
    wgrad_kernel(const __grid_constant__ WGradMaps maps, const __grid_constant__ WGradArgs g)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t base = tc::smem_u32(smem), bar = base + WG_BAR;
    auto FULL = [&](uint32_t s) { return bar + 8u * s; };
    auto EMPTY = [&](uint32_t s) { return bar + 8u * (WG_RING + s); };
    const uint32_t ACC = bar + 8u * (2 * WG_RING);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + WG_BAR + 8 * (2 * WG_RING + 1));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x, l = tile >> 1, m0 = (tile & 1) * 128;
    const int n_cols = l == 0 ? 16 : 256, n_rows = l == N_LAYERS - 1 ? 16 : 256;
    const int per = (g.chunks + gridDim.y - 1) / gridDim.y;
    const int c0 = blockIdx.y * per, c1 = min(g.chunks, c0 + per);
    if (warp == 1) tc::tmem_alloc(tc::smem_u32(tmem_slot), 256);
    if (threadIdx.x == 0) {
        for (int s = 0; s < WG_RING; s++) {
            tc::mbar_init(FULL(s), 1);
            tc::mbar_init(EMPTY(s), 1);
        }
        tc::mbar_init(ACC, 1);
        tc::fence_mbarrier_init();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            const uint32_t bytes = BOX + (uint32_t)n_cols * 128;
            uint32_t q = 0;
            for (int c = c0; c < c1; c++, q++) {
                const uint32_t s = q % WG_RING;
                if (q >= WG_RING && !tc::mbar_wait(EMPTY(s), (q / WG_RING - 1) & 1, WAIT_LIMIT)) {
                    ok = false;
                    break;
                }
                tc::mbar_expect_tx(FULL(s), bytes);
                tc::tma_load_2d(base + s * WG_STAGE, &maps.a[l], 64 * c, m0, FULL(s));
                tc::tma_load_2d(base + s * WG_STAGE + BOX, &maps.b[l], 64 * c, 0, FULL(s));
            }
            // copies still in flight (only after a failed wait) land before the CTA exits
            for (uint32_t j = q > WG_RING ? q - WG_RING : 0; j < q; ++j)
                if (!tc::mbar_wait(FULL(j % WG_RING), (j / WG_RING) & 1, WAIT_LIMIT)) ok = false;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = tc::idesc_bf16_f32(128, n_cols);
            uint32_t q = 0;
            for (int c = c0; c < c1 && ok; c++, q++) {
                const uint32_t s = q % WG_RING;
                ok = tc::mbar_wait(FULL(s), (q / WG_RING) & 1, WAIT_LIMIT);
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t a = desc_lo(base + s * WG_STAGE), b = a + (BOX >> 4);
                if (q == 0)
                    mma_lo<false>(tmem, a, b, idesc);
                else
                    mma_lo<true>(tmem, a, b, idesc);
#pragma unroll
                for (int kk = 1; kk < 4; kk++) mma_lo<true>(tmem, a + 2 * kk, b + 2 * kk, idesc);
                tc::mma_commit(EMPTY(s));
            }
            // completes once every issued MMA has: the epilogue's signal, and the accumulator's
            tc::mma_commit(ACC);
            if (!tc::mbar_wait(ACC, 0, WAIT_LIMIT)) ok = false;
        }
    } else if (c1 > c0) {
        const int quarter = warp & 3, half = (warp - 2) >> 2, n = m0 + quarter * 32 + lane;
        ok = tc::mbar_wait_warp(ACC, 0, WAIT_LIMIT);
        tc::fence_after_sync();
        for (int col = 32 * half; col < n_cols && ok; col += 64) {
            float v[32];
            tc::tmem_ld32(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col, v);
            if (n < n_rows) {
                float *p = g.g[l] + (int64_t)n * n_cols + col;
#pragma unroll
                for (int i = 0; i < 32; i += 4)
                    if (col + i < n_cols)
                        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p + i),
                                     "f"(v[i]), "f"(v[i + 1]), "f"(v[i + 2]), "f"(v[i + 3])
                                     : "memory");
            }
        }
    }
    if (!ok && g.err) atomicExch(g.err, 1);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 1) tc::tmem_dealloc(tmem, 256);
}

} // namespace

bool fused_prepare(FusedMaps *maps, const void *const w3[N_LAYERS], const void *const wt[N_LAYERS])
{
    for (int l = 0; l < N_LAYERS; l++) {
        if (!tma::make_map(&maps->w[l], w3[l], (uint64_t)OUT_DIM[l], 3 * (uint64_t)IN_DIM[l],
                           3 * (uint64_t)IN_DIM[l], OUT_DIM[l]))
            return false;
        if (!tma::make_map(&maps->wt[l], wt[l], (uint64_t)IN_DIM[l], (uint64_t)OUT_DIM[l],
                           (uint64_t)OUT_DIM[l], IN_DIM[l]))
            return false;
    }
    const cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return cudaFuncSetAttribute(fused_kernel<false>, smem, SMEM) == cudaSuccess &&
           cudaFuncSetAttribute(fused_kernel<true>, smem, SMEM) == cudaSuccess &&
           cudaFuncSetAttribute(wgrad_kernel, smem, WG_SMEM) == cudaSuccess;
}

int fused_grid(int64_t n, int sm_count)
{
    const int64_t tiles = (n + TILE - 1) / TILE;
    return (int)(tiles < sm_count ? tiles : sm_count);
}

cudaError_t launch_fused(const FusedMaps &maps, const FusedArgs &a, int sm_count, cudaStream_t s)
{
    if (a.n <= 0) return cudaSuccess;
    fused_kernel<false><<<fused_grid(a.n, sm_count), THREADS, SMEM, s>>>(maps, a);
    return cudaGetLastError();
}

cudaError_t launch_fused_train(const FusedMaps &maps, const FusedArgs &a, int sm_count,
                               cudaStream_t s)
{
    fused_kernel<true><<<fused_grid(a.n, sm_count), THREADS, SMEM, s>>>(maps, a);
    return cudaGetLastError();
}

bool wgrad_prepare(WGradMaps *maps, const TrainArgs &t)
{
    for (int l = 0; l < N_LAYERS; l++)
        if (!tma::make_map(&maps->a[l], t.dzt[l], (uint64_t)OUT_DIM[l], (uint64_t)t.ld, (uint64_t)t.ld,
                           128) ||
            !tma::make_map(&maps->b[l], t.xt[l], (uint64_t)IN_DIM[l], (uint64_t)t.ld, (uint64_t)t.ld,
                           IN_DIM[l]))
            return false;
    return true;
}

cudaError_t launch_wgrad(const WGradMaps &maps, float *const g[N_LAYERS], int64_t ld, int *err,
                         int sm_count, cudaStream_t s)
{
    WGradArgs a;
    for (int l = 0; l < N_LAYERS; l++) a.g[l] = g[l];
    a.chunks = (int)(ld / 64);
    a.err = err;
    const int fill = sm_count / WG_TILES > 0 ? sm_count / WG_TILES : 1;
    const int splits = a.chunks < fill ? a.chunks : fill;
    wgrad_kernel<<<dim3(WG_TILES, splits), 64 + 32 * WG_EPI, WG_SMEM, s>>>(maps, a);
    return cudaGetLastError();
}

} // namespace sg
} // namespace gt
