// lbm_nn.cu -- the learned coarse-grid corrector: a 3-layer 3-D convolutional network
// (16 channels, 3x3x3 kernels, BF16 weights and activations, FP32 accumulation), its backward
// pass and Adam training, the restriction of fine fields onto the coarse grid, and the C-ABI
// entry points lbm_corrector_* / lbm_restrict.
//
// The paper has no learned component; its Sec. 3.4 shows that a 2x coarser grid keeps useful
// accuracy at ~14x less cost.  The corrector nudges the coarse velocity toward the fine solution
// restricted onto the coarse grid, every K coarse steps.
//
// GB300 design:
//   * Activations are channels-last BF16 on the coarse box padded by one zero cell on every side
//     (16 channels = 32 B per cell), so a 3x3x3 neighbourhood never needs a bounds test.
//   * Only 4^3 tiles that hold fluid, dilated by one tile, are evaluated (the rest of the box
//     stays zero): the receptive field of the three layers is 3 cells, so outputs at fluid cells
//     equal those of the dense network.
//   * Convolution = implicit GEMM on the 5th-generation tensor cores (k_conv_tc): tcgen05.mma
//     with the accumulator in tensor memory, operands staged in shared memory by TMA, a CTA per
//     8 x 16 x 1 slab (M = 128 cells, N = 16 output channels, K = 27 offsets x 16 input
//     channels).  The data-gradient is the same kernel with the flipped, transposed kernel and
//     a ReLU gate.  The weight-gradient is a GEMM over cells (K) whose M stacks the offsets along
//     x with the input channels (k_wgrad_tc, also tcgen05): the three x-shifted copies of each
//     halo row are transposed into shared memory so that every operand is a plain canonical
//     layout, and the per-CTA partial sums are added in a fixed order.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cmath>
#include <cstddef>
#include <cstring>
#include <string>
#include <vector>

#include "lbm_internal.h"

using namespace lbm;

namespace {

constexpr int CH = 16;
constexpr int NW = 27 * CH * CH;         // weights per layer
constexpr int NP = 3 * (NW + CH);        // parameters: W1, b1, W2, b2, W3, b3

struct Box {
    int nx, ny, nz;  // interior
    int px, py, pz;  // padded (n + 2)
};

__device__ __forceinline__ size_t pidx(const Box& b, int x, int y, int z)
{
    return ((size_t)(z + 1) * b.py + (size_t)(y + 1)) * b.px + (size_t)(x + 1);
}

// du = du_scale * clamp(O[0:3], -clip, clip) at the masked cells of the slabs, 0 at their other
// cells (three planes; the caller zeroes the rest of the box).  The clamp lets a NaN through
// (fminf/fmaxf would turn it into -clip): a network that has gone non-finite must make the
// corrected state non-finite, which the caller's fallback detects, not apply a full-size
// correction everywhere.
__device__ __forceinline__ float clamp_keep_nan(float o, float clip)
{
    return o > clip ? clip : (o < -clip ? -clip : o);
}

// ------------------------------------------------------------------------------ tcgen05 conv
// out[p][co] = act(sum_o sum_ci w[o][co][ci] in[p + o][ci] + bias[co]), zeroed where gate <= 0,
// as an implicit GEMM on the 5th-generation tensor cores.  A slab is 8 (x) x 16 (y) x 1 (z)
// cells: M = 128 rows (cell x + 8 y), N = 16 output channels, K = 27 offsets x 16 input
// channels, i.e. 27 tcgen05.mma (kind::f16, BF16 in, FP32 accumulator of 128 lanes x 16 columns
// in tensor memory) issued by one thread.  The CTAs (128 threads) are persistent and walk over
// slabs blockIdx.x, + gridDim.x, ...: the weights are staged once per CTA, the halo of the next
// slab is loaded into the other of two buffers, and two accumulators alternate, so the 27 MMAs
// of slab j run while the epilogue of slab j - 1 drains and the halo of slab j + 1 arrives.
//   * The slab's halo (10 x 18 x 3 cells) comes in by two TMA tile loads of the channels-last
//     padded activations (a 4-D tensor map, box 8 channels x 10 x 18 x 3), one per group of 8
//     channels, so shared memory holds two "planes" of 16 bytes per cell.  For offset o the A
//     operand is a K-major, non-swizzled canonical layout read straight out of those planes:
//     8-row core matrices are 8 consecutive cells along x (16 B apart), core matrices along M
//     are the 16 y rows (160 B apart), and the two K core matrices are the two planes.  No
//     gather, no copy: the 27 descriptors differ only in their start address.
//   * B (the 27 weight blocks, N x K = 16 x 16) is stored in global memory in the same canonical
//     layout (core matrix (n-group, k-group) at 128-byte steps; k_prepare writes it) and comes in
//     with the first halo by one bulk copy.
//   * The epilogue reads each row back with tcgen05.ld (warp w owns lanes 32w..32w+31), adds the
//     bias, applies ReLU and the gate, and writes 32 bytes per cell.
// Every wait (TMA, MMA completion) is bounded; on a timeout the CTA flags the error, waits for
// what it issued, frees its tensor memory and returns.
constexpr int SL_X = 8, SL_Y = 16;                      // slab = M = 128 cells
constexpr int HX = SL_X + 2, HY = SL_Y + 2, HZ = 3;     // halo
constexpr uint32_t PLANE_BYTES = HX * HY * HZ * 16;     // 8640: one TMA box
constexpr uint32_t PLANE_STRIDE = 8704;                 // 128-byte aligned plane step
constexpr uint32_t HALO_BYTES = 2 * PLANE_STRIDE;       // one halo buffer: two planes
constexpr uint32_t W_OFF = 2 * HALO_BYTES;              // weights after the two halo buffers
constexpr uint32_t W_BYTES = 27 * 512;                  // one layer's weights, BF16
constexpr uint32_t CONV_SMEM = W_OFF + W_BYTES;         // 48640 B
constexpr int CONV_CTAS_PER_SM = 4;
constexpr uint32_t CONV_COLS = 64;  // tensor-memory columns of a CTA
constexpr int TC_WAIT_LIMIT = 1 << 22;

// Programmatic dependent launch along a pass's chain of kernels (features, then convolutions, loss, weight
// gradients, update): a kernel sets up its barriers, tensor memory and weights while the one before it
// drains, and waits before it touches what the chain computes.  The features kernel is a plain launch,
// so everything enqueued before the pass (weights, masks, fields) is complete when any kernel of the
// chain starts.  What the chain computes is read with plain loads, not through the read-only path.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ float ld_f32(const float* p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_u32(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld_u128(const void* p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
template <class... P, class... A>
cudaError_t launch_pdl(void (*k)(P...), dim3 grid, int block, size_t smem, cudaStream_t s, A&&... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&c, k, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // reported here: a later launch that asks must not find it again
    return e;
}

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start address, leading (K) and stride (M/N) byte offsets,
// descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, M = 128, N = 16
constexpr uint32_t CONV_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((16u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t phase)
{
    for (int it = 0; it < TC_WAIT_LIMIT; ++it) {
        uint32_t done;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                     : "=r"(done)
                     : "r"(su32(bar)), "r"(phase)
                     : "memory");
        if (done) return true;
    }
    return false;
}

// Output of a convolution: BF16 activations (padded, channels-last), FP32 O[0:4] (compact float4
// per cell), or the velocity correction du = scale clamp(O[0:3]) at the cells of `mask` (0 at the
// slabs' other cells; three planes) -- the last layer of an inference with the output step fused.
enum ConvOut { OUT_BF16 = 0, OUT_F32 = 1, OUT_DU = 2 };
struct DuArgs {
    const uint8_t* mask;
    float scale, clip;
};

template <int OUT>
__global__ void __launch_bounds__(128)
    k_conv_tc(const __grid_constant__ CUtensorMap tin, const __nv_bfloat16* __restrict__ w, const float* __restrict__ bias,
              int relu, const __nv_bfloat16* gate, void* out, const int4* __restrict__ slabs, int n_slabs, Box b,
              unsigned int* err, DuArgs dua)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar_tma[2], bar_mma[2];
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = gridDim.x;
    const int J = (n_slabs - (int)blockIdx.x + G - 1) / G;  // slabs of this CTA (>= 1)
    pdl_trigger();
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bar_tma[k])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bar_mma[k])) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {  // two accumulators of 16 columns, at columns 0 and 32
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_base)),
                     "n"(CONV_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    __syncthreads();
    // halo of slab j into buffer j & 1: padded coordinates (x0, y0, z) .. + (9, 17, 2), channels
    // 0-7 and 8-15 (issued by thread 0)
    // (the weights, one bulk copy already in the shared-memory layout, count towards slab 0's barrier)
    auto load_weights = [&]() {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(&bar_tma[0])),
                     "r"(2u * PLANE_BYTES + W_BYTES)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                su32(smem + W_OFF)),
            "l"(w), "r"(W_BYTES), "r"(su32(&bar_tma[0]))
            : "memory");
    };
    auto load_halo = [&](int j) {
        const int4 sl = slabs[blockIdx.x + j * G];
        uint64_t* bar = &bar_tma[j & 1];
        unsigned char* dst = smem + (j & 1) * HALO_BYTES;
        if (j > 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)), "r"(2u * PLANE_BYTES)
                         : "memory");
#pragma unroll
        for (int c = 0; c < 2; ++c)
            asm volatile(
                "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
                "%4, %5}], [%6];" ::"r"(su32(dst + c * PLANE_STRIDE)),
                "l"(reinterpret_cast<uint64_t>(&tin)), "r"(8 * c), "r"(sl.x), "r"(sl.y), "r"(sl.z), "r"(su32(bar))
                : "memory");
    };
    if (tid == 0) load_weights();
    const uint32_t tbase = tmem_base;
    float bz[CH];
#pragma unroll
    for (int co = 0; co < CH; ++co) bz[co] = bias ? __ldg(bias + co) : 0.0f;
    pdl_wait();
    if (tid == 0) {
        load_halo(0);
        if (J > 1) load_halo(1);
    }
    // epilogue of slab j: accumulator j & 1 -> bias, ReLU, gate -> output
    auto epilogue = [&](int j) {
        const int4 sl = slabs[blockIdx.x + j * G];
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(tbase + 32u * (uint32_t)(j & 1) + ((uint32_t)(warp * 32) << 16)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        const int m = warp * 32 + lane;
        const int x = sl.x + (m & 7), y = sl.y + (m >> 3), z = sl.z;
        if (x < b.nx && y < b.ny) {
            float v[CH];
            const size_t pc = pidx(b, x, y, z);
            uint4 gw[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
            if (gate) {  // the gate's 16 channels of this cell, two 16-byte loads
                gw[0] = ld_u128(gate + pc * CH);
                gw[1] = ld_u128(gate + pc * CH + 8);
            }
            const uint32_t* g32 = reinterpret_cast<const uint32_t*>(gw);
#pragma unroll
            for (int co = 0; co < CH; ++co) {
                float t = __uint_as_float(r[co]) + bz[co];
                if (relu) t = fmaxf(t, 0.0f);
                const uint32_t gb = (co & 1) ? (g32[co >> 1] & 0xFFFF0000u) : (g32[co >> 1] << 16);
                if (gate && !(__uint_as_float(gb) > 0.0f)) t = 0.0f;
                v[co] = t;
            }
            const size_t c = ((size_t)z * b.ny + y) * b.nx + x;
            if (OUT == OUT_F32) {
                *reinterpret_cast<float4*>(static_cast<float*>(out) + c * 4) = make_float4(v[0], v[1], v[2], v[3]);
            } else if (OUT == OUT_DU) {
                const size_t n = (size_t)b.nx * b.ny * b.nz;
                const bool on = dua.mask[c] != 0;
                float* du = static_cast<float*>(out);
#pragma unroll
                for (int k = 0; k < 3; ++k) du[k * n + c] = on ? clamp_keep_nan(v[k], dua.clip) * dua.scale : 0.0f;
            } else {
                uint32_t pk[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
                    pk[k] = *reinterpret_cast<const uint32_t*>(&h);
                }
                uint4* dst = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(out) + pc * CH);
                dst[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                dst[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    };
    // give up: flag the error, wait (bounded) for the halo loads t0..t1 and the MMA groups
    // m0..m1 still in flight
    auto abandon = [&](int t0, int t1, int m0, int m1) {
        if (tid == 0) atomicOr(err, 1u);
        for (int j = t0; j <= t1 && j < J; ++j) tc_wait(&bar_tma[j & 1], (j >> 1) & 1);
        for (int j = m0 < 0 ? 0 : m0; j <= m1; ++j) tc_wait(&bar_mma[j & 1], (j >> 1) & 1);
    };
    bool ok = true;
    for (int j = 0; j < J; ++j) {
        // in flight here: halo loads j (and 1 when j = 0), MMA group j - 1
        if (!__syncthreads_and(tc_wait(&bar_tma[j & 1], (j >> 1) & 1))) {  // one decision for the CTA
            abandon(j, j == 0 ? 1 : j, j - 1, j - 1);
            ok = false;
            break;
        }
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // a descriptor's start field is the address / 16 (no carry out of it below 256 KB): the
            // 27 offsets' descriptors are the buffer's plus constants
            const uint64_t a0 = smem_desc(su32(smem + (j & 1) * HALO_BYTES), PLANE_STRIDE, HX * 16);
            const uint64_t w0 = smem_desc(su32(smem + W_OFF), 128, 256);
            const uint32_t d = tbase + 32u * (uint32_t)(j & 1);
#pragma unroll
            for (int o = 0; o < 27; ++o) {
                const int ox = o % 3, oy = (o / 3) % 3, oz = o / 9;
                const uint64_t ad = a0 + (uint64_t)((oz * HY + oy) * HX + ox);
                const uint64_t bd = w0 + (uint64_t)(32 * o);
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, "
                    "p;\n}\n" ::"r"(d),
                    "l"(ad), "l"(bd), "r"(CONV_IDESC), "r"((uint32_t)(o > 0))
                    : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             su32(&bar_mma[j & 1]))
                         : "memory");
        }
        if (j >= 1) {
            const int p = j - 1;
            // in flight here: MMA groups j - 1 and j, no halo load
            if (!__syncthreads_and(tc_wait(&bar_mma[p & 1], (p >> 1) & 1))) {
                abandon(J, J - 1, p, j);
                ok = false;
                break;
            }
            epilogue(p);
            __syncthreads();  // accumulator p & 1 read; halo buffer p & 1 consumed by MMA p
            if (tid == 0 && j + 1 < J) load_halo(j + 1);
        }
    }
    if (ok) {
        const int p = J - 1;
        if (__syncthreads_and(tc_wait(&bar_mma[p & 1], (p >> 1) & 1))) {
            epilogue(p);
        } else if (tid == 0) {
            atomicOr(err, 1u);
        }
    }
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "n"(CONV_COLS) : "memory");
}

// Partial weight gradient of this CTA's slabs on the 5th-generation tensor cores:
// part[blockIdx.x] = (dW[o][co][ci] = sum_p dy[p][co] x[p + o][ci], db[co] = sum_p dy[p][co]) over
// the cells p of slabs blockIdx.x, + gridDim.x, ...  The sums over the CTAs are taken in a fixed
// order by k_wgrad_reduce, so that a training run is reproducible bit for bit.
//   GEMM per pair (dy, dz) of offsets along y and z: D[(s, ci)][co] = sum_k A[(s, ci)][k] B[co][k]
// with k running over the slab's cells (K = 16 per MMA: two x rows of 8 cells), A[(s, ci)][k] =
// x[cell(k) + (s - 1, dy, dz)][ci] and B[co][k] = dy[cell(k)][co]; rows s = 0, 1, 2 are the three
// offsets along x.  Both operands are K-major canonical layouts (8 x 16 B core matrices, no
// swizzle) built in shared memory: for every halo row (y, z) the 8 cells that start at x0 - 1,
// x0 and x0 + 1 are stored transposed, channel by channel ([ci][8 cells], 256 B each), one after
// the other, so the M core matrices (s, ci / 8) of one offset pair lie 128 B apart and the next
// 8 cells along K (the next x row) 768 B further.  An MMA has M = 128: rows s = 3..7 read the
// following halo rows and are discarded.  The nine accumulators (16 columns each) stay in tensor
// memory over all the CTA's slabs; two staging buffers let the threads transpose slab j + 1 while
// the 72 MMAs of slab j run.  Every wait is bounded; on a timeout the CTA flags `err`, waits for
// what it issued, frees its tensor memory and returns.
constexpr int WG_CTAS = 304;                           // weight-gradient CTAs (2 per SM): the partial buffer's depth
constexpr int WG_HROWS = HY * HZ;                      // 54 halo rows (y, z) of a slab
constexpr uint32_t WG_ROW = 3 * 256;                   // one halo row: three shifted copies
constexpr uint32_t WG_A = (WG_HROWS + 2) * WG_ROW;     // + 2 rows read only by the discarded M rows
constexpr uint32_t WG_B = SL_Y * 256;                  // dy of the slab: 16 x rows of [co][8 cells]
constexpr uint32_t WG_BUF = WG_A + WG_B;               // 47104
constexpr uint32_t WG_SMEM = 2 * WG_BUF;               // 94208
constexpr uint32_t WG_COLS = 256;                      // tensor-memory columns of a CTA
// furthest byte an MMA reads in a buffer: A of the last offset pair's last K step
static_assert((uint32_t)(((HZ - 1) * HY + (SL_Y - 2) + 2) * WG_ROW) + WG_ROW + 15 * 128 + 128 <= WG_A,
              "weight-gradient A operand reads past its buffer");
static_assert((SL_Y - 2) * 256 + 256 + 128 + 128 <= (int)WG_B, "weight-gradient B operand reads past its buffer");

// A convolution lets the next kernel start before its own CTAs have allocated their tensor memory, and the next one's
// CTAs hold theirs while they wait for it.  An allocation must therefore never need columns of a CTA that waits:
// whatever set of these CTAs fits on an SM by shared memory (228 KB, 1 KB of it reserved per CTA) also fits by columns.
constexpr bool tmem_fits()
{
    for (uint32_t w = 0; w <= 2; ++w)
        for (uint32_t c = 0; c <= 8; ++c)
            if (w * (WG_SMEM + 1024) + c * (CONV_SMEM + 1024) <= 228u * 1024 && w * WG_COLS + c * CONV_COLS > 512) return false;
    return 3 * (WG_SMEM + 1024) > 228u * 1024;
}
static_assert(tmem_fits(), "CTAs of overlapping kernels could wait for one another's tensor memory");

// The three layers run in one launch (blockIdx.y: the layer), so one layer's tail fills with the next
// one's CTAs: the three weight gradients depend on nothing but the back-propagated gradients.
struct WgradArgs {
    const __nv_bfloat16* dy[3];
    const __nv_bfloat16* x[3];
};
__global__ void __launch_bounds__(128)
    k_wgrad_tc(WgradArgs in, const int4* __restrict__ slabs, int n_slabs, Box b, float* part_all, unsigned int* err)
{
    const __nv_bfloat16 *dy = in.dy[blockIdx.y], *x = in.x[blockIdx.y];
    float* part = part_all + (size_t)blockIdx.y * WG_CTAS * (NW + CH);
    pdl_trigger();
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar_mma[2];
    __shared__ uint32_t tmem_base;
    __shared__ float sdb[128][4];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = gridDim.x;
    const int J = (n_slabs - (int)blockIdx.x + G - 1) / G;  // slabs of this CTA (>= 1)
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bar_mma[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bar_mma[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {  // nine accumulators of 16 columns at columns 0, 16, ..., 128
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_base)),
                     "n"(WG_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    __syncthreads();
    pdl_wait();
    const uint32_t tbase = tmem_base;
    const uint32_t* x32 = reinterpret_cast<const uint32_t*>(x);
    const uint32_t* dy32 = reinterpret_cast<const uint32_t*>(dy);
    // lane l holds, of an 8-cell x 8-channel block, cell l / 4 and channels 2 (l % 4), + 1 (one
    // 32-bit word of the channels-last data); stmatrix .trans writes the block channel by channel
    // (16 B rows of 8 cells), the canonical core-matrix rows
    const int ci8 = lane >> 2, cpw = lane & 3;
    float db[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};  // bias gradient of channels 8 g + 2 cpw + h
    // slab j's operands into buffer j & 1: warp w transposes halo rows w, w + 4, ... and x rows
    // w, w + 4, ... of dy.  Every load of the slab is issued before the first store, so the
    // warp waits for one memory latency per slab, not one per row.
    constexpr int RW = (WG_HROWS + 3) / 4;  // halo rows per warp (14; warps 2 and 3 have 13)
    auto stage = [&](int j) {
        const int4 sl = slabs[blockIdx.x + j * G];
        const uint32_t A = su32(smem + (j & 1) * WG_BUF), B = A + WG_A;
        uint32_t v[RW][3][2], u[SL_Y / 4][2];
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            const int r = warp + 4 * i;
            const int Y = sl.y + r % HY, Z = sl.z + r / HY;  // padded coordinates
            const bool row_ok = r < WG_HROWS && Y < b.py && Z < b.pz;
#pragma unroll
            for (int sx = 0; sx < 3; ++sx) {
                const int X = sl.x + ci8 + sx;
                const bool ok = row_ok && X < b.px;
                const size_t c8 = ok ? (((size_t)Z * b.py + Y) * b.px + X) * (CH / 2) : 0;
                v[i][sx][0] = ok ? ld_u32(x32 + c8 + cpw) : 0u;
                v[i][sx][1] = ok ? ld_u32(x32 + c8 + 4 + cpw) : 0u;
            }
        }
#pragma unroll
        for (int i = 0; i < SL_Y / 4; ++i) {
            const int X = sl.x + ci8, Y = sl.y + warp + 4 * i;
            const bool ok = X < b.nx && Y < b.ny;
            const size_t c8 = ok ? pidx(b, X, Y, sl.z) * (CH / 2) : 0;
#pragma unroll
            for (int g = 0; g < 2; ++g) u[i][g] = ok ? ld_u32(dy32 + c8 + 4 * g + cpw) : 0u;
        }
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            const int r = warp + 4 * i;
            if (r >= WG_HROWS) break;  // warp-uniform
            // blocks (sx, g) at row + 256 sx + 128 g: lane l gives the address of row l % 8 of
            // block l / 8 (x4: sx = 0, 1) and of block 4 + l / 8 (x2: sx = 2, lanes 0-15)
            const uint32_t row = A + (uint32_t)r * WG_ROW + 16u * (uint32_t)lane;
            asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(row),
                         "r"(v[i][0][0]), "r"(v[i][0][1]), "r"(v[i][1][0]), "r"(v[i][1][1])
                         : "memory");
            asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1, %2};" ::"r"(row + 512u * (lane < 16)),
                         "r"(v[i][2][0]), "r"(v[i][2][1])
                         : "memory");
        }
#pragma unroll
        for (int i = 0; i < SL_Y / 4; ++i) {
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                db[g][0] += __uint_as_float(u[i][g] << 16);
                db[g][1] += __uint_as_float(u[i][g] & 0xFFFF0000u);
            }
            const uint32_t row = B + (uint32_t)(warp + 4 * i) * 256u + 16u * (uint32_t)(lane & 15);
            asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1, %2};" ::"r"(row), "r"(u[i][0]),
                         "r"(u[i][1])
                         : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the tensor cores
    };
    // the 72 MMAs of slab j (thread 0); a descriptor's start field is the address / 16 (no carry
    // out of it below 256 KB), so the operands' descriptors are the buffer's plus constants
    auto issue = [&](int j) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t A = su32(smem + (j & 1) * WG_BUF), B = A + WG_A;
        const uint64_t a0 = smem_desc(A, WG_ROW, 128), b0 = smem_desc(B, 256, 128);
        const uint32_t acc = j > 0 ? 1u : 0u;
#pragma unroll
        for (int a = 0; a < 9; ++a) {
#pragma unroll
            for (int k = 0; k < SL_Y / 2; ++k) {
                const uint64_t ad = a0 + (uint64_t)(((a / 3) * HY + 2 * k + a % 3) * (int)(WG_ROW >> 4));
                const uint64_t bd = b0 + (uint64_t)(k * (512 >> 4));
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, "
                    "p;\n}\n" ::"r"(tbase + 16u * (uint32_t)a),
                    "l"(ad), "l"(bd), "r"(CONV_IDESC), "r"(k > 0 ? 1u : acc)
                    : "memory");
            }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         su32(&bar_mma[j & 1]))
                     : "memory");
    };
    bool ok = true;
    int issued = 0;  // MMA groups issued (the same count in every thread)
    for (int j = 0; j < J; ++j) {
        if (j >= 2) {  // buffer j & 1 is free once the MMAs of slab j - 2 are done
            const int p = j - 2;
            if (!__syncthreads_and(tc_wait(&bar_mma[p & 1], (p >> 1) & 1))) {
                ok = false;
                break;
            }
        }
        stage(j);
        __syncthreads();
        if (tid == 0) issue(j);
        ++issued;
    }
    // the last group's completion covers every MMA issued before it
    if (ok && !__syncthreads_and(tc_wait(&bar_mma[(J - 1) & 1], ((J - 1) >> 1) & 1))) ok = false;
    if (!ok) {
        if (tid == 0) atomicOr(err, 1u);
        // bounded waits for the groups that may still be in flight, so that the tensor memory is
        // idle when it is freed
        for (int p = issued >= 2 ? issued - 2 : 0; p < issued; ++p) tc_wait(&bar_mma[p & 1], (p >> 1) & 1);
    } else {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float* dW = part + (size_t)blockIdx.x * (NW + CH);
        if (warp < 2) {
            const int m = warp * 32 + lane, sx = m >> 4, ci = m & 15;
#pragma unroll 1
            for (int a = 0; a < 9; ++a) {
                uint32_t r[16];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                    "[%16];"
                    : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                      "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                      "=r"(r[15])
                    : "r"(tbase + 16u * (uint32_t)a + ((uint32_t)(warp * 32) << 16)));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (sx < 3) {
                    const int o = sx + 3 * (a % 3) + 9 * (a / 3);
#pragma unroll
                    for (int co = 0; co < CH; ++co) dW[(o * CH + co) * CH + ci] = __uint_as_float(r[co]);
                }
            }
        }
        sdb[tid][0] = db[0][0];
        sdb[tid][1] = db[0][1];
        sdb[tid][2] = db[1][0];
        sdb[tid][3] = db[1][1];
        __syncthreads();
        if (tid < CH) {  // channel 8 g + 2 c + h: the threads with tid' % 4 = c, in increasing tid'
            const int g = tid >> 3, c = (tid >> 1) & 3, h = tid & 1;
            float acc = 0.0f;
            for (int t = c; t < 128; t += 4) acc += sdb[t][2 * g + h];
            dW[NW + tid] = acc;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "n"(WG_COLS) : "memory");
}

// Position of weight (o, co, ci) in a layer's BF16 block, which is the convolution's shared-memory
// layout (copied in as is): block o of 512 B holds the core matrices (co / 8, ci / 8) at 128-byte
// steps, row co % 8 at 16-byte steps, ci % 8 within the row.
__device__ __forceinline__ int w_layout(int o, int co, int ci)
{
    return o * 256 + (2 * (co >> 3) + (ci >> 3)) * 64 + (co & 7) * 8 + (ci & 7);
}

// BF16 forward weight r of layer l and its place in the data-gradient kernel
// wt[o'][ci][co] = w[26 - o'][co][ci] (flipped offsets, transposed channels), both in w_layout.
__device__ __forceinline__ void put_weight(int l, int r, float v, __nv_bfloat16* wb, __nv_bfloat16* wt)
{
    const int o = r / (CH * CH), co = (r / CH) % CH, ci = r % CH;
    wb[l * NW + w_layout(o, co, ci)] = __float2bfloat16_rn(v);
    wt[l * NW + w_layout(26 - o, ci, co)] = __float2bfloat16_rn(v);
}

// Adam's update of one parameter
struct Adam {
    float *p, *m, *v;
    __nv_bfloat16 *wb, *wt;
    float lr, b1, b2, eps, bc1, bc2;
};

// grad[l][k] = sum over the n_part partial gradients of layer l (weights and biases, NW + CH values), in
// a fixed order: a CTA takes 32 consecutive k; its thread (c, k) adds the partials p = c, c + 8, ...
// in increasing p, and the eight chunk sums are then added in increasing c.  In a training step the
// thread that has the sum also takes the parameter's Adam step and writes its BF16 weights.
constexpr int WR_K = 32, WR_C = 8;
template <bool ADAM>
__global__ void __launch_bounds__(WR_K * WR_C)
    k_wgrad_reduce(const float* part_all, int n_part, float* grad, Adam ad)
{
    __shared__ float cs[WR_C][WR_K];
    const int kk = threadIdx.x % WR_K, c = threadIdx.x / WR_K, l = blockIdx.y;
    const int k = blockIdx.x * WR_K + kk;
    const float* part = part_all + (size_t)l * WG_CTAS * (NW + CH);
    pdl_wait();
    float s = 0.0f;
    if (k < NW + CH) {
#pragma unroll 8
        for (int p = c; p < n_part; p += WR_C) s += ld_f32(part + (size_t)p * (NW + CH) + k);
    }
    cs[c][kk] = s;
    __syncthreads();
    if (c == 0 && k < NW + CH) {
        float t = cs[0][kk];
#pragma unroll
        for (int q = 1; q < WR_C; ++q) t += cs[q][kk];
        const int i = l * (NW + CH) + k;
        grad[i] = t;
        if (ADAM) {
            const float mi = ad.b1 * ad.m[i] + (1.0f - ad.b1) * t;
            const float vi = ad.b2 * ad.v[i] + (1.0f - ad.b2) * t * t;
            const float pi = ad.p[i] - ad.lr * (mi / ad.bc1) / (sqrtf(vi / ad.bc2) + ad.eps);
            ad.m[i] = mi;
            ad.v[i] = vi;
            ad.p[i] = pi;
            if (k < NW) put_weight(l, k, pi, ad.wb, ad.wt);
        }
    }
}

// The elementwise kernels of the corrector run over the slabs of the convolutions (one CTA of
// 128 threads per 8 x 16 x 1 slab), which cover every cell a call's masks can select (they lie
// inside the creation mask) -- a tenth of the coarse box or less; the other cells of the padded
// activations and of the output gradient stay zero from creation.
__device__ __forceinline__ bool slab_cell(const int4* slabs, const Box& b, int& x, int& y, int& z, int64_t& c)
{
    const int4 sl = slabs[blockIdx.x];
    x = sl.x + (int)(threadIdx.x & 7u);
    y = sl.y + (int)(threadIdx.x >> 3);
    z = sl.z;
    c = ((int64_t)z * b.ny + y) * b.nx + x;
    return x < b.nx && y < b.ny;
}

// Input features on the padded box: u / u_scale (3), (rho - 1) / rho_scale, fluid mask, zeros.  On the way:
// the caller's correction box is zeroed (zero, n_zero values; the slabs' cells are written later by the
// last convolution), and the cells of a training step's output mask are counted.
__global__ void __launch_bounds__(128) k_features(const float* __restrict__ rho, const float* __restrict__ u,
                                                  const uint8_t* __restrict__ mask, Box b, float inv_us, float inv_rs,
                                                  __nv_bfloat16* __restrict__ x0, const int4* __restrict__ slabs,
                                                  float* __restrict__ zero, int64_t n_zero,
                                                  const uint8_t* __restrict__ out_mask, unsigned long long* count)
{
    pdl_trigger();
    int x, y, z;
    int64_t c;
    const bool in = slab_cell(slabs, b, x, y, z, c);
    if (zero) {
        const int64_t t = (int64_t)blockIdx.x * 128 + threadIdx.x, stride = (int64_t)gridDim.x * 128;
        if ((reinterpret_cast<uintptr_t>(zero) & 15u) == 0) {  // n_zero is a multiple of 4
            for (int64_t k = t; k < n_zero / 4; k += stride) reinterpret_cast<float4*>(zero)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            for (int64_t k = t; k < n_zero; k += stride) zero[k] = 0.0f;
        }
    }
    if (count) {
        const unsigned int ballot = __ballot_sync(0xffffffffu, in && out_mask[c] != 0);
        if ((threadIdx.x & 31) == 0 && ballot) atomicAdd(count, (unsigned long long)__popc(ballot));
    }
    if (!in) return;
    const int64_t n = (int64_t)b.nx * b.ny * b.nz;
    const float fl = mask[c] ? 1.0f : 0.0f;
    __nv_bfloat16 v[CH];
    v[0] = __float2bfloat16_rn(u[c] * inv_us * fl);
    v[1] = __float2bfloat16_rn(u[n + c] * inv_us * fl);
    v[2] = __float2bfloat16_rn(u[2 * n + c] * inv_us * fl);
    v[3] = __float2bfloat16_rn((rho[c] - 1.0f) * inv_rs * fl);
    v[4] = __float2bfloat16_rn(fl);
#pragma unroll
    for (int k = 5; k < CH; ++k) v[k] = __float2bfloat16_rn(0.0f);
    uint4* dst = reinterpret_cast<uint4*>(x0 + pidx(b, x, y, z) * CH);
    dst[0] = *reinterpret_cast<uint4*>(&v[0]);
    dst[1] = *reinterpret_cast<uint4*>(&v[8]);
}

// Loss = mean over fluid cells and components of (O - T)^2, T = (u_target - u) / du_scale;
// dO = 2 (O - T) / N at fluid cells (BF16, padded, channels 0..2).
__global__ void __launch_bounds__(128) k_loss(const float* o4, const float* __restrict__ u,
                                              const float* __restrict__ ut, const uint8_t* __restrict__ mask, Box b,
                                              float inv_du, const volatile unsigned long long* count,
                                              __nv_bfloat16* dO, double* loss, const int4* __restrict__ slabs)
{
    __shared__ double sh[4];
    pdl_trigger();
    pdl_wait();
    const unsigned long long cells = *count;
    const float two_over_n = cells ? 2.0f / (3.0f * (float)cells) : 0.0f;
    const int64_t n = (int64_t)b.nx * b.ny * b.nz;
    int x, y, z;
    int64_t c;
    double part = 0.0;
    if (slab_cell(slabs, b, x, y, z, c)) {
        // every slab cell is written (zero off the mask), so that a mask differing from the
        // previous call's leaves no stale gradient behind
        __nv_bfloat16* d = dO + pidx(b, x, y, z) * CH;
        const bool on = mask[c] != 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float r = 0.0f;
            if (on) {
                r = ld_f32(o4 + c * 4 + k) - (ut[k * n + c] - u[k * n + c]) * inv_du;
                part += (double)r * r;
            }
            d[k] = __float2bfloat16_rn(two_over_n * r);
        }
    }
    for (int off = 16; off > 0; off >>= 1) part += __shfl_down_sync(0xffffffffu, part, off);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(loss, (sh[0] + sh[1]) + (sh[2] + sh[3]));
}

// BF16 weights of all layers from the master parameters (at creation and after set_params)
__global__ void k_prepare(const float* __restrict__ master, __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * NW) return;
    put_weight(i / NW, i % NW, master[(i / NW) * (NW + CH) + i % NW], wb, wt);
}

// coarse (X,Y,Z) = mean of rho and u over the fluid fine children (2X+a, 2Y+b, 2Z+c); 0 if none.  A thread
// takes W consecutive coarse cells of a row: with W = 4 the mask comes as four 8-byte words, most of
// which are 0 (a vessel fills about 2% of its box), and the four planes go out as 16-byte stores.  WIDE: the
// fields of eight fine cells in a row come as two 16-byte words each, wherever one of them is fluid (one sector,
// which a single cell would fetch too); else the fluid children one by one.  The sum runs in the order z, y, x
// in every form.  What bounds it is memory traffic; us at 256^3 -> 128^3, one cell a thread / four / four and wide:
// vessel 24.8 / 11.1 / 10.3, one cell in fifty 39 / 54 / 37, all cells 52 / 99 / 52 (319 MB: 6.2 TB/s).
template <int W, bool WIDE>
__global__ void __launch_bounds__(256)
    k_restrict(const float* __restrict__ frho, const float* __restrict__ fu, const uint8_t* __restrict__ fmask, int fnx,
               int fny, int fnz, float* __restrict__ crho, float* __restrict__ cu)
{
    const int cnx = fnx / 2, cny = fny / 2, cnz = fnz / 2;
    const int64_t cn = (int64_t)cnx * cny * cnz, fn = (int64_t)fnx * fny * fnz;
    const int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * W;
    if (c >= cn) return;
    const uint32_t row = (uint32_t)(c / cnx);
    const int X = (int)(c - (int64_t)row * cnx), Y = (int)(row % (uint32_t)cny), Z = (int)(row / (uint32_t)cny);
    uint8_t m[4][2 * W];
    int64_t at[4];
    bool any[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        at[r] = 2 * X + (int64_t)fnx * ((2 * Y + (r & 1)) + (int64_t)fny * (2 * Z + (r >> 1)));
        if constexpr (W == 4) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(fmask + at[r]));
            memcpy(m[r], &v, 8);
            any[r] = (v.x | v.y) != 0;
        } else {
            any[r] = false;
#pragma unroll
            for (int x = 0; x < 2 * W; ++x) {
                m[r][x] = fmask[at[r] + x];
                any[r] = any[r] || m[r][x];
            }
        }
    }
    float o[4][W] = {};
    int k[W] = {};
    if constexpr (WIDE) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (!any[r]) continue;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4* f = reinterpret_cast<const float4*>((q ? fu + (q - 1) * fn : frho) + at[r]);
                const float4 a = __ldg(f), b = __ldg(f + 1);
                const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                for (int x = 0; x < 8; ++x)
                    if (m[r][x]) o[q][x / 2] += v[x];
            }
#pragma unroll
            for (int x = 0; x < 8; ++x) k[x / 2] += m[r][x] != 0;
        }
    } else if (any[0] || any[1] || any[2] || any[3]) {
#pragma unroll
        for (int w = 0; w < W; ++w)
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    if (!m[r][2 * w + x]) continue;
                    const int64_t f = at[r] + 2 * w + x;
                    ++k[w];
                    o[0][w] += frho[f];
                    o[1][w] += fu[f];
                    o[2][w] += fu[fn + f];
                    o[3][w] += fu[2 * fn + f];
                }
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const float inv = k[w] ? 1.0f / (float)k[w] : 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q][w] *= inv;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float* dst = q ? cu + (q - 1) * cn + c : crho + c;
        if constexpr (W == 4) *reinterpret_cast<float4*>(dst) = make_float4(o[q][0], o[q][1], o[q][2], o[q][3]);
        else dst[0] = o[q][0];
    }
}

int blocks(int64_t n, int t) { return (int)((n + t - 1) / t); }

// 4-D tensor map over a channels-last padded activation buffer [pz][py][px][16] (BF16) whose
// box is one slab halo of one 8-channel group: 8 channels x 10 x 18 x 3 cells.
cudaError_t encode_halo_map(CUtensorMap* tm, const void* base, const Box& b)
{
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static Encode encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q{};
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess || !fn || q != cudaDriverEntryPointSuccess) return e != cudaSuccess ? e : cudaErrorNotSupported;
        encode = reinterpret_cast<Encode>(fn);
    }
    const cuuint64_t dims[4] = {(cuuint64_t)CH, (cuuint64_t)b.px, (cuuint64_t)b.py, (cuuint64_t)b.pz};
    const cuuint64_t strides[3] = {(cuuint64_t)CH * 2, (cuuint64_t)b.px * CH * 2, (cuuint64_t)b.px * b.py * CH * 2};
    const cuuint32_t box[4] = {8, (cuuint32_t)HX, (cuuint32_t)HY, (cuuint32_t)HZ};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

namespace lbm {
// host-side helpers shared with lbm_domain.cu
lbm_status nn_fail(lbm_status s, const std::string& msg)
{
    set_last_error(msg.c_str());
    return s;
}
}  // namespace lbm

struct lbm_corrector {
    Box box{};
    int64_t n_cells = 0, n_fluid = 0, n_tiles = 0;
    float u_scale = 0.05f, rho_scale = 0.01f, du_scale = 0.005f, clip = 2.0f;
    cudaStream_t stream = nullptr;
    lbm_alloc_fn alloc = nullptr;
    lbm_free_fn release = nullptr;
    void* ctx = nullptr;
    std::vector<void*> owned;
    uint8_t* mask = nullptr;
    int4* slabs = nullptr;   // 8 x 16 x 1 slabs covering the 4^3 tiles with fluid, dilated by one tile
    int64_t n_slabs = 0;
    // what a training pass reports, read back in one copy: the loss sum, the cells it runs over, and the
    // error word set by a CTA whose bounded wait gave up
    struct Report {
        double loss;
        unsigned long long count;
        unsigned int err;
    };
    Report* report = nullptr;    // device
    Report* h_report = nullptr;  // pinned
    cudaEvent_t ev = nullptr;     // orders the corrector's stream and a domain's stream (apply)
    CUtensorMap tmaps[5];         // halo maps of x0, y1, y2, dO, dy2 (the convolutions' inputs)
    const void* tmap_of[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    __nv_bfloat16 *x0 = nullptr, *y1 = nullptr, *y2 = nullptr, *dO = nullptr, *dy = nullptr, *dy2 = nullptr;
    float* o4 = nullptr;
    float *rho = nullptr, *u = nullptr, *du = nullptr;  // staging on the coarse box
    float *master = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    float* wpart = nullptr;  // [3][WG_CTAS][NW + CH] partial weight gradients of the layers
    __nv_bfloat16 *wb = nullptr, *wt = nullptr;
    int64_t adam_t = 0;
    int sms = 0;  // SMs of the device the corrector was created on
    uint64_t export_serial = 0;  // the domain whose zeros rho, u hold outside its fluid cells (0: none)

    void* dev(size_t bytes)
    {
        bytes = (bytes + 255) & ~(size_t)255;
        void* p = nullptr;
        if (alloc) p = alloc(bytes, ctx);
        else if (cudaMalloc(&p, bytes) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        if (p) owned.push_back(p);
        return p;
    }
    void release_all()
    {
        if (ev) cudaEventDestroy(ev);
        ev = nullptr;
        if (h_report) cudaFreeHost(h_report);
        h_report = nullptr;
        for (void* p : owned) {
            if (release) release(p, ctx);
            else if (!alloc) cudaFree(p);
        }
        owned.clear();
    }
    float* wmaster(int l) { return master + (size_t)l * (NW + CH); }
    float* bmaster(int l) { return master + (size_t)l * (NW + CH) + NW; }

    cudaError_t conv(const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias, int relu,
                     const __nv_bfloat16* gate, void* out, int mode, DuArgs dua = DuArgs{nullptr, 0.0f, 0.0f})
    {
        if (n_slabs == 0) return cudaSuccess;
        int t = 0;
        while (t < 5 && tmap_of[t] != in) ++t;
        if (t == 5) return cudaErrorInvalidValue;
        const int grid = (int)std::min<int64_t>(n_slabs, (int64_t)sms * CONV_CTAS_PER_SM);
        auto k = mode == OUT_F32 ? k_conv_tc<OUT_F32> : mode == OUT_DU ? k_conv_tc<OUT_DU> : k_conv_tc<OUT_BF16>;
        return launch_pdl(k, dim3((unsigned)grid), 128, CONV_SMEM, stream, tmaps[t], w, bias, relu, gate, out, slabs,
                          (int)n_slabs, box, &report->err, dua);
    }
    // enqueues the copy of the report, waits, and gives the mean loss; TIMEOUT if a CTA gave up
    lbm_status finish(cudaError_t e, const char* what, double* loss)
    {
        if (e == cudaSuccess) e = cudaMemcpyAsync(h_report, report, sizeof(Report), cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return nn_fail(LBM_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
        if (h_report->err) {
            cudaMemset(&report->err, 0, sizeof(unsigned int));
            return nn_fail(LBM_ERR_TIMEOUT, "a convolution gave up waiting for its copies or MMAs");
        }
        *loss = h_report->count ? h_report->loss / (3.0 * (double)h_report->count) : 0.0;
        return LBM_OK;
    }
    // Whether the features kernel, one CTA a slab, clears the correction box on its way, which saves a launch (us a
    // forward pass: 128^3 vessel 45.4 -> 37.1, 256^3 vessel 113.1 -> 109.4).  With few slabs in a large box, or words
    // of 4 bytes in one, a clear by itself is faster: 256^3 with 24 slabs 45.5 us, 112.3 in the kernel; with 72, 46.0 and
    // 58.0; with 216 (78 k cells a slab), 51.8 and 51.4; 256^3 vessel off the 16-byte boundary 111.1 and 130.6.
    bool features_clear(const float* du) const
    {
        return n_cells <= ((int64_t)1 << 17) * n_slabs &&
               (reinterpret_cast<uintptr_t>(du) % 16 == 0 || sizeof(float) * 3 * n_cells <= ((size_t)32 << 20));
    }
    // the network on the slabs: O into o4 (du == nullptr), or, for an inference, the correction
    // du = scale clamp(O[0:3]) at the cells of out_mask straight from the last layer (zero_du: the rest
    // of the caller's box is zeroed).  A training pass counts the cells of out_mask.
    cudaError_t forward(const uint8_t* cmask, const float* r, const float* uu, float* du, const uint8_t* out_mask,
                        float scale, bool zero_du)
    {
        cudaError_t e = cudaSuccess;
        if (zero_du && !features_clear(du)) {
            e = cudaMemsetAsync(du, 0, sizeof(float) * 3 * n_cells, stream);
            zero_du = false;
        }
        if (n_slabs == 0 || e != cudaSuccess) return e;
        k_features<<<(unsigned)n_slabs, 128, 0, stream>>>(r, uu, cmask ? cmask : mask, box, 1.0f / u_scale,
                                                          1.0f / rho_scale, x0, slabs, zero_du ? du : nullptr,
                                                          3 * n_cells, out_mask, du ? nullptr : &report->count);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = conv(x0, wb, bmaster(0), 1, nullptr, y1, OUT_BF16);
        if (e == cudaSuccess) e = conv(y1, wb + NW, bmaster(1), 1, nullptr, y2, OUT_BF16);
        if (e == cudaSuccess && !du) e = conv(y2, wb + 2 * NW, bmaster(2), 0, nullptr, o4, OUT_F32);
        if (e == cudaSuccess && du) e = conv(y2, wb + 2 * NW, bmaster(2), 0, nullptr, du, OUT_DU, DuArgs{out_mask, scale, clip});
        return e;
    }
    // forward pass, loss and gradients into `grad` (FP32, parameter layout), the report, and, with `ad`, an
    // Adam step.  Convolutions first, then the three weight gradients in one launch and their sums in
    // another: 9 kernels and one clear, against 17 and 3 with a launch per layer and per elementwise step.
    cudaError_t train(const uint8_t* cmask, const uint8_t* mk, const float* r, const float* uu, const float* ut, const Adam* ad)
    {
        cudaError_t e = cudaMemsetAsync(report, 0, offsetof(Report, err), stream);
        if (e == cudaSuccess) e = forward(cmask, r, uu, nullptr, mk, 0.0f, false);
        if (e != cudaSuccess) return e;
        if (n_slabs == 0) {  // no cell: zero gradients, and Adam's moments decay
            e = cudaMemsetAsync(wpart, 0, sizeof(float) * 3 * (size_t)WG_CTAS * (NW + CH), stream);
        } else {
            e = launch_pdl(k_loss, dim3((unsigned)n_slabs), 128, 0, stream, o4, uu, ut, mk, box, 1.0f / du_scale, &report->count,
                           dO, &report->loss, slabs);
            // dz2 = W3^T dO gated by y2 > 0, dz1 = W2^T dz2 gated by y1 > 0
            if (e == cudaSuccess) e = conv(dO, wt + 2 * NW, nullptr, 0, y2, dy2, OUT_BF16);
            if (e == cudaSuccess) e = conv(dy2, wt + NW, nullptr, 0, y1, dy, OUT_BF16);
        }
        const int wg = (int)std::min<int64_t>(std::max<int64_t>(n_slabs, 1), WG_CTAS);
        if (e == cudaSuccess && n_slabs)
            e = launch_pdl(k_wgrad_tc, dim3((unsigned)wg, 3), 128, WG_SMEM, stream, WgradArgs{{dy, dy2, dO}, {x0, y1, y2}}, slabs,
                           (int)n_slabs, box, wpart, &report->err);
        if (e == cudaSuccess)
            e = launch_pdl(ad ? k_wgrad_reduce<true> : k_wgrad_reduce<false>, dim3((unsigned)blocks(NW + CH, WR_K), 3),
                           WR_K * WR_C, 0, stream, wpart, wg, grad, ad ? *ad : Adam{});
        return e;
    }
    cudaError_t prepare()
    {
        k_prepare<<<blocks(3 * NW, 256), 256, 0, stream>>>(master, wb, wt);
        return cudaGetLastError();
    }
};

extern "C" {

int64_t lbm_corrector_num_params(void) { return NP; }

lbm_status lbm_corrector_create(const uint8_t* mask, int32_t nx, int32_t ny, int32_t nz, double u_scale,
                                double rho_scale, double du_scale, const float* params, lbm_alloc_fn alloc,
                                lbm_free_fn release, void* alloc_ctx, void* cuda_stream, lbm_corrector** out)
{
    if (!out) return nn_fail(LBM_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!mask || !params) return nn_fail(LBM_ERR_INVALID_ARG, "NULL mask or params");
    if (nx <= 0 || ny <= 0 || nz <= 0 || nx % 4 || ny % 4 || nz % 4)
        return nn_fail(LBM_ERR_INVALID_ARG, "the corrector's box extents must be positive multiples of 4");
    if ((int64_t)(nx + 2) * (ny + 2) * (nz + 2) * CH >= ((int64_t)1 << 31))
        return nn_fail(LBM_ERR_INVALID_ARG, "box too large for the corrector");
    if (!(u_scale > 0 && rho_scale > 0 && du_scale > 0)) return nn_fail(LBM_ERR_INVALID_ARG, "scales must be > 0");
    if ((alloc == nullptr) != (release == nullptr)) return nn_fail(LBM_ERR_INVALID_ARG, "give both allocator callbacks or neither");
    lbm_corrector* K = new (std::nothrow) lbm_corrector();
    if (!K) return nn_fail(LBM_ERR_OOM, "host allocation failed");
    K->box = Box{nx, ny, nz, nx + 2, ny + 2, nz + 2};
    K->n_cells = (int64_t)nx * ny * nz;
    K->u_scale = (float)u_scale;
    K->rho_scale = (float)rho_scale;
    K->du_scale = (float)du_scale;
    K->stream = static_cast<cudaStream_t>(cuda_stream);
    K->alloc = alloc;
    K->release = release;
    K->ctx = alloc_ctx;
    // tiles holding fluid, dilated by one tile
    const int tx = nx / 4, ty = ny / 4, tz = nz / 4;
    std::vector<uint8_t> has((size_t)tx * ty * tz, 0), use((size_t)tx * ty * tz, 0);
    for (int64_t c = 0; c < K->n_cells; ++c)
        if (mask[c]) {
            ++K->n_fluid;
            const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / ((int64_t)nx * ny));
            has[(size_t)(x / 4) + (size_t)tx * ((size_t)(y / 4) + (size_t)ty * (size_t)(z / 4))] = 1;
        }
    std::vector<int4> tl;
    for (int z = 0; z < tz; ++z)
        for (int y = 0; y < ty; ++y)
            for (int x = 0; x < tx; ++x) {
                bool near = false;
                for (int dz = -1; dz <= 1 && !near; ++dz)
                    for (int dy = -1; dy <= 1 && !near; ++dy)
                        for (int dx = -1; dx <= 1 && !near; ++dx) {
                            const int X = x + dx, Y = y + dy, Z = z + dz;
                            if (X < 0 || Y < 0 || Z < 0 || X >= tx || Y >= ty || Z >= tz) continue;
                            near = has[(size_t)X + (size_t)tx * ((size_t)Y + (size_t)ty * (size_t)Z)] != 0;
                        }
                if (near) {
                    tl.push_back(make_int4(4 * x, 4 * y, 4 * z, 0));
                    use[(size_t)x + (size_t)tx * ((size_t)y + (size_t)ty * (size_t)z)] = 1;
                }
            }
    K->n_tiles = (int64_t)tl.size();
    // slabs of 8 x 16 x 1 cells that meet a tile of that set
    std::vector<int4> sv;
    for (int z = 0; z < nz; ++z)
        for (int y0 = 0; y0 < ny; y0 += SL_Y)
            for (int x0 = 0; x0 < nx; x0 += SL_X) {
                bool any = false;
                for (int y = y0; y < std::min(ny, y0 + SL_Y) && !any; y += 4)
                    for (int x = x0; x < std::min(nx, x0 + SL_X) && !any; x += 4)
                        any = use[(size_t)(x / 4) + (size_t)tx * ((size_t)(y / 4) + (size_t)ty * (size_t)(z / 4))] != 0;
                if (any) sv.push_back(make_int4(x0, y0, z, 0));
            }
    K->n_slabs = (int64_t)sv.size();
    const size_t act = (size_t)K->box.px * K->box.py * K->box.pz * CH * sizeof(__nv_bfloat16);
    const size_t cells = (size_t)K->n_cells;
    bool ok = true;
    auto D = [&](size_t bytes) {
        void* p = K->dev(bytes);
        ok = ok && p;
        return p;
    };
    K->mask = static_cast<uint8_t*>(D(cells));
    K->slabs = static_cast<int4*>(D(sizeof(int4) * std::max<size_t>(sv.size(), 1)));
    K->report = static_cast<lbm_corrector::Report*>(D(sizeof(lbm_corrector::Report)));
    K->x0 = static_cast<__nv_bfloat16*>(D(act));
    K->y1 = static_cast<__nv_bfloat16*>(D(act));
    K->y2 = static_cast<__nv_bfloat16*>(D(act));
    K->dO = static_cast<__nv_bfloat16*>(D(act));
    K->dy = static_cast<__nv_bfloat16*>(D(act));
    K->dy2 = static_cast<__nv_bfloat16*>(D(act));
    K->o4 = static_cast<float*>(D(sizeof(float) * 4 * cells));
    K->rho = static_cast<float*>(D(sizeof(float) * cells));
    K->u = static_cast<float*>(D(sizeof(float) * 3 * cells));
    K->du = static_cast<float*>(D(sizeof(float) * 3 * cells));
    K->master = static_cast<float*>(D(sizeof(float) * NP));
    K->grad = static_cast<float*>(D(sizeof(float) * NP));
    K->m = static_cast<float*>(D(sizeof(float) * NP));
    K->v = static_cast<float*>(D(sizeof(float) * NP));
    K->wpart = static_cast<float*>(D(sizeof(float) * 3 * (size_t)WG_CTAS * (NW + CH)));
    K->wb = static_cast<__nv_bfloat16*>(D(sizeof(__nv_bfloat16) * 3 * NW));
    K->wt = static_cast<__nv_bfloat16*>(D(sizeof(__nv_bfloat16) * 3 * NW));
    if (!ok) {
        K->release_all();
        delete K;
        return nn_fail(LBM_ERR_OOM, "allocation failed: corrector buffers");
    }
    cudaError_t e = cudaMemcpyAsync(K->mask, mask, cells, cudaMemcpyHostToDevice, K->stream);
    if (e == cudaSuccess && !sv.empty())
        e = cudaMemcpyAsync(K->slabs, sv.data(), sizeof(int4) * sv.size(), cudaMemcpyHostToDevice, K->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(K->report, 0, sizeof(lbm_corrector::Report), K->stream);
    if (e == cudaSuccess) e = cudaMallocHost((void**)&K->h_report, sizeof(lbm_corrector::Report));
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&K->ev, cudaEventDisableTiming);
    {  // the convolutions' grid and their shared-memory sizes, once
        int dev = 0;
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&K->sms, cudaDevAttrMultiProcessorCount, dev);
        const auto smem_attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_conv_tc<OUT_BF16>, smem_attr, (int)CONV_SMEM);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_conv_tc<OUT_F32>, smem_attr, (int)CONV_SMEM);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_conv_tc<OUT_DU>, smem_attr, (int)CONV_SMEM);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_wgrad_tc, smem_attr, (int)WG_SMEM);
    }
    {
        const __nv_bfloat16* ins[5] = {K->x0, K->y1, K->y2, K->dO, K->dy2};
        for (int t = 0; t < 5 && e == cudaSuccess; ++t) {
            e = encode_halo_map(&K->tmaps[t], ins[t], K->box);
            K->tmap_of[t] = ins[t];
        }
    }
    for (__nv_bfloat16* p : {K->x0, K->y1, K->y2, K->dO, K->dy, K->dy2})
        if (e == cudaSuccess) e = cudaMemsetAsync(p, 0, act, K->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(K->o4, 0, sizeof(float) * 4 * cells, K->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(K->du, 0, sizeof(float) * 3 * cells, K->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(K->master, params, sizeof(float) * NP, cudaMemcpyHostToDevice, K->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(K->m, 0, sizeof(float) * NP, K->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(K->v, 0, sizeof(float) * NP, K->stream);
    if (e == cudaSuccess) e = K->prepare();
    if (e == cudaSuccess) e = cudaStreamSynchronize(K->stream);
    if (e != cudaSuccess) {
        K->release_all();
        delete K;
        return nn_fail(LBM_ERR_CUDA, std::string("corrector set-up: ") + cudaGetErrorString(e));
    }
    *out = K;
    return LBM_OK;
}

lbm_status lbm_corrector_get_params(lbm_corrector* K, float* params)
{
    if (!K || !params) return nn_fail(LBM_ERR_INVALID_ARG, "NULL argument");
    cudaError_t e = cudaMemcpyAsync(params, K->master, sizeof(float) * NP, cudaMemcpyDeviceToHost, K->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(K->stream);
    if (e != cudaSuccess) return nn_fail(LBM_ERR_CUDA, std::string("get params: ") + cudaGetErrorString(e));
    return LBM_OK;
}

lbm_status lbm_corrector_set_params(lbm_corrector* K, const float* params)
{
    if (!K || !params) return nn_fail(LBM_ERR_INVALID_ARG, "NULL argument");
    cudaError_t e = cudaMemcpyAsync(K->master, params, sizeof(float) * NP, cudaMemcpyHostToDevice, K->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(K->m, 0, sizeof(float) * NP, K->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(K->v, 0, sizeof(float) * NP, K->stream);
    if (e == cudaSuccess) e = K->prepare();
    if (e == cudaSuccess) e = cudaStreamSynchronize(K->stream);
    if (e != cudaSuccess) return nn_fail(LBM_ERR_CUDA, std::string("set params: ") + cudaGetErrorString(e));
    K->adam_t = 0;
    return LBM_OK;
}

lbm_status lbm_corrector_forward(lbm_corrector* K, const uint8_t* mask, const uint8_t* out_mask, const float* rho,
                                 const float* u, float* du)
{
    NvtxRange nvtx_range("lbm_corrector_forward");
    if (!K || !rho || !u || !du) return nn_fail(LBM_ERR_INVALID_ARG, "NULL argument");
    const uint8_t* om = out_mask ? out_mask : (mask ? mask : K->mask);
    // the slabs write their cells; the rest of the caller's box is zero
    cudaError_t e = K->forward(mask, rho, u, du, om, K->du_scale, true);
    if (e != cudaSuccess) return nn_fail(LBM_ERR_CUDA, std::string("corrector forward: ") + cudaGetErrorString(e));
    return LBM_OK;
}

lbm_status lbm_corrector_gradients(lbm_corrector* K, const uint8_t* mask, const uint8_t* out_mask, const float* rho,
                                   const float* u, const float* u_target, float* grad, double* loss)
{
    NvtxRange nvtx_range("lbm_corrector_gradients");
    if (!K || !rho || !u || !u_target || !grad || !loss) return nn_fail(LBM_ERR_INVALID_ARG, "NULL argument");
    cudaError_t e = K->train(mask, out_mask ? out_mask : (mask ? mask : K->mask), rho, u, u_target, nullptr);
    if (e == cudaSuccess) e = cudaMemcpyAsync(grad, K->grad, sizeof(float) * NP, cudaMemcpyDeviceToHost, K->stream);
    return K->finish(e, "corrector gradients", loss);
}

lbm_status lbm_corrector_train_step(lbm_corrector* K, const uint8_t* mask, const uint8_t* out_mask, const float* rho,
                                    const float* u, const float* u_target, double lr, double* loss)
{
    NvtxRange nvtx_range("lbm_corrector_train_step");
    if (!K || !rho || !u || !u_target) return nn_fail(LBM_ERR_INVALID_ARG, "NULL argument");
    if (!(lr > 0.0)) return nn_fail(LBM_ERR_INVALID_ARG, "lr must be > 0");
    K->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float bc1 = 1.0f - std::pow(b1, (float)K->adam_t), bc2 = 1.0f - std::pow(b2, (float)K->adam_t);
    const Adam ad{K->master, K->m, K->v, K->wb, K->wt, (float)lr, b1, b2, 1e-8f, bc1, bc2};
    cudaError_t e = K->train(mask, out_mask ? out_mask : (mask ? mask : K->mask), rho, u, u_target, &ad);
    if (loss) return K->finish(e, "corrector train step", loss);
    if (e != cudaSuccess) return nn_fail(LBM_ERR_CUDA, std::string("corrector train step: ") + cudaGetErrorString(e));
    return LBM_OK;
}

lbm_status lbm_corrector_apply(lbm_corrector* K, lbm_domain* dom, const uint8_t* mask, const uint8_t* out_mask,
                               double gain)
{
    NvtxRange nvtx_range("lbm_corrector_apply");
    if (!K || !dom) return nn_fail(LBM_ERR_INVALID_ARG, "NULL argument");
    if (!(gain > 0.0 && gain <= 1.0)) return nn_fail(LBM_ERR_INVALID_ARG, "gain must lie in (0, 1]");
    lbm_info I{};
    lbm_get_info(dom, &I);
    if (I.nx != K->box.nx || I.ny != K->box.ny || I.nz != K->box.nz)
        return nn_fail(LBM_ERR_INVALID_ARG, "the domain's box differs from the corrector's");
    DomainAccess da{};
    if (!domain_access(dom, &da)) return nn_fail(LBM_ERR_INVALID_ARG, "NULL domain");
    // rho, u are exported on the domain's stream and the correction is applied there: the
    // corrector's own stream waits for the one and the domain's stream for the other.  The cells
    // that are not fluid are cleared only when the staging last held another domain's export
    // (the box is cleared once per domain, not on every call)
    cudaError_t e = enqueue_macroscopic_dense(dom, K->rho, K->u, da.serial != K->export_serial);
    K->export_serial = e == cudaSuccess ? da.serial : 0;
    if (e == cudaSuccess && da.stream != K->stream) {
        e = cudaEventRecord(K->ev, da.stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(K->stream, K->ev, 0);
    }
    const uint8_t* om = out_mask ? out_mask : (mask ? mask : K->mask);
    // cells outside the slabs keep the zero of set-up
    if (e == cudaSuccess) e = K->forward(mask, K->rho, K->u, K->du, om, (float)(K->du_scale * gain), false);
    if (e == cudaSuccess && da.stream != K->stream) {
        e = cudaEventRecord(K->ev, K->stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(da.stream, K->ev, 0);
    }
    // the correction reuses the rho, u exported above (the domain has not stepped since)
    if (e == cudaSuccess) e = enqueue_velocity_correction(dom, K->rho, K->u, K->du);
    if (e != cudaSuccess) return nn_fail(LBM_ERR_CUDA, std::string("corrector apply: ") + cudaGetErrorString(e));
    return LBM_OK;
}

void lbm_corrector_destroy(lbm_corrector* K)
{
    if (!K) return;
    cudaStreamSynchronize(K->stream);
    K->release_all();
    delete K;
}

lbm_status lbm_restrict(const float* fine_rho, const float* fine_u, const uint8_t* fine_mask, int32_t fnx, int32_t fny,
                        int32_t fnz, float* coarse_rho, float* coarse_u, void* cuda_stream)
{
    NvtxRange nvtx_range("lbm_restrict");
    if (!fine_rho || !fine_u || !fine_mask || !coarse_rho || !coarse_u) return nn_fail(LBM_ERR_INVALID_ARG, "NULL argument");
    if (fnx <= 0 || fny <= 0 || fnz <= 0 || fnx % 2 || fny % 2 || fnz % 2)
        return nn_fail(LBM_ERR_INVALID_ARG, "fine extents must be positive and even");
    const int64_t cn = (int64_t)(fnx / 2) * (fny / 2) * (fnz / 2);
    const cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // four cells a thread: rows of whole groups, arrays on the boundaries of the wide accesses, and enough groups for
    // the chip (128^3 -> 64^3: vessel 6.5 us with four and 4.5 with one, all cells 8.1 and 6.5; 144^3: 6.3 and 8.4)
    const auto aligned = [](const void* p, uintptr_t n) { return reinterpret_cast<uintptr_t>(p) % n == 0; };
    const bool four = cn > (1 << 18) && fnx % 8 == 0 && aligned(fine_mask, 8) && aligned(coarse_rho, 16) && aligned(coarse_u, 16);
    const bool wide = four && aligned(fine_rho, 16) && aligned(fine_u, 16);
    auto k = wide ? k_restrict<4, true> : four ? k_restrict<4, false> : k_restrict<1, false>;
    k<<<blocks(four ? cn / 4 : cn, 256), 256, 0, st>>>(fine_rho, fine_u, fine_mask, fnx, fny, fnz, coarse_rho, coarse_u);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return nn_fail(LBM_ERR_CUDA, std::string("restrict: ") + cudaGetErrorString(e));
    return LBM_OK;
}

}  // extern "C"
