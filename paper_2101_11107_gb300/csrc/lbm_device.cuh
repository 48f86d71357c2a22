// lbm_device.cuh -- device code of the fused stream-collide step and its companions, templated
// on the storage precision, the streaming scheme and the launch shape.  Included by one
// translation unit per storage precision (lbm_step_fp32.cu, lbm_step_fp16.cu, lbm_step_bf16.cu).
//
// Method (Hosseini et al.):
//   LBE f_i(x + c_i, n + 1) = f_i(x, n) + Omega_i             (Sec. 2.1.1, first equation)
//   Omega = T^-1 S T (f_eq - f), central Hermite moments       (Sec. 2.1.3)
//   T f_eq = (rho, 0, ..., 0) with the full-expansion f_eq     (Eq. Hermite_coeff_eq)
//   Bouzidi interpolated bounce-back, q = |x_f - x_s| / |c|    (Sec. 2.1.4)
//
// GB300 design:
//   * Populations are SoA, pop[i][slot], slot = brick * 64 + local cell of a 4x4x4 brick; only
//     bricks with fluid (and, for the twist, their +{0,1}^3 neighbours) are stored.  One thread
//     per slot, BRICKS bricks per CTA; a warp covers half a brick and hands the brick's
//     neighbour row out with shuffles, so streaming reads no per-cell neighbour index and the
//     kernel has no CTA barrier.
//   * Two streaming schemes, same arithmetic, bitwise-equal results:
//       A-B (pull from array A, write to array B): 26 neighbour cells per update;
//       esoteric twist (in place, one array): the thread of cell x touches only the 8 cells
//       x + {0,1}^3.  On even levels it reads f_i from slot i of cell x + p_opp(i) and writes
//       f*_i to slot opp(i) of cell x + p_i; odd levels swap the two slot roles
//       (p_i = max(c_i, 0)).  Every location is read and then written by one thread only.
//   * Every lane issues all 27 loads unconditionally; halfway bounce-back is folded into the
//     address (A-B: the cell's own opposite slot; twist: the swapped slot of the same cell).
//   * A per-slot 32-bit word carries the wall mask and the cell kind, so bulk cells take no
//     boundary branch.
//   * Arithmetic is FP32 on deviations d_i = f_i - w_i throughout (moments, transforms,
//     relaxation, closures): the O(1) rest-state weights never enter a rounding.
//   * The 27x27 transform runs as three passes of nine 1-D three-point transforms
//     (T = M(u_x) (x) M(u_y) (x) M(u_z)), forward and inverse, about 500 FP32 flops per cell;
//     with the default rates (third to sixth order = 1) the forward part reduces to the moments
//     up to second order (about 350 flops per cell in all).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "lbm_internal.h"

namespace lbm {
namespace dev {

constexpr float CS2 = 1.0f / 3.0f;

// ------------------------------------------------------------------------------ LBM_DEBUG
// Built with -DLBM_DEBUG, every access of a population array, the Bouzidi q and side lists and
// the open-boundary records is checked against the array's extent first: an access out of range
// is skipped (a load gives 0) and the check's code is kept in a device flag of this translation
// unit (the first one wins), which the host reads at its next synchronising call.  Codes:
// 1 A-B pull, 2 twist load, 3 twist store, 4 A-B store, 5 Bouzidi q / side list, 6 open-boundary
// record, 7 velocity-correction update.  Without the macro every check is the constant true.
#ifdef LBM_DEBUG
static __device__ unsigned int g_debug_fault = 0u;
__device__ __forceinline__ bool dbg_in_range(uint64_t i, uint64_t n, unsigned code)
{
    if (i < n) return true;
    atomicCAS(&g_debug_fault, 0u, code);
    return false;
}
#define LBM_IN_RANGE(i, n, code) ::lbm::dev::dbg_in_range((uint64_t)(i), (uint64_t)(n), (code))
#else
#define LBM_IN_RANGE(i, n, code) true
#endif

// ------------------------------------------------------------------------------ storage
// FP32 stores d_i; FP16 / BF16 store d_i / w_i.  Loads are plain, not of the read-only path: a kernel may
// start while the step before it still writes (pdl_wait).
template <int ST>
struct Store;

template <>
struct Store<LBM_STORE_FP32> {
    using T = float;
    static constexpr bool SCALED = false;  // the stored value is d itself
    // with a 256-byte L2 fetch on a miss: a warp reads 128 bytes of a brick's 256-byte plane
    // row and the other half-brick warp (or the neighbour brick's shifted read) the rest, so
    // the second request finds it in L2 (measured: -3% per step cold for the two-cell kernel,
    // neutral to slightly worse for 16-bit storage, which keeps plain loads).  Volatile, so that
    // it stays behind pdl_wait; every caller's stores to a location it loaded depend on the
    // loaded value.
    static __device__ __forceinline__ float load_rw(const void* p, int, uint32_t off)
    {
        float v;
        asm volatile("ld.global.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(static_cast<const float*>(p) + off));
        return v;
    }
    static __device__ __forceinline__ float load_rw_h(const void* p, uint32_t off) { return load_rw(p, 0, off); }
    static __device__ __forceinline__ void store(void* p, int, uint32_t off, float v)
    {
        static_cast<float*>(p)[off] = v;
    }
    static __device__ __forceinline__ void store_h(void* p, uint32_t off, float v) { static_cast<float*>(p)[off] = v; }
    // v carries the factor 2^nnz(c_i) of the deferred-halving inverse transform (exact)
    static __device__ __forceinline__ void store_x(void* p, int i, uint32_t off, float v)
    {
        static_cast<float*>(p)[off] = nnz_of(i) ? v * pow2_neg(nnz_of(i)) : v;
    }
};

template <>
struct Store<LBM_STORE_FP16> {
    using T = __half;
    static __device__ __forceinline__ float load_rw(const void* p, int i, uint32_t off)
    {
        return w_of(i) * __half2float(static_cast<const __half*>(p)[off]);
    }
    // the stored h = d / w as a float (the caller multiplies by w_i: scale_in)
    static constexpr bool SCALED = true;
    static __device__ __forceinline__ float load_rw_h(const void* p, uint32_t off)
    {
        return __half2float(static_cast<const __half*>(p)[off]);
    }
    // v already multiplied by the direction's store factor (scale_out)
    static __device__ __forceinline__ void store_h(void* p, uint32_t off, float v)
    {
        static_cast<__half*>(p)[off] = __float2half_rn(v);
    }
    static __device__ __forceinline__ void store(void* p, int i, uint32_t off, float v)
    {
        static_cast<__half*>(p)[off] = __float2half_rn(v * inv_w_of(i));
    }
    // v carries the factor 2^nnz(c_i): one multiply by the exact constant 2^-nnz / w_i
    static __device__ __forceinline__ void store_x(void* p, int i, uint32_t off, float v)
    {
        static_cast<__half*>(p)[off] = __float2half_rn(v * (inv_w_of(i) * pow2_neg(nnz_of(i))));
    }
};

template <>
struct Store<LBM_STORE_BF16> {
    using T = __nv_bfloat16;
    static __device__ __forceinline__ float load_rw(const void* p, int i, uint32_t off)
    {
        return w_of(i) * __bfloat162float(static_cast<const __nv_bfloat16*>(p)[off]);
    }
    // the stored h = d / w as a float (the caller multiplies by w_i: scale_in)
    static constexpr bool SCALED = true;
    static __device__ __forceinline__ float load_rw_h(const void* p, uint32_t off)
    {
        return __bfloat162float(static_cast<const __nv_bfloat16*>(p)[off]);
    }
    // v already multiplied by the direction's store factor (scale_out)
    static __device__ __forceinline__ void store_h(void* p, uint32_t off, float v)
    {
        static_cast<__nv_bfloat16*>(p)[off] = __float2bfloat16_rn(v);
    }
    static __device__ __forceinline__ void store(void* p, int i, uint32_t off, float v)
    {
        static_cast<__nv_bfloat16*>(p)[off] = __float2bfloat16_rn(v * inv_w_of(i));
    }
    static __device__ __forceinline__ void store_x(void* p, int i, uint32_t off, float v)
    {
        static_cast<__nv_bfloat16*>(p)[off] = __float2bfloat16_rn(v * (inv_w_of(i) * pow2_neg(nnz_of(i))));
    }
};

// The multiplies around the raw accessors, with packed FP32x2 instructions where two directions
// share the factor (the same product as the per-direction load / store above, so bit-identical).
// In: d_i = w_i h_i for the 16-bit storages; the directions j and j + 18 (c_z = -1 and +1, same
// c_x, c_y) share w.
template <int ST>
__device__ __forceinline__ void scale_in(float (&d)[Q])
{
    if constexpr (Store<ST>::SCALED) {
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const float2 v = __fmul2_rn(make_float2(d[j], d[j + 18]), make_float2(w_of(j), w_of(j)));
            d[j] = v.x;
            d[j + 18] = v.y;
            d[j + 9] = d[j + 9] * w_of(j + 9);
        }
    }
}

// Out: the factor taking a post-collision d_i to the stored value -- 1/w_i for the 16-bit
// storages, times 2^-nnz(c_i) when d carries the deferred-halving factors (X).
template <int ST, bool X>
__host__ __device__ constexpr float out_factor(int i)
{
    return (Store<ST>::SCALED ? inv_w_of(i) : 1.0f) * (X ? pow2_neg(nnz_of(i)) : 1.0f);
}

// the directions 3k and 3k + 2 (c_x = -1 and +1, same c_y, c_z) share the factor
template <int ST, bool X>
__device__ __forceinline__ void scale_out(float (&d)[Q])
{
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        constexpr float one = 1.0f;
        if (out_factor<ST, X>(3 * k) != one) {
            const float c = out_factor<ST, X>(3 * k);
            const float2 v = __fmul2_rn(make_float2(d[3 * k], d[3 * k + 2]), make_float2(c, c));
            d[3 * k] = v.x;
            d[3 * k + 2] = v.y;
        }
        if (out_factor<ST, X>(3 * k + 1) != one) d[3 * k + 1] = d[3 * k + 1] * out_factor<ST, X>(3 * k + 1);
    }
}

// two cells at once (a lane of the two-cell kernel): every direction one packed multiply
template <int ST, bool X>
__device__ __forceinline__ void scale_out2(float2 (&d)[Q])
{
#pragma unroll
    for (int i = 0; i < Q; ++i)
        if (out_factor<ST, X>(i) != 1.0f) d[i] = __fmul2_rn(d[i], make_float2(out_factor<ST, X>(i), out_factor<ST, X>(i)));
}

// Programmatic dependent launch between consecutive steps: a step kernel lets the next one start as
// soon as all its own CTAs are running (pdl_trigger), and the next one loads what no step writes (cell
// words, records, brick rows) before it waits for this one's populations to be complete and visible
// (pdl_wait).  Every thread waits before it reads or writes a population, and a kernel ends only after
// its waiting threads, so the order of more than two kernels follows.  Populations are read with plain
// loads (not the read-only path: another step may still be writing when a kernel starts).  Both are
// no-ops in a launch without the attribute.  The step is bound by latency on small domains: the launch
// gap and the index loads of one step hide behind the tail of the one before.  Measured, per step:
// 32x32x64 pipe 5.9 -> 4.05 us, 150 k cell aneurysm 14.0 -> 11.9 us, 633 k cell pipe 26.3 -> 24.2 us
// (FP32 twist), 31.6 -> 29.6 us (A-B), 21.8 -> 19.9 us (FP16); batch of 178 k cells 20.5 -> 19.3 us.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------------------ streaming
template <int ST>
__device__ __forceinline__ void fetch_ab_at(const void* src, uint32_t n, const uint32_t (&off)[Q], float (&d)[Q])
{
#pragma unroll
    for (int i = 0; i < Q; ++i) d[i] = LBM_IN_RANGE(off[i], (uint64_t)Q * n, 1) ? Store<ST>::load_rw_h(src, off[i]) : 0.0f;
    scale_in<ST>(d);
}

// A-B pull: f_i(x, n) = f*_i(x - c_i, n - 1) from `src`; a wall link reads the cell's own
// opposite slot (halfway bounce-back f_i(x, n) = f*_opp(i)(x, n - 1)).
template <int ST>
__device__ __forceinline__ void fetch_ab(const void* src, uint32_t n, const int32_t* nbrow, uint32_t slot, uint32_t wm,
                                         float (&d)[Q])
{
    const int l = (int)(slot & (BRICK_CELLS - 1));
    const int lx = l & (BX - 1), ly = (l >> LBX) & (BY - 1), lz = l >> (LBX + LBY);
    uint32_t off[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int sx = lx - cx_of(i), sy = ly - cy_of(i), sz = lz - cz_of(i);
        // sx in [-1, BX]: the arithmetic shift gives the brick offset -1, 0 or +1
        const int ob = 13 + (sx >> LBX) + 3 * (sy >> LBY) + 9 * (sz >> LBZ);
        const uint32_t nb = (uint32_t)__ldg(nbrow + ob);
        const uint32_t s = nb * BRICK_CELLS + (uint32_t)brick_local(sx & (BX - 1), sy & (BY - 1), sz & (BZ - 1));
        const bool wall = (wm >> i) & 1u;
        off[i] = wall ? (uint32_t)(Q - 1 - i) * n + slot : (uint32_t)i * n + s;
    }
    pdl_wait();
    fetch_ab_at<ST>(src, n, off, d);
}

// A-B pull in the step kernel: the brick's 27-entry neighbour row is held by lanes 0..26 of the
// warp (a warp covers half of one brick) and handed out with shuffles, so no CTA barrier or
// shared staging is needed.  All 32 lanes must call this; the offset of direction i.
__device__ __forceinline__ uint32_t ab_offset_shfl(uint32_t n, int32_t row_lane, uint32_t slot, uint32_t wm, int i)
{
    const int l = (int)(slot & (BRICK_CELLS - 1));
    const int lx = l & (BX - 1), ly = (l >> LBX) & (BY - 1), lz = l >> (LBX + LBY);
    const int sx = lx - cx_of(i), sy = ly - cy_of(i), sz = lz - cz_of(i);
    const int ob = 13 + (sx >> LBX) + 3 * (sy >> LBY) + 9 * (sz >> LBZ);
    const uint32_t nb = (uint32_t)__shfl_sync(0xffffffffu, row_lane, ob);
    const uint32_t s = nb * BRICK_CELLS + (uint32_t)brick_local(sx & (BX - 1), sy & (BY - 1), sz & (BZ - 1));
    return ((wm >> i) & 1u) ? (uint32_t)(Q - 1 - i) * n + slot : (uint32_t)i * n + s;
}

// How many offsets an A-B step forms before it loads from them.  Loads are plain (a step may start while the one
// before it still writes) and stay in order with the shuffles, and a shuffle waits for the loads before it, so
// between groups few loads are in flight.  All 27 in one group is the fastest but for the default rates in FP32
// (one by one) and in 16 bits without links (three).  us a step, one by one / threes / all:
//   2.7 M cell Bouzidi pipe  FP16 170 / 149 / 98    FP16 TRT 197 / - / 108    FP32 TRT 124 / - / 118
//   633 k cell pipe          FP16 22.3 / 21.9 / 20.8    FP16 TRT 43.5 / - / 25.0
//   95 k cell pipe           FP16 5.4 / 5.4 / 6.2
//   FP32, default rates: 2.7 M cells 109 / 109 / 116, 95 k cells 4.6 / 4.9 / 6.1
template <int ST, int COLL, int LINKS>
__host__ __device__ constexpr int ab_group()
{
    if (COLL != COLL_CHM_FAST) return Q;
    return ST == LBM_STORE_FP32 ? 1 : LINKS == 0 ? 3 : Q;
}

// Twist corner slots in the step kernel: lanes hold the brick's nb8 row (lane & 7).
__device__ __forceinline__ void corner_slots_shfl(int32_t row_lane, uint32_t slot, uint32_t (&cs)[8])
{
    const int l = (int)(slot & (BRICK_CELLS - 1));
    const int lx = l & (BX - 1), ly = (l >> LBX) & (BY - 1), lz = l >> (LBX + LBY);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int tx = lx + (e & 1), ty = ly + ((e >> 1) & 1), tz = lz + (e >> 2);
        const int ob = (tx >> LBX) | ((ty >> LBY) << 1) | ((tz >> LBZ) << 2);
        const uint32_t nb = (uint32_t)__shfl_sync(0xffffffffu, row_lane, ob);
        cs[e] = nb * BRICK_CELLS + (uint32_t)brick_local(tx & (BX - 1), ty & (BY - 1), tz & (BZ - 1));
    }
}

// Slots of the 8 cells x + e, e in {0,1}^3 (index ex + 2 ey + 4 ez), from the brick's nb8 row.
__device__ __forceinline__ void corner_slots(const int32_t* nb8, uint32_t slot, uint32_t (&cs)[8])
{
    const int l = (int)(slot & (BRICK_CELLS - 1));
    const int lx = l & (BX - 1), ly = (l >> LBX) & (BY - 1), lz = l >> (LBX + LBY);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int tx = lx + (e & 1), ty = ly + ((e >> 1) & 1), tz = lz + (e >> 2);
        const int ob = (tx >> LBX) | ((ty >> LBY) << 1) | ((tz >> LBZ) << 2);
        cs[e] = (uint32_t)nb8[ob] * BRICK_CELLS + (uint32_t)brick_local(tx & (BX - 1), ty & (BY - 1), tz & (BZ - 1));
    }
}

// Esoteric twist read at level parity P: f_i from slot (P ? opp(i) : i) of cell x + p_opp(i);
// on a wall link the other slot of the same cell, which holds f*_opp(i)(x, n - 1).
// PC >= 0 fixes the parity at compile time; with `clean` (warp-uniform: no lane of the warp has a
// wall link) every plane index is then a constant.
template <int ST, int PC = -1>
__device__ __forceinline__ void fetch_et(const void* pop, uint32_t n, const uint32_t (&cs)[8], uint32_t wm,
                                         int parity, float (&d)[Q], bool clean = false)
{
    if (PC >= 0 && clean) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const uint32_t off = (PC ? (uint32_t)(Q - 1 - i) : (uint32_t)i) * n + cs[corner_neg(i)];
            d[i] = LBM_IN_RANGE(off, (uint64_t)Q * n, 2) ? Store<ST>::load_rw_h(pop, off)
                                                        : 0.0f;
        }
        scale_in<ST>(d);
        return;
    }
    if (PC >= 0) parity = PC;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const uint32_t flip = ((uint32_t)parity ^ (wm >> i)) & 1u;
        const uint32_t dir = flip ? (uint32_t)(Q - 1 - i) : (uint32_t)i;
        const uint32_t off = dir * n + cs[corner_neg(i)];
        d[i] = LBM_IN_RANGE(off, (uint64_t)Q * n, 2) ? Store<ST>::load_rw_h(pop, off)
                                                    : 0.0f;
    }
    scale_in<ST>(d);
}

// Esoteric twist write after a step of parity P: f*_i to slot (P ? i : opp(i)) of cell x + p_i
// (PC >= 0: the parity fixed at compile time; X: d carries the factors 2^nnz(c_i); H: d has been
// through scale_out, the stored values as floats).
template <int ST, int PC = -1, bool X = false, bool H = false>
__device__ __forceinline__ void store_et(void* pop, uint32_t n, const uint32_t (&cs)[8], int parity,
                                         const float (&d)[Q])
{
    if (PC >= 0) {
        parity = PC;
        // with constant planes a write address equals the read address of the opposite
        // direction; an opaque copy of n keeps the compiler from holding 27 addresses live
        // through the collision (it recomputes them instead)
        asm("mov.b32 %0, %0;" : "+r"(n));
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const uint32_t dir = parity ? (uint32_t)i : (uint32_t)(Q - 1 - i);
        const uint32_t off = dir * n + cs[corner_pos(i)];
        if (!LBM_IN_RANGE(off, (uint64_t)Q * n, 3)) continue;
        if (H) Store<ST>::store_h(pop, off, d[i]);
        else if (X) Store<ST>::store_x(pop, i, off, d[i]);
        else Store<ST>::store(pop, i, off, d[i]);
    }
}

// ------------------------------------------------------------------------------ boundaries
// Open-boundary closure of an inlet (velocity) or outlet (density) cell on an axis-aligned face
// with inward normal n = sign e_axis, in deviation form.  Known: c.n <= 0.  With
// D = sum_{c.n=0} d + 2 sum_{c.n<0} d (and sum_{c.n=0} w + 2 sum_{c.n<0} w = 1):
//   inlet:  u.n = U phi, rho = (1 + D)/(1 - u.n);   outlet: rho = rho_out, u.n = 1 - (1 + D)/rho.
// Both are evaluated as deviations from 1 (rho - 1 = (D + u.n)/(1 - u.n),
// u.n = (rho_out - 1 - D)/rho_out), so that D is never rounded against 1.
// The nine unknowns (c.n = +1) by non-equilibrium bounce-back with the full equilibrium; since
// u has no tangential part, f_eq_i - f_eq_opp(i) = 6 w_i rho u.n.  Then the tangential momentum
// is zeroed by d_i += c_it D_t / 6, D_t = -sum_j c_jt d_j, which leaves mass and normal
// momentum unchanged.
template <int AXIS, int SGN>
__device__ __forceinline__ void close_face(float (&d)[Q], int kind, float phi, float U, float rho_out, float drho_out)
{
    auto normal = [](int i) { return SGN * (AXIS == 0 ? cx_of(i) : AXIS == 1 ? cy_of(i) : cz_of(i)); };
    float D = 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (normal(i) == 0) D += d[i];
        if (normal(i) < 0) D += 2.0f * d[i];
    }
    float rho, un;
    if (kind == KIND_INLET) {
        un = U * phi;
        rho = 1.0f + (D + un) / (1.0f - un);
    } else {
        rho = rho_out;
        un = (drho_out - D) / rho_out;
    }
    const float ru6 = 6.0f * rho * un;
#pragma unroll
    for (int i = 0; i < Q; ++i)
        if (normal(i) == 1) d[i] = d[Q - 1 - i] + w_of(i) * ru6;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        if (t == AXIS) continue;
        float mom = 0.0f;
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            const int ct = t == 0 ? cx_of(j) : t == 1 ? cy_of(j) : cz_of(j);
            if (ct == 1) mom += d[j];
            if (ct == -1) mom -= d[j];
        }
        const float corr = -mom * (1.0f / 6.0f);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int ct = t == 0 ? cx_of(i) : t == 1 ? cy_of(i) : cz_of(i);
            if (normal(i) == 1 && ct != 0) d[i] += ct == 1 ? corr : -corr;
        }
    }
}

// One instance per face: the lanes of a warp that meet open cells meet one face's, and step through about
// 90 instructions; with the face as run-time selects in one body they were about 450, on the longest path
// of the step of a small domain.
__device__ __forceinline__ void close_open(float (&d)[Q], int kind, int axis, int sgn, float phi, float U,
                                           float rho_out, float drho_out)
{
    switch (2 * axis + (sgn > 0)) {
    case 0: close_face<0, -1>(d, kind, phi, U, rho_out, drho_out); break;
    case 1: close_face<0, 1>(d, kind, phi, U, rho_out, drho_out); break;
    case 2: close_face<1, -1>(d, kind, phi, U, rho_out, drho_out); break;
    case 3: close_face<1, 1>(d, kind, phi, U, rho_out, drho_out); break;
    case 4: close_face<2, -1>(d, kind, phi, U, rho_out, drho_out); break;
    default: close_face<2, 1>(d, kind, phi, U, rho_out, drho_out); break;
    }
}

// Interpolated bounce-back on top of the bounce-back already in d (Sec. 2.1.4 in pull form, beta = opp(alpha)
// pointing into the wall):
//   q <  1/2: f_a(x) = 2q f*_b(x) + (1 - 2q) f*_b(x + c_a)  [= the value pulled for b]
//   q >= 1/2: f_a(x) = f*_b(x)/(2q) + (2q - 1)/(2q) f*_a(x)
// with halfway bounce-back kept if x + c_a is not fluid in the first branch.  f*_a(x, n - 1) comes from
// the cell's own slot (A-B) or from the side buffer (twist: that slot is the one x + c_a pulls and
// overwrites in this step).  Explicit roundings: every kernel gives the same bits.
__device__ __forceinline__ float wall_low(float k, float fb, float fb_pulled)
{
    return __fmaf_rn(k, fb, __fmul_rn(__fadd_rn(1.0f, -k), fb_pulled));
}
__device__ __forceinline__ float wall_high(float k, float fb, float fa)
{
    return __fmaf_rn(__fadd_rn(1.0f, -k), fa, __fmul_rn(k, fb));
}

// Position of wall link i of a Bouzidi cell in the packed link lists (coefficients, and the twist side
// buffer): the cell's entries start at its aux record and follow the set bits of its wall mask
// in direction order.
__device__ __forceinline__ uint32_t link_index(uint32_t off, uint32_t wm, int i)
{
    return off + (uint32_t)__popc(wm & ((1u << i) - 1u));
}

// The open-boundary closure of a cell, if it is an inlet or outlet cell (aux: its record).
__device__ __forceinline__ void open_rules(const DomainView& v, uint32_t word, int64_t rec, const LevelArgs& a,
                                           float (&d)[Q])
{
    const int kind = (int)((word >> WORD_KIND_SHIFT) & 3u);
    if (kind >= KIND_INLET && LBM_IN_RANGE(rec, v.n_io, 6))
        close_open(d, kind, v.io_axis[rec], v.io_sign[rec], v.io_phi[rec], a.U, a.rho_out, a.drho_out);
}

// The wall rules and closures of one cell by its own thread (the two-cell step and the kernels that only
// read; the one-cell steps share a warp's links out among its lanes, BouzidiLinks).  Returns the mask
// of the q >= 1/2 links, whose f*_a the twist must keep in the side buffer.
// aux: the cell's record (v.aux[slot]) when the caller has loaded it already, else -1
template <int ST, int SCHEME>
__device__ __forceinline__ uint32_t wall_rules(const DomainView& v, const void* src_ab, uint32_t slot,
                                               uint32_t word, const LevelArgs& a, float (&d)[Q], int32_t aux = -1)
{
    const uint32_t wm = word & WORD_WALL_MASK;
    const int kind = (int)((word >> WORD_KIND_SHIFT) & 3u);
    uint32_t half = 0u;
    if (kind == KIND_BOUZIDI) {
        const uint32_t off = (uint32_t)(aux >= 0 ? aux : v.aux[slot]);
        // A direction's rule reads d_i and, only when opp(i) has no link, d_opp(i), which no other
        // direction's rule changes: the order of the directions does not matter.  The links of nine
        // directions at a time (their coefficients and f*_a requested before the first is used: one memory
        // latency per group, not per link; the A-B exports of a 48 k cell vessel took 13 us link by link).
        constexpr int GS = 9;
#pragma unroll
        for (int g = 0; g < Q / GS; ++g) {
            float qg[GS], fg[GS];
#pragma unroll
            for (int j = 0; j < GS; ++j) {
                const int i = GS * g + j;
                const uint32_t li = link_index(off, wm, i);
                const bool has = ((wm >> i) & 1u) && LBM_IN_RANGE(li, v.n_bq, 5);
                qg[j] = has ? __ldg(v.bq + li) : 0.0f;
                // loaded whatever q is, so that the two loads do not wait on each other
                fg[j] = !has ? 0.0f
                             : (SCHEME == LBM_SCHEME_ESOTERIC)
                                   ? Store<ST>::load_rw(v.side, i, li)
                                   : Store<ST>::load_rw(src_ab, i, (uint32_t)i * (uint32_t)v.n_slots + slot);
            }
#pragma unroll
            for (int j = 0; j < GS; ++j) {
                const int i = GS * g + j;
                const float k = qg[j];
                if (k > 0.0f) {  // 0: no link (or halfway bounce-back on this link)
                    if (!(wm & (1u << (Q - 1 - i)))) d[i] = wall_low(k, d[i], d[Q - 1 - i]);
                } else if (k < 0.0f) {
                    d[i] = wall_high(-k, d[i], fg[j]);
                    half |= 1u << i;
                }
            }
        }
    } else if (kind >= KIND_INLET) {
        open_rules(v, word, aux >= 0 ? aux : v.aux[slot], a, d);
    }
    return half;
}

// ------------------------------------------------------------------------------ collide
__device__ __forceinline__ void fwd3(float& gm, float& g0, float& gp, float u, float u2mcs)
{
    // (g(-1), g(0), g(+1)) -> central Hermite moments (m0, m1, m2) about u
    const float m0 = gm + g0 + gp;
    const float s1 = gp - gm;
    const float s2 = gp + gm;
    gm = m0;
    g0 = fmaf(-u, m0, s1);
    gp = fmaf(u2mcs, m0, fmaf(-2.0f * u, s1, s2));
}

__device__ __forceinline__ void inv3(float& m0, float& m1, float& m2, float u, float u2pcs)
{
    // (m0, m1, m2) -> (g(-1), g(0), g(+1)): raw sums S1 = g+ - g-, S2 = g+ + g-
    const float S1 = fmaf(u, m0, m1);
    const float S2 = fmaf(u2pcs, m0, fmaf(2.0f * u, m1, m2));
    const float g0 = m0 - S2;
    m0 = 0.5f * (S2 - S1);
    m2 = 0.5f * (S2 + S1);
    m1 = g0;
}

__host__ __device__ constexpr int order_of(int m) { return m % 3 + (m / 3) % 3 + m / 9; }

struct Moments {
    float rho, ux, uy, uz;
};

__device__ __forceinline__ Moments moments(const float (&d)[Q], const float g[3])
{
    float drho = 0.0f, jx = 0.0f, jy = 0.0f, jz = 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        drho += d[i];
        if (cx_of(i) == 1) jx += d[i];
        if (cx_of(i) == -1) jx -= d[i];
        if (cy_of(i) == 1) jy += d[i];
        if (cy_of(i) == -1) jy -= d[i];
        if (cz_of(i) == 1) jz += d[i];
        if (cz_of(i) == -1) jz -= d[i];
    }
    Moments m;
    m.rho = 1.0f + drho;
    const float ir = 1.0f / m.rho;
    m.ux = fmaf(jx, ir, 0.5f * g[0]);
    m.uy = fmaf(jy, ir, 0.5f * g[1]);
    m.uz = fmaf(jz, ir, 0.5f * g[2]);
    return m;
}

// CHM-MRT collision in deviation form.  With a = T(u) f, a_w = T(u) w (per axis (1, -u, u^2))
// and the post-collision moments a* (a*_0 = rho, first order rho g / 2 from the half-force
// forcing, a*_m = (1 - s_m) a_m for order >= 2 since a_eq = 0 there), the outgoing deviation
// is d* = T^-1(u) (a* - a_w), with a - a_w = T(u) d.
__device__ __forceinline__ void collide(float (&d)[Q], const LevelArgs& a)
{
    const Moments M = moments(d, a.g);
    const float ux = M.ux, uy = M.uy, uz = M.uz;
    const float ux2 = ux * ux, uy2 = uy * uy, uz2 = uz * uz;
    // forward T(u) d: passes along x, y, z
#pragma unroll
    for (int k = 0; k < 9; ++k) fwd3(d[3 * k], d[3 * k + 1], d[3 * k + 2], ux, ux2 - CS2);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int p = 0; p < 3; ++p) fwd3(d[p + 9 * r], d[p + 3 + 9 * r], d[p + 6 + 9 * r], uy, uy2 - CS2);
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int p = 0; p < 3; ++p) fwd3(d[p + 3 * q], d[p + 3 * q + 9], d[p + 3 * q + 18], uz, uz2 - CS2);
    // relaxation: b = a* - a_w
    const float ex[3] = {1.0f, -ux, ux2}, ey[3] = {1.0f, -uy, uy2}, ez[3] = {1.0f, -uz, uz2};
    const float s[7] = {0.0f, 0.0f, a.s2, a.s3, a.s4, a.s5, a.s6};
#pragma unroll
    for (int m = 0; m < Q; ++m) {
        const int o = order_of(m);
        if (o == 1) {
            const float gk = (m == 1) ? a.g[0] : (m == 3) ? a.g[1] : a.g[2];
            const float uk = (m == 1) ? ux : (m == 3) ? uy : uz;
            d[m] = fmaf(0.5f * M.rho, gk, uk);
        } else if (o >= 2) {
            const float aw = ex[m % 3] * ey[(m / 3) % 3] * ez[m / 9];
            d[m] = (1.0f - s[o]) * d[m] - s[o] * aw;
        }
    }
    // inverse T(u)^-1
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int p = 0; p < 3; ++p) inv3(d[p + 3 * q], d[p + 3 * q + 9], d[p + 3 * q + 18], uz, uz2 + CS2);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int p = 0; p < 3; ++p) inv3(d[p + 9 * r], d[p + 3 + 9 * r], d[p + 6 + 9 * r], uy, uy2 + CS2);
#pragma unroll
    for (int k = 0; k < 9; ++k) inv3(d[3 * k], d[3 * k + 1], d[3 * k + 2], ux, ux2 + CS2);
}

// The same collision when every third- to sixth-order rate is 1 (the default): the
// post-collision moments of order >= 3 are then their equilibrium values (zero), so the forward
// transform is needed only up to second order.  rho - 1, j and the six raw second moments of d
// come from one pass of 1-D sums (S0 = g- + g0 + g+, S1 = g+ - g-, S2 = g+ + g- along x, then
// the same along y and z); the central second moments follow from them,
//   a_200 = P_xx - 2 u_x j_x + (u_x^2 - c_s^2)(rho - 1),
//   a_110 = P_xy - u_x j_y - u_y j_x + u_x u_y (rho - 1),
// and the inverse transform is unchanged.  Same arithmetic as `collide` up to rounding order.
// Lane arithmetic of the fast collision: one cell (float) or two cells at once (float2, packed
// FP32x2 instructions of sm_100+).  Every operation is an explicit round-to-nearest add,
// multiply or fused multiply-add, and the two forms apply them in the same order, so a cell
// gives bit-identical results whichever form updates it.
struct Lane1 {
    using V = float;
    static __device__ __forceinline__ V add(V a, V b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ V sub(V a, V b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ V mul(V a, V b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __fmaf_rn(a, b, c); }
    static __device__ __forceinline__ V neg(V a) { return -a; }
    static __device__ __forceinline__ V splat(float s) { return s; }
    static __device__ __forceinline__ V rcp1p(V drho) { return 1.0f / (1.0f + drho); }
    static __device__ __forceinline__ V one_plus(V x) { return __fadd_rn(1.0f, x); }
};
struct Lane2 {
    using V = float2;
    static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
    static __device__ __forceinline__ V sub(V a, V b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
    static __device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
    static __device__ __forceinline__ V neg(V a) { return make_float2(-a.x, -a.y); }
    static __device__ __forceinline__ V splat(float s) { return make_float2(s, s); }
    static __device__ __forceinline__ V rcp1p(V drho)
    {
        return make_float2(1.0f / (1.0f + drho.x), 1.0f / (1.0f + drho.y));
    }
    static __device__ __forceinline__ V one_plus(V x) { return __fadd2_rn(make_float2(1.0f, 1.0f), x); }
};

// 1-D inverse: (m0, m1, m2) -> (g(-1), g(0), g(+1)).  DEFER leaves out the halving of
// g(+-1): the outputs at +-1 come out doubled, exactly (a power of two), and since the three
// inputs of every later 1-D inverse share one such factor, each post-collision d_i leaves the
// three passes multiplied by 2^nnz(c_i), which the store removes (Store::store_x) -- for 16-bit
// storage inside the multiply by 1/w_i that it does anyway.  Bit-identical results, two fewer
// instructions per 1-D inverse.
template <class L, bool DEFER = false>
__device__ __forceinline__ void inv3_t(typename L::V& m0, typename L::V& m1, typename L::V& m2, typename L::V u,
                                       typename L::V u2pcs, typename L::V two_u)
{
    using V = typename L::V;
    const V S1 = L::fma(u, m0, m1);
    const V S2 = L::fma(u2pcs, m0, L::fma(two_u, m1, m2));
    const V g0 = L::sub(m0, S2);
    if (DEFER) {
        m0 = L::sub(S2, S1);
        m2 = L::add(S2, S1);
    } else {
        m0 = L::mul(L::splat(0.5f), L::sub(S2, S1));
        m2 = L::mul(L::splat(0.5f), L::add(S2, S1));
    }
    m1 = g0;
}

template <class L, bool DEFER = false>
__device__ __forceinline__ void collide_fast_t(typename L::V (&d)[Q], typename L::V s2, const float g[3])
{
    using V = typename L::V;
    V S0[9], S1[9], S2[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        S2[k] = L::add(d[3 * k], d[3 * k + 2]);
        S0[k] = L::add(S2[k], d[3 * k + 1]);
        S1[k] = L::sub(d[3 * k + 2], d[3 * k]);
    }
    V T0[3], T1[3], T2[3], U0[3], U1[3], W[3];
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        T2[z] = L::add(S0[3 * z], S0[3 * z + 2]);
        T0[z] = L::add(T2[z], S0[3 * z + 1]);
        T1[z] = L::sub(S0[3 * z + 2], S0[3 * z]);
        U0[z] = L::add(L::add(S1[3 * z], S1[3 * z + 1]), S1[3 * z + 2]);
        U1[z] = L::sub(S1[3 * z + 2], S1[3 * z]);
        W[z] = L::add(L::add(S2[3 * z], S2[3 * z + 1]), S2[3 * z + 2]);
    }
    const V drho = L::add(L::add(T0[0], T0[1]), T0[2]);
    const V jz = L::sub(T0[2], T0[0]);
    const V Pzz = L::add(T0[2], T0[0]);
    const V jy = L::add(L::add(T1[0], T1[1]), T1[2]);
    const V Pyz = L::sub(T1[2], T1[0]);
    const V Pyy = L::add(L::add(T2[0], T2[1]), T2[2]);
    const V jx = L::add(L::add(U0[0], U0[1]), U0[2]);
    const V Pxz = L::sub(U0[2], U0[0]);
    const V Pxy = L::add(L::add(U1[0], U1[1]), U1[2]);
    const V Pxx = L::add(L::add(W[0], W[1]), W[2]);
    const V rho = L::one_plus(drho);
    const V ir = L::rcp1p(drho);
    const V ux = L::fma(jx, ir, L::splat(0.5f * g[0]));
    const V uy = L::fma(jy, ir, L::splat(0.5f * g[1]));
    const V uz = L::fma(jz, ir, L::splat(0.5f * g[2]));
    const V ux2 = L::mul(ux, ux), uy2 = L::mul(uy, uy), uz2 = L::mul(uz, uz);
    const V uxy = L::mul(ux, uy), uxz = L::mul(ux, uz), uyz = L::mul(uy, uz);
    const V k2 = L::sub(L::splat(1.0f), s2), ns2 = L::neg(s2);
    const V mcs = L::splat(-CS2);
    // central second moments of d (deviation form)
    const V a200 = L::fma(L::add(ux2, mcs), drho, L::fma(L::mul(L::splat(-2.0f), ux), jx, Pxx));
    const V a020 = L::fma(L::add(uy2, mcs), drho, L::fma(L::mul(L::splat(-2.0f), uy), jy, Pyy));
    const V a002 = L::fma(L::add(uz2, mcs), drho, L::fma(L::mul(L::splat(-2.0f), uz), jz, Pzz));
    const V a110 = L::fma(uxy, drho, L::fma(L::neg(ux), jy, L::fma(L::neg(uy), jx, Pxy)));
    const V a101 = L::fma(uxz, drho, L::fma(L::neg(ux), jz, L::fma(L::neg(uz), jx, Pxz)));
    const V a011 = L::fma(uyz, drho, L::fma(L::neg(uy), jz, L::fma(L::neg(uz), jy, Pyz)));
    // post-collision central moments of d: third and higher orders -w's moments (products of
    // the 1-D moments (1, -u, u^2) of the D1Q3 weights), second order relaxed
    const V ex[3] = {L::splat(1.0f), L::neg(ux), ux2}, ey[3] = {L::splat(1.0f), L::neg(uy), uy2},
            ez[3] = {L::splat(1.0f), L::neg(uz), uz2};
#pragma unroll
    for (int m = 0; m < Q; ++m) {
        const int p = m % 3, q = (m / 3) % 3, r = m / 9;
        if (p + q + r < 3) continue;
        // a product with unit factors skipped (multiplication by 1 is exact)
        V aw = ex[p];
        if (q) aw = p ? L::mul(aw, ey[q]) : ey[q];
        if (r) aw = (p || q) ? L::mul(aw, ez[r]) : ez[r];
        d[m] = L::neg(aw);
    }
    d[0] = drho;
    d[1] = L::fma(L::mul(L::splat(0.5f), rho), L::splat(g[0]), ux);
    d[3] = L::fma(L::mul(L::splat(0.5f), rho), L::splat(g[1]), uy);
    d[9] = L::fma(L::mul(L::splat(0.5f), rho), L::splat(g[2]), uz);
    d[2] = L::fma(k2, a200, L::mul(ns2, ux2));
    d[6] = L::fma(k2, a020, L::mul(ns2, uy2));
    d[18] = L::fma(k2, a002, L::mul(ns2, uz2));
    d[4] = L::fma(k2, a110, L::mul(ns2, uxy));
    d[10] = L::fma(k2, a101, L::mul(ns2, uxz));
    d[12] = L::fma(k2, a011, L::mul(ns2, uyz));
    // inverse T(u)^-1: z, then y, then x
    const V zc = L::add(uz2, L::splat(CS2)), yc = L::add(uy2, L::splat(CS2)), xc = L::add(ux2, L::splat(CS2));
    const V z2 = L::mul(L::splat(2.0f), uz), y2 = L::mul(L::splat(2.0f), uy), x2 = L::mul(L::splat(2.0f), ux);
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int p = 0; p < 3; ++p) inv3_t<L, DEFER>(d[p + 3 * q], d[p + 3 * q + 9], d[p + 3 * q + 18], uz, zc, z2);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int p = 0; p < 3; ++p) inv3_t<L, DEFER>(d[p + 9 * r], d[p + 3 + 9 * r], d[p + 6 + 9 * r], uy, yc, y2);
#pragma unroll
    for (int k = 0; k < 9; ++k) inv3_t<L, DEFER>(d[3 * k], d[3 * k + 1], d[3 * k + 2], ux, xc, x2);
}

// The fast collision of one cell with packed FP32x2 instructions inside the cell: the 1-D
// sums along x and then y run on the z = -1 and z = +1 rows as pairs (their z = 0 rows alone),
// and the inverse passes along z and then y on the x = -1 and x = +1 columns as pairs (x = 0
// alone); the final pass along x mixes the members of a pair and stays scalar.  Every element
// sees the operations of collide_fast_t<Lane1> in the same order, so results are bit-identical.
template <bool DEFER = false>
__device__ __forceinline__ void collide_fast_p(float (&d)[Q], float s2, const float g[3])
{
    using L = Lane1;
    using P = Lane2;
    // x sums of row k = q + 3 r; index q, .x the row at r = 0 (k = q), .y the row at r = 2 (k = q + 6)
    float2 S0p[3], S1p[3], S2p[3];
    float S0m[3], S1m[3], S2m[3];  // rows at r = 1 (k = q + 3)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int k0 = q, k2 = q + 6, k1 = q + 3;
        const float2 gm = make_float2(d[3 * k0], d[3 * k2]), g0 = make_float2(d[3 * k0 + 1], d[3 * k2 + 1]),
                     gp = make_float2(d[3 * k0 + 2], d[3 * k2 + 2]);
        S2p[q] = P::add(gm, gp);
        S0p[q] = P::add(S2p[q], g0);
        S1p[q] = P::sub(gp, gm);
        S2m[q] = L::add(d[3 * k1], d[3 * k1 + 2]);
        S0m[q] = L::add(S2m[q], d[3 * k1 + 1]);
        S1m[q] = L::sub(d[3 * k1 + 2], d[3 * k1]);
    }
    // y sums at z = -1 and z = +1 (pairs) and z = 0
    const float2 T2p = P::add(S0p[0], S0p[2]);
    const float2 T0p = P::add(T2p, S0p[1]);
    const float2 T1p = P::sub(S0p[2], S0p[0]);
    const float2 U0p = P::add(P::add(S1p[0], S1p[1]), S1p[2]);
    const float2 U1p = P::sub(S1p[2], S1p[0]);
    const float2 Wp = P::add(P::add(S2p[0], S2p[1]), S2p[2]);
    const float T2m = L::add(S0m[0], S0m[2]);
    const float T0m = L::add(T2m, S0m[1]);
    const float T1m = L::sub(S0m[2], S0m[0]);
    const float U0m = L::add(L::add(S1m[0], S1m[1]), S1m[2]);
    const float U1m = L::sub(S1m[2], S1m[0]);
    const float Wm = L::add(L::add(S2m[0], S2m[1]), S2m[2]);
    const float T0[3] = {T0p.x, T0m, T0p.y}, T1[3] = {T1p.x, T1m, T1p.y}, T2[3] = {T2p.x, T2m, T2p.y};
    const float U0[3] = {U0p.x, U0m, U0p.y}, U1[3] = {U1p.x, U1m, U1p.y}, W[3] = {Wp.x, Wm, Wp.y};
    const float drho = L::add(L::add(T0[0], T0[1]), T0[2]);
    const float jz = L::sub(T0[2], T0[0]);
    const float Pzz = L::add(T0[2], T0[0]);
    const float jy = L::add(L::add(T1[0], T1[1]), T1[2]);
    const float Pyz = L::sub(T1[2], T1[0]);
    const float Pyy = L::add(L::add(T2[0], T2[1]), T2[2]);
    const float jx = L::add(L::add(U0[0], U0[1]), U0[2]);
    const float Pxz = L::sub(U0[2], U0[0]);
    const float Pxy = L::add(L::add(U1[0], U1[1]), U1[2]);
    const float Pxx = L::add(L::add(W[0], W[1]), W[2]);
    const float rho = L::one_plus(drho);
    const float ir = L::rcp1p(drho);
    const float ux = L::fma(jx, ir, 0.5f * g[0]);
    const float uy = L::fma(jy, ir, 0.5f * g[1]);
    const float uz = L::fma(jz, ir, 0.5f * g[2]);
    const float ux2 = L::mul(ux, ux), uy2 = L::mul(uy, uy), uz2 = L::mul(uz, uz);
    const float uxy = L::mul(ux, uy), uxz = L::mul(ux, uz), uyz = L::mul(uy, uz);
    const float k2 = L::sub(1.0f, s2), ns2 = L::neg(s2);
    const float mcs = -CS2;
    const float a200 = L::fma(L::add(ux2, mcs), drho, L::fma(L::mul(-2.0f, ux), jx, Pxx));
    const float a020 = L::fma(L::add(uy2, mcs), drho, L::fma(L::mul(-2.0f, uy), jy, Pyy));
    const float a002 = L::fma(L::add(uz2, mcs), drho, L::fma(L::mul(-2.0f, uz), jz, Pzz));
    const float a110 = L::fma(uxy, drho, L::fma(L::neg(ux), jy, L::fma(L::neg(uy), jx, Pxy)));
    const float a101 = L::fma(uxz, drho, L::fma(L::neg(ux), jz, L::fma(L::neg(uz), jx, Pxz)));
    const float a011 = L::fma(uyz, drho, L::fma(L::neg(uy), jz, L::fma(L::neg(uz), jy, Pyz)));
    const float ex[3] = {1.0f, L::neg(ux), ux2}, ey[3] = {1.0f, L::neg(uy), uy2}, ez[3] = {1.0f, L::neg(uz), uz2};
#pragma unroll
    for (int m = 0; m < Q; ++m) {
        const int p = m % 3, q = (m / 3) % 3, r = m / 9;
        if (p + q + r < 3) continue;
        float aw = ex[p];
        if (q) aw = p ? L::mul(aw, ey[q]) : ey[q];
        if (r) aw = (p || q) ? L::mul(aw, ez[r]) : ez[r];
        d[m] = L::neg(aw);
    }
    d[0] = drho;
    d[1] = L::fma(L::mul(0.5f, rho), g[0], ux);
    d[3] = L::fma(L::mul(0.5f, rho), g[1], uy);
    d[9] = L::fma(L::mul(0.5f, rho), g[2], uz);
    d[2] = L::fma(k2, a200, L::mul(ns2, ux2));
    d[6] = L::fma(k2, a020, L::mul(ns2, uy2));
    d[18] = L::fma(k2, a002, L::mul(ns2, uz2));
    d[4] = L::fma(k2, a110, L::mul(ns2, uxy));
    d[10] = L::fma(k2, a101, L::mul(ns2, uxz));
    d[12] = L::fma(k2, a011, L::mul(ns2, uyz));
    const float zc = L::add(uz2, CS2), yc = L::add(uy2, CS2), xc = L::add(ux2, CS2);
    const float z2 = L::mul(2.0f, uz), y2 = L::mul(2.0f, uy), x2 = L::mul(2.0f, ux);
    // inverse along z: columns (p, q) with p = 0 and p = 2 as pairs
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        float2 m0 = make_float2(d[3 * q], d[3 * q + 2]), m1 = make_float2(d[3 * q + 9], d[3 * q + 11]),
               m2 = make_float2(d[3 * q + 18], d[3 * q + 20]);
        inv3_t<P, DEFER>(m0, m1, m2, P::splat(uz), P::splat(zc), P::splat(z2));
        d[3 * q] = m0.x, d[3 * q + 2] = m0.y, d[3 * q + 9] = m1.x, d[3 * q + 11] = m1.y;
        d[3 * q + 18] = m2.x, d[3 * q + 20] = m2.y;
        inv3_t<L, DEFER>(d[3 * q + 1], d[3 * q + 10], d[3 * q + 19], uz, zc, z2);
    }
    // inverse along y: columns (p, r), the same pairs
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        float2 m0 = make_float2(d[9 * r], d[9 * r + 2]), m1 = make_float2(d[9 * r + 3], d[9 * r + 5]),
               m2 = make_float2(d[9 * r + 6], d[9 * r + 8]);
        inv3_t<P, DEFER>(m0, m1, m2, P::splat(uy), P::splat(yc), P::splat(y2));
        d[9 * r] = m0.x, d[9 * r + 2] = m0.y, d[9 * r + 3] = m1.x, d[9 * r + 5] = m1.y;
        d[9 * r + 6] = m2.x, d[9 * r + 8] = m2.y;
        inv3_t<L, DEFER>(d[9 * r + 1], d[9 * r + 4], d[9 * r + 7], uy, yc, y2);
    }
    // inverse along x: rows, scalar
#pragma unroll
    for (int k = 0; k < 9; ++k) inv3_t<L, DEFER>(d[3 * k], d[3 * k + 1], d[3 * k + 2], ux, xc, x2);
}

template <bool DEFER = false>
__device__ __forceinline__ void collide_fast(float (&d)[Q], const LevelArgs& a)
{
    collide_fast_p<DEFER>(d, a.s2, a.g);
}

// The classical operators the paper compares against (Sec. 2.1.2), with the second-order
// equilibrium f_eq2_i = w_i rho [1 + 3 c.u + 4.5 (c.u)^2 - 1.5 u.u] and the second-order (Guo)
// force term F_i = w_i [3 (c - u) + 9 (c.u) c] . F, F = rho g, u = j / rho + g / 2.
// TRT: the even and odd parts of each pair (i, opp(i)) relax with a.s2 and a.wm; the even and
// odd parts of F_i are scaled by (1 - s2/2) and (1 - wm/2).  SRT2 is the case wm = s2.
// Deviation form throughout: with d = f - w, f_eq2 - w = w [(rho - 1) + rho (3 c.u + 4.5 (c.u)^2
// - 1.5 u.u)], so the O(1) weights never enter a rounding.  The FP32 weights are not exact:
// sum_i w_i and sum_i 3 w_i c_i c_i differ from 1 and the identity by ~3e-8, so relaxing toward
// f_eq2 would create mass omega * 3e-8 * (rho - 1) and momentum omega * 3e-8 * rho u every step
// (a systematic drift that grows with time, unlike rounding).  The post-collision mass and
// momentum are therefore restored to their exact values rho and j + F: mass through the rest
// population, momentum through the three face pairs (each pair's difference carries one axis
// and leaves the mass unchanged).
template <bool TRT>
__device__ __forceinline__ void collide_trt2(float (&d)[Q], const LevelArgs& a)
{
    float drho = 0.0f, jx = 0.0f, jy = 0.0f, jz = 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        drho += d[i];
        if (cx_of(i)) jx += cx_of(i) > 0 ? d[i] : -d[i];
        if (cy_of(i)) jy += cy_of(i) > 0 ? d[i] : -d[i];
        if (cz_of(i)) jz += cz_of(i) > 0 ? d[i] : -d[i];
    }
    const float rho = 1.0f + drho, ir = 1.0f / rho;
    const float ux = fmaf(jx, ir, 0.5f * a.g[0]), uy = fmaf(jy, ir, 0.5f * a.g[1]), uz = fmaf(jz, ir, 0.5f * a.g[2]);
    const float Fx = rho * a.g[0], Fy = rho * a.g[1], Fz = rho * a.g[2];
    const float uu15 = 1.5f * (ux * ux + uy * uy + uz * uz);
    const float uF3 = 3.0f * (ux * Fx + uy * Fy + uz * Fz);
    const float wp = a.s2, wm = TRT ? a.wm : a.s2;
    const float kp = 1.0f - 0.5f * wp, km = 1.0f - 0.5f * wm;
    {  // rest population: even only
        constexpr float w = w_of(13);
        const float peq = w * (drho - rho * uu15);
        d[13] = d[13] - wp * (d[13] - peq) - kp * w * uF3;
    }
#pragma unroll
    for (int i = 0; i < 13; ++i) {
        const int o = Q - 1 - i;
        const float w = w_of(i);
        const float cu = (float)cx_of(i) * ux + (float)cy_of(i) * uy + (float)cz_of(i) * uz;
        const float cF = (float)cx_of(i) * Fx + (float)cy_of(i) * Fy + (float)cz_of(i) * Fz;
        const float peq = w * (drho + rho * (4.5f * cu * cu - uu15));
        const float meq = w * rho * 3.0f * cu;
        const float Fe = w * (9.0f * cu * cF - uF3), Fo = w * 3.0f * cF;
        const float p = 0.5f * (d[i] + d[o]), m = 0.5f * (d[i] - d[o]);
        const float ev = kp * Fe - wp * (p - peq), od = km * Fo - wm * (m - meq);
        d[i] = d[i] + ev + od;
        d[o] = d[o] + ev - od;
    }
    float pm = 0.0f, px = 0.0f, py = 0.0f, pz = 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        pm += d[i];
        if (cx_of(i)) px += cx_of(i) > 0 ? d[i] : -d[i];
        if (cy_of(i)) py += cy_of(i) > 0 ? d[i] : -d[i];
        if (cz_of(i)) pz += cz_of(i) > 0 ? d[i] : -d[i];
    }
    // face pairs (-x, +x) = (12, 14), (-y, +y) = (10, 16), (-z, +z) = (4, 22)
    const float hx = 0.5f * ((jx + Fx) - px), hy = 0.5f * ((jy + Fy) - py), hz = 0.5f * ((jz + Fz) - pz);
    d[14] += hx;
    d[12] -= hx;
    d[16] += hy;
    d[10] -= hy;
    d[22] += hz;
    d[4] -= hz;
    d[13] += drho - pm;
}

// DEFER (the default rates only): d leaves with the factors 2^nnz(c_i), for Store::store_x
template <int COLL, bool DEFER = false>
__device__ __forceinline__ void collide_model(float (&d)[Q], const LevelArgs& a)
{
    static_assert(!DEFER || COLL == COLL_CHM_FAST, "deferred halving is a form of the fast collision");
    if (COLL == COLL_CHM_FAST) collide_fast<DEFER>(d, a);
    else if (COLL == COLL_CHM) collide(d, a);
    else collide_trt2<COLL == COLL_TRT2>(d, a);
}

// A cell's own second-order rate s2 (an absorbing layer): SRT2 relaxes both parities with it,
// TRT2 derives its odd rate from it through Lambda.
template <int COLL>
__device__ __forceinline__ void set_own_rate(LevelArgs& la, float s2)
{
    la.s2 = s2;
    if (COLL == COLL_SRT2) la.wm = s2;
    if (COLL == COLL_TRT2) la.wm = 1.0f / (la.magic / (1.0f / s2 - 0.5f) + 0.5f);
}

// ------------------------------------------------------------------------------ gather (read-only)
// Populations of level n of one fluid cell, for the export and diagnostics kernels.  These are programmatic
// dependents of the step before them: their index tables load while it drains (pdl_wait is in here).
template <int ST, int SCHEME>
__device__ __forceinline__ void gather(const DomainView& v, const void* src, uint32_t slot, uint32_t word,
                                       const LevelArgs& a, float (&d)[Q])
{
    const uint32_t wm = word & WORD_WALL_MASK;
    const uint32_t n = (uint32_t)v.n_slots;
    const int32_t aux = __ldg(v.aux + slot);
    if (SCHEME == LBM_SCHEME_ESOTERIC) {
        uint32_t cs[8];
        corner_slots(v.nb8 + (slot / BRICK_CELLS) * 8, slot, cs);
        pdl_wait();
        fetch_et<ST>(src, n, cs, wm, a.parity, d);
    } else {
        fetch_ab<ST>(src, n, v.nbr + (slot / BRICK_CELLS) * Q, slot, wm, d);
    }
    if (wm) wall_rules<ST, SCHEME>(v, src, slot, word, a, d, aux);
}

// ------------------------------------------------------------------------------ kernels
// Rounds of links a warp holds in registers: six cover every run of the vessels, so no warp of a small
// domain, whose step is as long as its slowest warp, waits for the reloading loop (25 k cells: 6.5 -> 5.3 us,
// 150 k: 10.3 -> 9.5 us against three); on a large domain (LARGE_BRICKS) the warps hide one another's latency and the fewer
// registers win (2.7 M cells, 45 k bricks: 124 us with three, 129 us with six; 11 k bricks: 26.0 and 26.9 us).
constexpr int LINK_ROUNDS = 6, LINK_ROUNDS_LARGE = 3;

// Bouzidi links of a warp's cells, shared out among its lanes: the links of a half-brick are one run of the
// packed list, so a lane takes entry k0 + lane, + 32, ...: code and coefficient (coalesced, before
// pdl_wait: they never change), f*_a of the q >= 1/2 links (coalesced from the side buffer).  The cells'
// values go through the warp's exchange area, sm[i * STRIDE + cell]: Bouzidi cells put their 27 values there,
// the lanes apply their links in place (a link writes f_a and reads f_b only if b has no link, so the
// order does not matter), and the cells take them back; after the collision the cells put their stored
// values there, from which the lanes keep f*_a.  About 60 instructions a cell and 25 per 32 links, and one
// memory latency, against 27 directions x (test, position, two predicated loads, mix) in three groups
// of a latency each when every cell handled its own links; a boundary half-brick has 50 to 100 links.
// Per step, each cell by itself -> this: 256^3 aneurysm FP32 11.9 -> 9.9 us, 2.7 M cell Bouzidi pipe 133.5 ->
// 122.6 us, 25 k cell TRT aneurysm 7.7 -> 5.3 us, batch of 8 FP16 aneurysms 19.3 -> 15.6 us (with the closure
// by face above and the register budget of large domains).
// R: rounds of 32 links held in registers, in groups of three whose exchange reads come before their writes
// (one shared-memory latency a group); longer runs reload their codes, a memory latency each.  On the synthetic
// vessels a half-brick with links has 70 on average, up to 183, a fifth of them over 96 (LINK_ROUNDS).
template <int ST, int SCHEME, int STRIDE, int R>
struct BouzidiLinks {
    static constexpr int G = 3;
    static_assert(R % G == 0, "whole groups");
    uint32_t k0, k1, lane;
    uint32_t code[(R + 1) / 2];  // two 16-bit codes each
    float coef[R], fa[R];

    __device__ __forceinline__ bool any() const { return k0 < k1; }
    __device__ __forceinline__ bool round(int r) const { return k0 + 32u * r < k1; }  // the same in every lane
    __device__ __forceinline__ uint32_t code_of(int r) const { return (code[r / 2] >> (16 * (r & 1))) & 0xffffu; }
    __device__ __forceinline__ uint32_t load_code(const DomainView& v, uint32_t k) const
    {
        return k < k1 && LBM_IN_RANGE(k, v.n_bq, 5) ? (uint32_t)__ldg(v.blink + k) : 0u;
    }
    __device__ __forceinline__ float load_coef(const DomainView& v, uint32_t k) const
    {
        return k < k1 && LBM_IN_RANGE(k, v.n_bq, 5) ? __ldg(v.bq + k) : 0.0f;
    }
    // the run's bounds, then (prefetch) its codes and coefficients: the bounds are loaded beside the warp's other
    // tables, so that the branch on them does not hold those back
    __device__ __forceinline__ void begin(const DomainView& v, uint32_t half_brick, uint32_t lane_)
    {
        lane = lane_;
        k0 = k1 = 0u;
        if (v.bstart) {
            k0 = (uint32_t)__ldg(v.bstart + half_brick);
            k1 = (uint32_t)__ldg(v.bstart + half_brick + 1);
        }
    }
    __device__ __forceinline__ void prefetch(const DomainView& v)
    {
#pragma unroll
        for (int r = 0; r < R; ++r) coef[r] = 0.0f;
#pragma unroll
        for (int r = 0; r < (R + 1) / 2; ++r) code[r] = 0u;
#pragma unroll
        for (int r = 0; r < R; r += 2) {
            if (!round(r)) break;  // the warps without links skip all of it
            const uint32_t k = k0 + 32u * r + lane;
            code[r / 2] = load_code(v, k);
            coef[r] = load_coef(v, k);
            if (r + 1 < R) {
                code[r / 2] |= load_code(v, k + 32u) << 16;
                coef[r + 1] = load_coef(v, k + 32u);
            }
        }
    }
    // f*_a of a q >= 1/2 link, as stored
    __device__ __forceinline__ float load_fa(const DomainView& v, const void* src, uint32_t slot0, uint32_t k, uint32_t c,
                                             float b) const
    {
        if (!(b < 0.0f)) return 0.0f;
        if (SCHEME == LBM_SCHEME_ESOTERIC) return Store<ST>::load_rw_h(v.side, k);
        const uint32_t off = ((c >> 5) & 31u) * (uint32_t)v.n_slots + slot0 + (c & 31u);
        return LBM_IN_RANGE(off, (uint64_t)Q * (uint64_t)v.n_slots, 1) ? Store<ST>::load_rw_h(src, off) : 0.0f;
    }
    __device__ __forceinline__ void issue(const DomainView& v, const void* src, uint32_t slot0)
    {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r % 2 == 0 && !round(r)) break;
            fa[r] = load_fa(v, src, slot0, k0 + 32u * r + lane, code_of(r), coef[r]);
        }
    }
    static __device__ __forceinline__ uint32_t at(uint32_t c) { return ((c >> 5) & 31u) * STRIDE + (c & 31u); }
    // whether the link changes its value (past the end, halfway bounce-back, walls on both sides: no)
    static __device__ __forceinline__ bool active(uint32_t c, float b) { return b < 0.0f || (b > 0.0f && !(c & (1u << 10))); }
    static __device__ __forceinline__ float mix(uint32_t c, float b, float f, float other)
    {
        if (b > 0.0f) return wall_low(b, f, other);
        // 16-bit storages: w = w_of(13) 4^-nnz, the same float as w_of of the direction
        const float w = Store<ST>::SCALED ? __int_as_float(__float_as_int(w_of(13)) - (int)(((c >> 11) & 3u) << 24)) : 1.0f;
        return wall_high(-b, f, Store<ST>::SCALED ? __fmul_rn(w, other) : other);
    }
    static __device__ __forceinline__ float other_value(uint32_t c, float b, float fa_, const float* sm)
    {
        return b < 0.0f ? fa_ : sm[(Q - 1 - ((c >> 5) & 31u)) * STRIDE + (c & 31u)];
    }
    __device__ __forceinline__ void apply(const DomainView& v, const void* src, uint32_t slot0, float* sm)
    {
        __syncwarp();
#pragma unroll
        for (int g = 0; g < R; g += G) {
            if (!round(g)) break;
            float f[G], o[G];
#pragma unroll
            for (int r = 0; r < G; ++r) {
                const uint32_t c = code_of(g + r);
                if (active(c, coef[g + r])) {
                    f[r] = sm[at(c)];
                    o[r] = other_value(c, coef[g + r], fa[g + r], sm);
                }
            }
#pragma unroll
            for (int r = 0; r < G; ++r) {
                const uint32_t c = code_of(g + r);
                if (active(c, coef[g + r])) sm[at(c)] = mix(c, coef[g + r], f[r], o[r]);
            }
        }
        for (uint32_t k = k0 + 32u * R + lane; k < k1; k += 32u) {
            const uint32_t c = load_code(v, k);
            const float b = load_coef(v, k);
            if (active(c, b)) sm[at(c)] = mix(c, b, sm[at(c)], other_value(c, b, load_fa(v, src, slot0, k, c, b), sm));
        }
        __syncwarp();
    }
    __device__ __forceinline__ void keep(const DomainView& v, const float* sm) const
    {
        __syncwarp();
#pragma unroll
        for (int g = 0; g < R; g += G) {
            if (!round(g)) break;
            float f[G];
#pragma unroll
            for (int r = 0; r < G; ++r)
                if (coef[g + r] < 0.0f) f[r] = sm[at(code_of(g + r))];
#pragma unroll
            for (int r = 0; r < G; ++r)
                if (coef[g + r] < 0.0f) Store<ST>::store_h(v.side, k0 + 32u * (g + r) + lane, f[r]);
        }
        for (uint32_t k = k0 + 32u * R + lane; k < k1; k += 32u)
            if (load_coef(v, k) < 0.0f) Store<ST>::store_h(v.side, k, sm[at(load_code(v, k))]);
    }
};

// One fused update of the cell at `slot` (a lane of a warp that covers half of one brick; all
// 32 lanes must call it together: the neighbour row goes round by shuffle, the Bouzidi links are shared
// out).  PDL: the kernel is launched as a programmatic dependent (not the persistent batch).  LINKS: the rounds
// of BouzidiLinks, 0 for a domain without Bouzidi cells; else sm is the warp's [27][32] exchange area.
template <int ST, int SCHEME, int COLL, int PC = -1, bool PDL = true, int LINKS = LINK_ROUNDS>
__device__ __forceinline__ void step_cell(const DomainView& v, const void* src, void* dst, const LevelArgs& a,
                                          uint32_t slot, uint32_t lane, float* sm)
{
    constexpr bool X = COLL == COLL_CHM_FAST;  // deferred halving in the inverse transform
    constexpr bool TWIST = SCHEME == LBM_SCHEME_ESOTERIC;
    const uint32_t brick = slot / BRICK_CELLS;
    const uint32_t word = __ldg(v.word + slot);
    // the cell's record, loaded beside its word rather than after it: an open cell then waits for one
    // memory latency fewer (4 bytes per slot of traffic)
    const int32_t auxv = __ldg(v.aux + slot);
    BouzidiLinks<ST, SCHEME, 32, LINKS ? LINKS : 3> links;
    if (LINKS) links.begin(v, slot / 32u, lane);
    const bool fluid = (word & WORD_FLUID) != 0u;
    const bool bouzidi = ((word >> WORD_KIND_SHIFT) & 3u) == KIND_BOUZIDI;
    const uint32_t wm = word & WORD_WALL_MASK;
    const uint32_t n = (uint32_t)v.n_slots, slot0 = slot - lane;
    float d[Q];
    uint32_t cs[8];
    LevelArgs la = a;
    if (word & WORD_OWN_TAU) set_own_rate<COLL>(la, __ldg(v.s2_cell + slot));
    if (TWIST) {
        const int32_t row = __ldg(v.nb8 + brick * 8u + (lane & 7u));
        corner_slots_shfl(row, slot, cs);
        const bool clean = PC >= 0 && __all_sync(0xffffffffu, wm == 0u);
        if (LINKS) links.prefetch(v);
        if (PDL) pdl_wait();
        if (fluid) fetch_et<ST, PC>(dst, n, cs, wm, a.parity, d, clean);
    } else {
        const int32_t row = __ldg(v.nbr + brick * (uint32_t)Q + (lane < (uint32_t)Q ? lane : 0u));
        constexpr int G = ab_group<ST, COLL, LINKS>();
        uint32_t off[Q];
        if (G == Q)
#pragma unroll
            for (int i = 0; i < Q; ++i) off[i] = ab_offset_shfl(n, row, slot, wm, i);
        if (LINKS) links.prefetch(v);
        if (PDL) pdl_wait();
        if (G == Q) {
            if (fluid) fetch_ab_at<ST>(src, n, off, d);
        } else {
#pragma unroll
            for (int g = 0; g < Q; g += G) {
#pragma unroll
                for (int j = 0; j < G; ++j) off[g + j] = ab_offset_shfl(n, row, slot, wm, g + j);
                if (fluid)
#pragma unroll
                    for (int j = 0; j < G; ++j)
                        d[g + j] = LBM_IN_RANGE(off[g + j], (uint64_t)Q * n, 1) ? Store<ST>::load_rw_h(src, off[g + j]) : 0.0f;
            }
            if (fluid) scale_in<ST>(d);
        }
    }
    if (LINKS && links.any()) {
        links.issue(v, src, slot0);
        if (bouzidi)
#pragma unroll
            for (int i = 0; i < Q; ++i) sm[i * 32 + lane] = d[i];
        links.apply(v, src, slot0, sm);
        if (bouzidi)
#pragma unroll
            for (int i = 0; i < Q; ++i) d[i] = sm[i * 32 + lane];
    }
    if (fluid) {
        open_rules(v, word, auxv, a, d);
        collide_model<COLL, X>(d, la);
        scale_out<ST, X>(d);
        if (TWIST) {
            store_et<ST, PC, X, true>(dst, n, cs, a.parity, d);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (LBM_IN_RANGE((uint32_t)i * n + slot, (uint64_t)Q * n, 4)) Store<ST>::store_h(dst, (uint32_t)i * n + slot, d[i]);
        }
    }
    if (LINKS && TWIST && links.any()) {
        if (bouzidi)
#pragma unroll
            for (int i = 0; i < Q; ++i) sm[i * 32 + lane] = d[i];
        links.keep(v, sm);
    }
}

// The block's place in the sweep over the bricks.  Where the state outgrows what L2 keeps, odd levels sweep backwards: a
// step then begins with the bricks that the step before it touched last, which L2 still holds; in one fixed order
// such a state evicts itself before it comes round again.  The line is measured, half of this GPU's 126 MB of L2
// (two partitions).  us a step, one order -> backwards on odd levels:
//   twist FP32  42 MB 12.2 -> 12.4   64 MB 17.5 -> 17.5   85 MB 23.2 -> 23.1 (with links 24.5 -> 24.1)   106 MB 32.4 -> 29.7
//               132 MB 44.2 -> 38.1   321 MB 117.3 -> 110.5;   FP16  66 MB 27.7 -> 27.7   161 MB 88.9 -> 84.3
//   A-B FP32    73 MB 12.5 -> 12.0   109 MB 22.3 -> 19.2   145 MB 27.8 -> 26.7   591 MB 109.4 -> 109.0
//       FP16    54 MB 16.7 -> 16.7   73 MB 22.4 -> 21.9   180 MB 61.6 -> 59.5   296 MB 98.2 -> 96.3
constexpr int64_t SWEEP_BYTES = (int64_t)64 << 20;
__device__ __forceinline__ uint32_t sweep_block(int backwards) { return backwards ? gridDim.x - 1u - blockIdx.x : blockIdx.x; }
template <int ST, int SCHEME>
LevelArgs with_sweep(const DomainView& v, LevelArgs a)
{
    const int64_t arrays = SCHEME == LBM_SCHEME_ESOTERIC ? 1 : 2;
    const int64_t bytes = arrays * Q * v.n_slots * (int64_t)sizeof(typename Store<ST>::T);
    a.backwards = (a.parity & 1) && bytes > SWEEP_BYTES;
    return a;
}

template <int ST, int SCHEME, int BRICKS, int MINB, int COLL, int PC = -1, int LINKS = LINK_ROUNDS>
__global__ void __launch_bounds__(BRICKS * BRICK_CELLS, MINB)
    k_step(DomainView v, const void* src, void* dst, LevelArgs a)
{
    __shared__ float sm[LINKS ? BRICKS * 2 : 1][LINKS ? Q * 32 : 1];
    pdl_trigger();
    const uint32_t slot = sweep_block(a.backwards) * (uint32_t)(BRICKS * BRICK_CELLS) + threadIdx.x;
    // the active slots are a multiple of 64, so this exit is taken by whole warps
    if (slot >= (uint32_t)(v.n_bricks * BRICK_CELLS)) return;
    step_cell<ST, SCHEME, COLL, PC, true, LINKS>(v, src, dst, a, slot, threadIdx.x & 31u, sm[LINKS ? threadIdx.x >> 5 : 0]);
}

// Esoteric-twist step with two cells per thread: lane l of a warp updates cells l and l + 32 of
// one brick (its lower and upper halves along z), and their collisions run as one stream of packed
// FP32x2 instructions (the default rates only), which halves the issue slots of the arithmetic;
// loads, wall rules and stores stay per cell.  A warp covers one brick, so the brick's corner
// row still goes round by shuffle.  Results are bit-identical to the one-cell kernels.
template <int ST, int PC>
__device__ __forceinline__ void store_twist_cell(const DomainView& v, void* pop, const LevelArgs& a, uint32_t word,
                                                 int32_t aux, const uint32_t (&cs)[8], uint32_t half,
                                                 const float (&d)[Q])
{
    store_et<ST, PC, true, true>(pop, (uint32_t)v.n_slots, cs, a.parity, d);
    if (half) {
        const uint32_t off = (uint32_t)aux;
        const uint32_t wm = word & WORD_WALL_MASK;
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if ((half & (1u << i)) && LBM_IN_RANGE(link_index(off, wm, i), v.n_bq, 5))
                Store<ST>::store_h(v.side, link_index(off, wm, i), d[i]);
    }
}

template <int ST, int BRICKS, int MINB, int PC>
__global__ void __launch_bounds__(BRICKS * 32, MINB)
    k_step2(DomainView v, void* pop, LevelArgs a)
{
    pdl_trigger();
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t brick = sweep_block(a.backwards) * (uint32_t)BRICKS + (threadIdx.x >> 5);
    if (brick >= (uint32_t)v.n_bricks) return;  // whole warps
    const uint32_t n = (uint32_t)v.n_slots;
    const uint32_t slotA = brick * BRICK_CELLS + lane, slotB = slotA + 32u;
    const int32_t row = __ldg(v.nb8 + brick * 8u + (lane & 7u));
    uint32_t csA[8], csB[8];
    corner_slots_shfl(row, slotA, csA);
    corner_slots_shfl(row, slotB, csB);
    const uint32_t wA = __ldg(v.word + slotA), wB = __ldg(v.word + slotB);
    const int32_t xA = __ldg(v.aux + slotA), xB = __ldg(v.aux + slotB);  // records, beside the words
    const bool fA = (wA & WORD_FLUID) != 0u, fB = (wB & WORD_FLUID) != 0u;
    const bool clean = PC >= 0 && __all_sync(0xffffffffu, ((wA | wB) & WORD_WALL_MASK) == 0u);
    pdl_wait();
    if (!fA && !fB) return;
    float dA[Q], dB[Q];
    if (fA) fetch_et<ST, PC>(pop, n, csA, wA & WORD_WALL_MASK, a.parity, dA, clean);
    if (fB) fetch_et<ST, PC>(pop, n, csB, wB & WORD_WALL_MASK, a.parity, dB, clean);
    const uint32_t halfA =
        (fA && (wA & WORD_WALL_MASK)) ? wall_rules<ST, LBM_SCHEME_ESOTERIC>(v, nullptr, slotA, wA, a, dA, xA) : 0u;
    const uint32_t halfB =
        (fB && (wB & WORD_WALL_MASK)) ? wall_rules<ST, LBM_SCHEME_ESOTERIC>(v, nullptr, slotB, wB, a, dB, xB) : 0u;
    const float s2A = (wA & WORD_OWN_TAU) ? __ldg(v.s2_cell + slotA) : a.s2;
    const float s2B = (wB & WORD_OWN_TAU) ? __ldg(v.s2_cell + slotB) : a.s2;
    float2 d2[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) d2[i] = make_float2(fA ? dA[i] : 0.0f, fB ? dB[i] : 0.0f);  // a solid lane: rest
    collide_fast_t<Lane2, true>(d2, make_float2(s2A, s2B), a.g);
    scale_out2<ST, true>(d2);  // the store factors of both cells, one packed multiply per direction
    if (fA) {
#pragma unroll
        for (int i = 0; i < Q; ++i) dA[i] = d2[i].x;
        store_twist_cell<ST, PC>(v, pop, a, wA, xA, csA, halfA, dA);
    }
    if (fB) {
#pragma unroll
        for (int i = 0; i < Q; ++i) dB[i] = d2[i].y;
        store_twist_cell<ST, PC>(v, pop, a, wB, xB, csB, halfB, dB);
    }
}

// Software-pipelined persistent variant of the FP32 esoteric-twist step.  Each CTA walks over
// chunks of BRICKS bricks; before computing chunk c, every thread issues cp.async copies of the
// 27 populations its cell of chunk c + gridDim will read (shared memory, one stage per chunk,
// two stages), so that the next cell's loads are in flight during the current cell's
// arithmetic without holding registers.  Each thread copies and reads only its own staging
// slots, so no CTA barrier is needed; and every location of the in-place array is owned by one
// cell, so prefetching another cell's locations before this cell's stores cannot race.
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem)
{
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_one() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

template <int BRICKS, int MINB, int COLL>
__global__ void __launch_bounds__(BRICKS * BRICK_CELLS, MINB)
    k_step_et_pipe(DomainView v, float* __restrict__ pop, LevelArgs a)
{
    constexpr int T = BRICKS * BRICK_CELLS;
    pdl_trigger();
    pdl_wait();
    extern __shared__ float stage[];  // [2][27][T]
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const uint32_t n = (uint32_t)v.n_slots;
    const int64_t n_chunks = (v.n_bricks + BRICKS - 1) / BRICKS;
    // issue the copies of chunk c into stage st (all lanes run the shuffles)
    auto prefetch = [&](int64_t c, int st) {
        const uint32_t slot = (uint32_t)(c * T) + tid;
        if (slot < (uint32_t)(v.n_bricks * BRICK_CELLS)) {
            const uint32_t word = __ldg(v.word + slot);
            const int32_t row = __ldg(v.nb8 + (slot / BRICK_CELLS) * 8u + (lane & 7u));
            uint32_t cs[8];
            corner_slots_shfl(row, slot, cs);
            if (word & WORD_FLUID) {
                const uint32_t wm = word & WORD_WALL_MASK;
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const uint32_t flip = ((uint32_t)a.parity ^ (wm >> i)) & 1u;
                    const uint32_t dir = flip ? (uint32_t)(Q - 1 - i) : (uint32_t)i;
                    if (LBM_IN_RANGE(dir * n + cs[corner_neg(i)], (uint64_t)Q * n, 2))
                        cp_async4(&stage[(st * Q + i) * T + tid], pop + dir * n + cs[corner_neg(i)]);
                }
            }
        }
        cp_async_commit();
    };
    int st = 0;
    int64_t c = blockIdx.x;
    if (c < n_chunks) prefetch(c, 0);
    for (; c < n_chunks; c += gridDim.x) {
        prefetch(c + gridDim.x, st ^ 1);  // an empty group past the end keeps the count aligned
        cp_async_wait_one();
        const uint32_t slot = (uint32_t)(c * T) + tid;
        if (slot < (uint32_t)(v.n_bricks * BRICK_CELLS)) {
            const uint32_t word = __ldg(v.word + slot);
            const int32_t row = __ldg(v.nb8 + (slot / BRICK_CELLS) * 8u + (lane & 7u));
            uint32_t cs[8];
            corner_slots_shfl(row, slot, cs);
            if (word & WORD_FLUID) {
                const uint32_t wm = word & WORD_WALL_MASK;
                LevelArgs la = a;
                if (word & WORD_OWN_TAU) set_own_rate<COLL>(la, __ldg(v.s2_cell + slot));
                float d[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) d[i] = stage[(st * Q + i) * T + tid];
                const uint32_t half = wm ? wall_rules<LBM_STORE_FP32, LBM_SCHEME_ESOTERIC>(v, nullptr, slot, word, a, d) : 0u;
                collide_model<COLL>(d, la);
                store_et<LBM_STORE_FP32>(pop, n, cs, a.parity, d);
                if (half) {
                    const uint32_t off = (uint32_t)v.aux[slot];
#pragma unroll
                    for (int i = 0; i < Q; ++i)
                        if ((half & (1u << i)) && LBM_IN_RANGE(link_index(off, wm, i), v.n_bq, 5))
                            Store<LBM_STORE_FP32>::store(v.side, i, link_index(off, wm, i), d[i]);
                }
            }
        }
        st ^= 1;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// Several domains (esoteric twist, one storage precision) in one launch: the CTAs run over the
// concatenated brick lists; each warp finds its domain by binary search in the brick prefix
// sums and updates one of that domain's half-bricks with the domain's own level arguments.
template <int ST, int BRICKS, int MINB, int COLL, int PC = -1>
__global__ void __launch_bounds__(BRICKS * BRICK_CELLS, MINB)
    k_step_batch(const BatchEntry* __restrict__ ent, const int64_t* __restrict__ brick_start, int n_dom,
                 const LevelArgs* __restrict__ args)
{
    __shared__ float sm[BRICKS * 2][Q * 32];
    pdl_trigger();
    const int64_t gslot = (int64_t)blockIdx.x * (BRICKS * BRICK_CELLS) + threadIdx.x;
    const int64_t gbrick = gslot / BRICK_CELLS;
    if (gbrick >= __ldg(brick_start + n_dom)) return;  // whole warps
    int lo = 0, hi = n_dom - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(brick_start + mid) <= gbrick) lo = mid;
        else hi = mid - 1;
    }
    const DomainView& v = ent[lo].view;
    const LevelArgs a = args[lo];
    const uint32_t slot = (uint32_t)((gbrick - __ldg(brick_start + lo)) * BRICK_CELLS) + (threadIdx.x & 63u);
    step_cell<ST, LBM_SCHEME_ESOTERIC, COLL, PC>(v, ent[lo].pop, ent[lo].pop, a, slot, threadIdx.x & 31u,
                                                 sm[threadIdx.x >> 5]);
}

// Persistent form of the batched step: one launch advances every domain `steps` steps.  The CTAs
// (all resident: the launch is cooperative) stride over the concatenated brick list, BRICKS bricks
// per unit of work, and meet at a grid-wide barrier after each step, since the twist's next step
// reads what neighbouring CTAs wrote.  Every wait at the barrier is bounded by `limit_ns` of the
// global timer: a CTA that gives up raises bar->fail and every CTA leaves at its next barrier, so
// a chunk that cannot complete ends instead of hanging (the host then reports LBM_ERR_TIMEOUT).
// One body for both parities and a budget of 80 registers (6 CTAs per SM): two bodies, one per parity, with six
// link rounds in 64 registers spilled 2 KB a thread.  Per step, default rates, two bodies in 64 registers -> this:
// 2 vessels FP16 12.6 -> 8.1 us, 8 vessels 34.3 -> 20.8 us, 16 vessels 56.6 -> 34.2 us (FP32 60.4 -> 34.2 us); one
// body in 64 registers with three rounds: 10.8, 23.7 and 35.7 us.
__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// true when every CTA has finished step s; false when this CTA or another gave up
__device__ __forceinline__ bool grid_barrier(GridBarrier* bar, unsigned int target, uint64_t limit_ns)
{
    __shared__ int ok;
    __syncthreads();  // this CTA's writes of the step are done
    if (threadIdx.x == 0) {
        int good = 1;
        __threadfence();  // release them at GPU scope before arriving
        atomicAdd(&bar->count, 1u);
        const uint64_t t0 = global_ns();
        while (true) {
            unsigned int c, f;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&bar->count) : "memory");
            if (c >= target) break;
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(f) : "l"(&bar->fail) : "memory");
            if (f) {
                good = 0;
                break;
            }
            if (global_ns() - t0 > limit_ns) {
                atomicExch(&bar->fail, 1u);
                good = 0;
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

template <int ST, int BRICKS, int MINB, int COLL>
__global__ void __launch_bounds__(BRICKS * BRICK_CELLS, MINB)
    k_step_batch_persistent(const BatchEntry* __restrict__ ent, const int64_t* __restrict__ brick_start, int n_dom,
                            const LevelArgs* __restrict__ args, int steps, GridBarrier* bar, unsigned int* tickets,
                            uint64_t limit_ns)
{
    const int64_t total = __ldg(brick_start + n_dom);
    const int64_t n_units = (total + BRICKS - 1) / BRICKS;
    __shared__ unsigned int next;
    __shared__ float sm[BRICKS * 2][Q * 32];
    for (int s = 0; s < steps; ++s) {
        // units of step s are handed out by a ticket counter (tickets[s], cleared before the
        // launch), so that CTAs that finish early take more
        for (;;) {
            __syncthreads();  // every thread has read the previous ticket
            if (threadIdx.x == 0) next = atomicAdd(&tickets[s], 1u);
            __syncthreads();
            const int64_t unit = next;
            if (unit >= n_units) break;
            const int64_t gbrick = unit * BRICKS + (threadIdx.x / BRICK_CELLS);
            if (gbrick < total) {  // whole warps
                int lo = 0, hi = n_dom - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (__ldg(brick_start + mid) <= gbrick) lo = mid;
                    else hi = mid - 1;
                }
                const DomainView& v = ent[lo].view;
                const LevelArgs a = args[(size_t)s * n_dom + lo];
                const uint32_t slot =
                    (uint32_t)((gbrick - __ldg(brick_start + lo)) * BRICK_CELLS) + (threadIdx.x & 63u);
                step_cell<ST, LBM_SCHEME_ESOTERIC, COLL, -1, false>(v, ent[lo].pop, ent[lo].pop, a, slot, threadIdx.x & 31u,
                                                                    sm[threadIdx.x >> 5]);
            }
        }
        if (s + 1 < steps && !grid_barrier(bar, (unsigned int)(s + 1) * gridDim.x, limit_ns)) return;
    }
}

// Running means (the time averaging of Sec. 3.3): sums[k] += (rho, ux, uy, uz) of fluid cell k at
// the current level, in FP64 so that thousands of samples add without loss.
template <int ST, int SCHEME>
__global__ void __launch_bounds__(256)
    k_mean_sample(DomainView v, const void* src, LevelArgs a, const int32_t* fl_slot, int64_t n_fluid, Sum4* sums)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_fluid) return;
    const uint32_t slot = (uint32_t)fl_slot[k];
    float d[Q];
    gather<ST, SCHEME>(v, src, slot, v.word[slot], a, d);
    const Moments M = moments(d, a.g);
    Sum4 s = sums[k];
    s.x += (double)M.rho;
    s.y += (double)M.ux;
    s.z += (double)M.uy;
    s.w += (double)M.uz;
    sums[k] = s;
}

// Monitoring-point probes (Sec. 2.2.2 follows the velocity at points around the sac):
// out[p] = (rho, ux, uy, uz) of fluid cell idx[p] (fluid index: box order, x fastest); an index
// outside [0, n_fluid) gives NaNs.
template <int ST, int SCHEME>
__global__ void __launch_bounds__(128)
    k_probe(DomainView v, const void* src, LevelArgs a, const int32_t* fl_slot, int64_t n_fluid, const int64_t* idx,
            int n, float4* out)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int64_t k = idx[p];
    if (k < 0 || k >= n_fluid) {
        out[p] = make_float4(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000), __int_as_float(0x7fc00000),
                             __int_as_float(0x7fc00000));
        return;
    }
    const uint32_t slot = (uint32_t)fl_slot[k];
    float d[Q];
    gather<ST, SCHEME>(v, src, slot, v.word[slot], a, d);
    const Moments M = moments(d, a.g);
    out[p] = make_float4(M.rho, M.ux, M.uy, M.uz);
}

template <int ST, int SCHEME>
__global__ void __launch_bounds__(256)
    k_macroscopic(DomainView v, const void* src, LevelArgs a, const int32_t* fl_slot, const int32_t* fl_box,
                  int64_t n_fluid, int dense, float* rho, float* u, int64_t n_out)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_fluid) return;
    const uint32_t slot = (uint32_t)fl_slot[k];
    float d[Q];
    gather<ST, SCHEME>(v, src, slot, v.word[slot], a, d);
    const Moments M = moments(d, a.g);
    const int64_t o = dense ? (int64_t)fl_box[k] : k;
    rho[o] = M.rho;
    u[o] = M.ux;
    u[n_out + o] = M.uy;
    u[2 * n_out + o] = M.uz;
}

// Post-collision populations of the previous level := f_eq(rho, u) (full expansion, product
// form), written as deviations d_i = rho (prod psi - w_i) + (rho - 1) w_i with
// prod psi - w = dpx psi_y psi_z + w1x dpy psi_z + w1x w1y dpz, dpsi(0) = -u^2,
// dpsi(+-1) = (+-u + u^2)/2.  A-B: into the cell's own slots; twist: where the step of parity
// `parity_prev` would have written them, plus every direction into the side buffer of a
// Bouzidi cell.
template <int ST, int SCHEME>
__global__ void __launch_bounds__(256)
    k_init_equilibrium(DomainView v, void* dst, int parity_prev, const int32_t* fl_slot, const int32_t* fl_box,
                       int64_t n_fluid, const float* rho_in, const float* u_in, int64_t n_box)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_fluid) return;
    const int64_t b = fl_box[k];
    const uint32_t slot = (uint32_t)fl_slot[k];
    const float rho = rho_in[b];
    const float u[3] = {u_in[b], u_in[n_box + b], u_in[2 * n_box + b]};
    float dp[3][3], ps[3][3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const float uu = u[ax] * u[ax];
        dp[ax][0] = 0.5f * (uu - u[ax]);
        dp[ax][1] = -uu;
        dp[ax][2] = 0.5f * (uu + u[ax]);
        ps[ax][0] = 1.0f / 6.0f + dp[ax][0];
        ps[ax][1] = 2.0f / 3.0f + dp[ax][1];
        ps[ax][2] = 1.0f / 6.0f + dp[ax][2];
    }
    float d[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int ix = cx_of(i) + 1, iy = cy_of(i) + 1, iz = cz_of(i) + 1;
        const float w1x = w1_of(cx_of(i)), w1y = w1_of(cy_of(i));
        const float dprod = dp[0][ix] * ps[1][iy] * ps[2][iz] + w1x * dp[1][iy] * ps[2][iz] + w1x * w1y * dp[2][iz];
        d[i] = fmaf(rho, dprod, (rho - 1.0f) * w_of(i));
    }
    const uint32_t n = (uint32_t)v.n_slots;
    if (SCHEME == LBM_SCHEME_ESOTERIC) {
        uint32_t cs[8];
        corner_slots(v.nb8 + (slot / BRICK_CELLS) * 8, slot, cs);
        store_et<ST>(dst, n, cs, parity_prev, d);
        const uint32_t word = v.word[slot];
        if (((word >> WORD_KIND_SHIFT) & 3u) == KIND_BOUZIDI) {
            const uint32_t off = (uint32_t)v.aux[slot];
            const uint32_t wm = word & WORD_WALL_MASK;
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (((wm >> i) & 1u) && LBM_IN_RANGE(link_index(off, wm, i), v.n_bq, 5))
                    Store<ST>::store(v.side, i, link_index(off, wm, i), d[i]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if (LBM_IN_RANGE((uint32_t)i * n + slot, (uint64_t)Q * n, 4)) Store<ST>::store(dst, i, (uint32_t)i * n + slot, d[i]);
    }
}

// Velocity correction (learned corrector): the post-collision populations of the previous level
// gain rho (prod psi(u + du) - prod psi(u)) at every fluid cell except inlet and outlet cells,
// rho and u those of the current level.  The product difference is expanded, (a + da)(b + db)(c + dc) - abc =
// da (b + db)(c + dc) + a db (c + dc) + a b dc, with dpsi(0) = -(2u + du) du and
// dpsi(+-1) = (+-du + (2u + du) du)/2, so that no O(1) value is rounded against a small one.
template <int ST, int SCHEME>
__global__ void __launch_bounds__(256)
    k_apply_du(DomainView v, void* pop, int parity_prev, const int32_t* fl_slot, const int32_t* fl_box, int64_t n_fluid,
               const float* rho_in, const float* u_in, const float* du_in, int64_t n_box)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_fluid) return;
    const int64_t b = fl_box[k];
    const uint32_t slot = (uint32_t)fl_slot[k];
    // open-boundary cells are left alone: their closures rebuild the unknowns every step
    const uint32_t word = v.word[slot];
    if (((word >> WORD_KIND_SHIFT) & 3u) >= KIND_INLET) return;
    const float rho = rho_in[b];
    float ps[3][3], dp[3][3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const float u = u_in[ax * n_box + b], du = du_in[ax * n_box + b];
        const float uu = u * u;
        ps[ax][0] = 1.0f / 6.0f + 0.5f * (uu - u);
        ps[ax][1] = 2.0f / 3.0f - uu;
        ps[ax][2] = 1.0f / 6.0f + 0.5f * (uu + u);
        const float s2 = (2.0f * u + du) * du;
        dp[ax][0] = 0.5f * (s2 - du);
        dp[ax][1] = -s2;
        dp[ax][2] = 0.5f * (s2 + du);
    }
    float delta[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int ix = cx_of(i) + 1, iy = cy_of(i) + 1, iz = cz_of(i) + 1;
        const float by = ps[1][iy] + dp[1][iy], bz = ps[2][iz] + dp[2][iz];
        delta[i] = rho * (dp[0][ix] * by * bz + ps[0][ix] * dp[1][iy] * bz + ps[0][ix] * ps[1][iy] * dp[2][iz]);
    }
    // every read is issued before the first write: the compiler cannot tell that a write does not
    // alias the next read, so read-modify-write pairs in one loop would wait for one memory
    // latency each
    const uint32_t n = (uint32_t)v.n_slots;
    uint32_t off[Q];
    float f[Q];
    if (SCHEME == LBM_SCHEME_ESOTERIC) {
        uint32_t cs[8];
        corner_slots(v.nb8 + (slot / BRICK_CELLS) * 8, slot, cs);
#pragma unroll
        for (int i = 0; i < Q; ++i) off[i] = (parity_prev ? (uint32_t)i : (uint32_t)(Q - 1 - i)) * n + cs[corner_pos(i)];
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) off[i] = (uint32_t)i * n + slot;
    }
    const bool bouzidi = SCHEME == LBM_SCHEME_ESOTERIC && ((word >> WORD_KIND_SHIFT) & 3u) == KIND_BOUZIDI;
    const uint32_t wm = bouzidi ? (word & WORD_WALL_MASK) : 0u;
    const uint32_t off0 = bouzidi ? (uint32_t)v.aux[slot] : 0u;
    float fs[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = LBM_IN_RANGE(off[i], (uint64_t)Q * n, 7) ? Store<ST>::load_rw(pop, i, off[i]) : 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i)
        fs[i] = (((wm >> i) & 1u) && LBM_IN_RANGE(link_index(off0, wm, i), v.n_bq, 5))
                    ? Store<ST>::load_rw(v.side, i, link_index(off0, wm, i))
                    : 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i)
        if (LBM_IN_RANGE(off[i], (uint64_t)Q * n, 7)) Store<ST>::store(pop, i, off[i], f[i] + delta[i]);
#pragma unroll
    for (int i = 0; i < Q; ++i)
        if (((wm >> i) & 1u) && LBM_IN_RANGE(link_index(off0, wm, i), v.n_bq, 5))
            Store<ST>::store(v.side, i, link_index(off0, wm, i), fs[i] + delta[i]);
}

// FP64 diagnostics: per-block partial sums in a fixed order; one block then reduces the
// partials in a fixed order (reproducible run to run).  The FP64 pipe is narrow (a warp-wide double addition
// takes about 16 cycles of an SM), so it gets the mass sum and the few flux terms only: the largest speed is
// kept as its square and compared as integers (the bits of non-negative doubles order like their values; one
// square root at the end, which is monotonic, gives the same number), the non-finite cells are
// counted as integers, and a warp without open cells leaves the flux sums out.
constexpr int DIAG_THREADS = 256;
constexpr int DIAG_FIELDS = 5;  // mass, flux_in, flux_out, max |u|^2, non-finite count

struct Diag {
    double mass, in, out;
    unsigned long long u2;  // bits of max |u|^2
    unsigned int bad;
};
__device__ __forceinline__ void diag_add(Diag& x, const Diag& y)
{
    x.mass += y.mass;
    x.in += y.in;
    x.out += y.out;
    x.u2 = x.u2 > y.u2 ? x.u2 : y.u2;
    x.bad += y.bad;
}
// the block's total in thread 0, in a fixed order (every warp's tree, then the warps in turn)
__device__ __forceinline__ void block_reduce(Diag& x, Diag* sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool flux = __any_sync(0xffffffffu, x.in != 0.0 || x.out != 0.0);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        x.mass += __shfl_down_sync(0xffffffffu, x.mass, off);
        const unsigned long long o = __shfl_down_sync(0xffffffffu, x.u2, off);
        x.u2 = x.u2 > o ? x.u2 : o;
        if (flux) {
            x.in += __shfl_down_sync(0xffffffffu, x.in, off);
            x.out += __shfl_down_sync(0xffffffffu, x.out, off);
        }
    }
    x.bad = __reduce_add_sync(0xffffffffu, x.bad);
    if (lane == 0) sh[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < DIAG_THREADS / 32; ++w) diag_add(x, sh[w]);
}

template <int ST, int SCHEME>
__global__ void __launch_bounds__(DIAG_THREADS)
    k_diagnostics(DomainView v, const void* src, LevelArgs a, const int32_t* fl_slot, int64_t n_fluid,
                  double* partials)
{
    __shared__ Diag sh[DIAG_THREADS / 32];
    Diag x{0.0, 0.0, 0.0, 0ull, 0u};
    pdl_trigger();
    const int64_t k = (int64_t)blockIdx.x * DIAG_THREADS + threadIdx.x;
    if (k < n_fluid) {
        const uint32_t slot = (uint32_t)fl_slot[k];
        const uint32_t word = v.word[slot];
        float d[Q];
        gather<ST, SCHEME>(v, src, slot, word, a, d);
        const Moments M = moments(d, a.g);
        const bool finite = isfinite(M.rho) && isfinite(M.ux) && isfinite(M.uy) && isfinite(M.uz);
        if (finite) {
            x.mass = (double)M.rho;
            const int kind = (int)((word >> WORD_KIND_SHIFT) & 3u);
            if (kind >= KIND_INLET && LBM_IN_RANGE(v.aux[slot], v.n_io, 6)) {
                const int64_t rec = v.aux[slot];
                const int ax = v.io_axis[rec];
                const float un = v.io_sign[rec] * (ax == 0 ? M.ux : ax == 1 ? M.uy : M.uz);
                if (kind == KIND_INLET) x.in = (double)M.rho * (double)un;
                else x.out = -(double)M.rho * (double)un;
            }
            x.u2 = (unsigned long long)__double_as_longlong((double)M.ux * M.ux + (double)M.uy * M.uy + (double)M.uz * M.uz);
        } else {
            x.bad = 1u;
        }
    }
    block_reduce(x, sh);
    if (threadIdx.x == 0) {
        if (n_fluid == 0) pdl_wait();  // no cell has waited: the partials are those of the call before
        double* p = partials + (int64_t)blockIdx.x * DIAG_FIELDS;
        p[0] = x.mass;
        p[1] = x.in;
        p[2] = x.out;
        p[3] = __longlong_as_double((long long)x.u2);
        p[4] = (double)x.bad;
    }
}

inline int grid_for(int64_t n, int threads) { return (int)((n + threads - 1) / threads); }

// Calls f(std::integral_constant<int, COLL>{}) for the collision kernel `coll`.
template <class F>
cudaError_t with_coll(int coll, F&& f)
{
    switch (coll) {
    case COLL_CHM: return f(std::integral_constant<int, COLL_CHM>{});
    case COLL_CHM_FAST: return f(std::integral_constant<int, COLL_CHM_FAST>{});
    case COLL_SRT2: return f(std::integral_constant<int, COLL_SRT2>{});
    default: return f(std::integral_constant<int, COLL_TRT2>{});
    }
}

// ------------------------------------------------------------------------------ launchers
// A launch that may start while the kernel before it on the stream drains (see pdl_wait)
template <class... P, class... A>
cudaError_t launch_pdl(void (*k)(P...), int grid, int block, size_t smem, cudaStream_t s, A&&... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&c, k, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // reported here: a later launch that asks must not find it again
    return e;
}

// Launch configurations of the step kernel: (bricks per CTA, minimum resident CTAs per SM);
// the second number sets the register budget, 65536 / (threads * CTAs).
template <int ST, int SCHEME, int BRICKS, int MINB>
cudaError_t launch_step_t(const DomainView& v, const void* src, void* dst, const LevelArgs& a, cudaStream_t s)
{
    if (v.n_bricks == 0) return cudaSuccess;
    const int grid = grid_for(v.n_bricks, BRICKS);
    return with_coll(a.coll, [&](auto c) {
        constexpr int C = decltype(c)::value;
        constexpr int T = BRICKS * BRICK_CELLS;
        // The kernel's link rounds: 0 (neither link code nor exchange area) for a domain without Bouzidi cells, where
        // that is faster: default rates (633 k cell pipe FP16 19.5 us a step, 20.8 us with them), SRT and TRT
        // on large domains (TRT at 8 CTAs per SM 25.2 and 34.6 us; on 87 k cells 5.4 and 5.1 us), not general
        // rates (26.4 and 26.0 us); fewer for a large domain with links (2.7 M cells, TRT at 8 CTAs 137 and 152 us).
        // The twist with the default rates has one kernel per parity (constant plane indices).
        constexpr bool TWIST = SCHEME == LBM_SCHEME_ESOTERIC, FAST = C == COLL_CHM_FAST;
        constexpr int P0 = TWIST && FAST ? 0 : -1, P1 = TWIST && FAST ? 1 : -1;
        constexpr int L = LINK_ROUNDS, LL = LINK_ROUNDS_LARGE, L0 = C == COLL_CHM ? L : 0;
        const bool large = v.n_bricks > LARGE_BRICKS;
        auto k = !v.bstart && (FAST || large) ? (a.parity ? k_step<ST, SCHEME, BRICKS, MINB, C, P1, L0> : k_step<ST, SCHEME, BRICKS, MINB, C, P0, L0>)
                 : v.bstart && large          ? (a.parity ? k_step<ST, SCHEME, BRICKS, MINB, C, P1, LL> : k_step<ST, SCHEME, BRICKS, MINB, C, P0, LL>)
                                              : (a.parity ? k_step<ST, SCHEME, BRICKS, MINB, C, P1, L> : k_step<ST, SCHEME, BRICKS, MINB, C, P0, L>);
        return launch_pdl(k, grid, T, 0, s, v, src, dst, a);
    });
}

template <int ST, int BRICKS, int MINB>
cudaError_t launch_step2(const DomainView& v, void* pop, const LevelArgs& a, cudaStream_t s)
{
    if (v.n_bricks == 0) return cudaSuccess;
    // runtime parity: the constant-plane form of the one-cell kernels was slower here (the two
    // cells' addresses compete with the packed collision for the 128-register budget)
    return launch_pdl(k_step2<ST, BRICKS, MINB, -1>, grid_for(v.n_bricks, BRICKS), BRICKS * 32, 0, s, v, pop, a);
}

template <int BRICKS, int MINB>
cudaError_t launch_step_et_pipe(const DomainView& v, void* pop, const LevelArgs& a, cudaStream_t s)
{
    if (v.n_bricks == 0) return cudaSuccess;
    constexpr int T = BRICKS * BRICK_CELLS;
    const size_t smem = sizeof(float) * 2 * Q * T;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t n_chunks = (v.n_bricks + BRICKS - 1) / BRICKS;
    const int grid = (int)std::min<int64_t>(n_chunks, (int64_t)sms * MINB);
    return with_coll(a.coll, [&](auto c) {
        auto k = k_step_et_pipe<BRICKS, MINB, decltype(c)::value>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        return launch_pdl(k, grid, T, smem, s, v, static_cast<float*>(pop), a);
    });
}

template <int ST, int SCHEME>
cudaError_t launch_step_scheme(int config, const DomainView& v, const void* src, void* dst, const LevelArgs& level,
                               cudaStream_t s)
{
    const LevelArgs a = with_sweep<ST, SCHEME>(v, level);
    if (config == 5) {
        if (ST == LBM_STORE_FP32 && SCHEME == LBM_SCHEME_ESOTERIC) return launch_step_et_pipe<2, 6>(v, dst, a, s);
        config = 3;  // the pipelined variant exists for FP32 twist only
    }
    if (config >= 6) {
        if (SCHEME == LBM_SCHEME_ESOTERIC && a.coll == COLL_CHM_FAST)
            return config == 6 ? launch_step2<ST, 4, 4>(v, dst, a, s) : launch_step2<ST, 4, 3>(v, dst, a, s);
        config = 2;  // the two-cell kernels exist for the twist with the default rates only
    }
    switch (config) {
    case 0: return launch_step_t<ST, SCHEME, 4, 3>(v, src, dst, a, s);
    case 1: return launch_step_t<ST, SCHEME, 2, 7>(v, src, dst, a, s);
    case 2: return launch_step_t<ST, SCHEME, 2, 6>(v, src, dst, a, s);
    case 3: return launch_step_t<ST, SCHEME, 2, 8>(v, src, dst, a, s);
    default: return launch_step_t<ST, SCHEME, 2, 10>(v, src, dst, a, s);
    }
}

template <int ST>
cudaError_t launch_step(int scheme, int config, const DomainView& v, const void* src, void* dst,
                        const LevelArgs& a, cudaStream_t s)
{
    return scheme == LBM_SCHEME_ESOTERIC ? launch_step_scheme<ST, LBM_SCHEME_ESOTERIC>(config, v, src, dst, a, s)
                                         : launch_step_scheme<ST, LBM_SCHEME_AB>(config, v, src, dst, a, s);
}

// the export, the means and the correction run one thread per fluid cell; with small CTAs a domain of a few
// ten thousand cells still spreads over every SM (its latency chains overlap on all of them)
constexpr int PER_CELL_THREADS = 64;

template <int ST>
cudaError_t launch_macroscopic(int scheme, const DomainView& v, const void* src, const LevelArgs& a,
                               const int32_t* fl_slot, const int32_t* fl_box, int64_t n_fluid, int dense, float* rho,
                               float* u, int64_t n_out, cudaStream_t s)
{
    if (n_fluid == 0) return cudaSuccess;
    if (scheme == LBM_SCHEME_ESOTERIC)
        return launch_pdl(k_macroscopic<ST, LBM_SCHEME_ESOTERIC>, grid_for(n_fluid, PER_CELL_THREADS), PER_CELL_THREADS, 0, s, v,
                          src, a, fl_slot, fl_box, n_fluid, dense, rho, u, n_out);
    return launch_pdl(k_macroscopic<ST, LBM_SCHEME_AB>, grid_for(n_fluid, PER_CELL_THREADS), PER_CELL_THREADS, 0, s, v, src, a,
                      fl_slot, fl_box, n_fluid, dense, rho, u, n_out);
}

template <int ST>
cudaError_t launch_mean_sample(int scheme, const DomainView& v, const void* src, const LevelArgs& a,
                               const int32_t* fl_slot, int64_t n_fluid, Sum4* sums, cudaStream_t s)
{
    if (n_fluid == 0) return cudaSuccess;
    if (scheme == LBM_SCHEME_ESOTERIC)
        return launch_pdl(k_mean_sample<ST, LBM_SCHEME_ESOTERIC>, grid_for(n_fluid, PER_CELL_THREADS), PER_CELL_THREADS, 0, s, v,
                          src, a, fl_slot, n_fluid, sums);
    return launch_pdl(k_mean_sample<ST, LBM_SCHEME_AB>, grid_for(n_fluid, PER_CELL_THREADS), PER_CELL_THREADS, 0, s, v, src, a,
                      fl_slot, n_fluid, sums);
}

template <int ST>
cudaError_t launch_probe(int scheme, const DomainView& v, const void* src, const LevelArgs& a, const int32_t* fl_slot,
                         int64_t n_fluid, const int64_t* idx, int n, float4* out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    if (scheme == LBM_SCHEME_ESOTERIC)
        k_probe<ST, LBM_SCHEME_ESOTERIC><<<grid_for(n, 128), 128, 0, s>>>(v, src, a, fl_slot, n_fluid, idx, n, out);
    else
        k_probe<ST, LBM_SCHEME_AB><<<grid_for(n, 128), 128, 0, s>>>(v, src, a, fl_slot, n_fluid, idx, n, out);
    return cudaGetLastError();
}

template <int ST>
cudaError_t launch_init_equilibrium(int scheme, const DomainView& v, void* dst, int parity_prev,
                                    const int32_t* fl_slot, const int32_t* fl_box, int64_t n_fluid,
                                    const float* rho, const float* u, int64_t n_box, cudaStream_t s)
{
    if (n_fluid == 0) return cudaSuccess;
    if (scheme == LBM_SCHEME_ESOTERIC)
        k_init_equilibrium<ST, LBM_SCHEME_ESOTERIC><<<grid_for(n_fluid, 256), 256, 0, s>>>(
            v, dst, parity_prev, fl_slot, fl_box, n_fluid, rho, u, n_box);
    else
        k_init_equilibrium<ST, LBM_SCHEME_AB><<<grid_for(n_fluid, 256), 256, 0, s>>>(
            v, dst, parity_prev, fl_slot, fl_box, n_fluid, rho, u, n_box);
    return cudaGetLastError();
}

template <int ST>
cudaError_t launch_diagnostics(int scheme, const DomainView& v, const void* src, const LevelArgs& a,
                               const int32_t* fl_slot, int64_t n_fluid, double* partials, cudaStream_t s)
{
    const int nb = (int)diagnostics_blocks(n_fluid);
    if (scheme == LBM_SCHEME_ESOTERIC)
        return launch_pdl(k_diagnostics<ST, LBM_SCHEME_ESOTERIC>, nb, DIAG_THREADS, 0, s, v, src, a, fl_slot, n_fluid, partials);
    return launch_pdl(k_diagnostics<ST, LBM_SCHEME_AB>, nb, DIAG_THREADS, 0, s, v, src, a, fl_slot, n_fluid, partials);
}

template <int ST>
cudaError_t launch_apply_du(int scheme, const DomainView& v, void* pop, int parity_prev, const int32_t* fl_slot,
                           const int32_t* fl_box, int64_t n_fluid, const float* rho, const float* u, const float* du,
                           int64_t n_box, cudaStream_t s)
{
    if (n_fluid == 0) return cudaSuccess;
    if (scheme == LBM_SCHEME_ESOTERIC)
        k_apply_du<ST, LBM_SCHEME_ESOTERIC><<<grid_for(n_fluid, PER_CELL_THREADS), PER_CELL_THREADS, 0, s>>>(v, pop, parity_prev, fl_slot, fl_box,
                                                                               n_fluid, rho, u, du, n_box);
    else
        k_apply_du<ST, LBM_SCHEME_AB><<<grid_for(n_fluid, PER_CELL_THREADS), PER_CELL_THREADS, 0, s>>>(v, pop, parity_prev, fl_slot, fl_box, n_fluid,
                                                                         rho, u, du, n_box);
    return cudaGetLastError();
}

template <int ST, int BRICKS, int MINB>
cudaError_t launch_step_batch_t(const BatchEntry* ent, const int64_t* brick_start, int n_dom, int64_t total_bricks,
                                const LevelArgs* args, int coll, int parity, cudaStream_t s)
{
    if (total_bricks == 0) return cudaSuccess;
    const int grid = grid_for(total_bricks, BRICKS);
    return with_coll(coll, [&](auto c) {
        constexpr int C = decltype(c)::value;
        constexpr int T = BRICKS * BRICK_CELLS;
        // one kernel per parity when every domain has the same one (constant plane indices)
        if constexpr (C == COLL_CHM_FAST) {
            if (parity >= 0)
                return launch_pdl(parity ? k_step_batch<ST, BRICKS, MINB, C, 1> : k_step_batch<ST, BRICKS, MINB, C, 0>, grid,
                                  T, 0, s, ent, brick_start, n_dom, args);
        }
        return launch_pdl(k_step_batch<ST, BRICKS, MINB, C>, grid, T, 0, s, ent, brick_start, n_dom, args);
    });
}

// one cooperative launch of k_step_batch_persistent (128 threads, 6 CTAs per SM): as many
// CTAs as can be resident, never more than units of work; bar is followed by `steps` ticket
// counters, all cleared before the launch
template <int ST, int COLL>
cudaError_t launch_persistent_t(const BatchEntry* ent, const int64_t* brick_start, int n_dom, int64_t total_bricks,
                                const LevelArgs* args, int steps, GridBarrier* bar, uint64_t limit_ns, cudaStream_t s)
{
    constexpr int BRICKS = 2, MINB = 6;
    unsigned int* tickets = reinterpret_cast<unsigned int*>(bar + 1);  // [steps] after the barrier word
    auto k = k_step_batch_persistent<ST, BRICKS, MINB, COLL>;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, BRICKS * BRICK_CELLS, 0);
    if (e != cudaSuccess) return e;
    const int64_t units = (total_bricks + BRICKS - 1) / BRICKS;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(units, (int64_t)sms * per_sm));
    void* kargs[] = {(void*)&ent, (void*)&brick_start, (void*)&n_dom, (void*)&args, (void*)&steps, (void*)&bar,
                     (void*)&tickets, (void*)&limit_ns};
    return cudaLaunchCooperativeKernel((const void*)k, dim3(grid), dim3(BRICKS * BRICK_CELLS), kargs, 0, s);
}

template <int ST>
cudaError_t launch_step_batch_persistent(const BatchEntry* ent, const int64_t* brick_start, int n_dom,
                                         int64_t total_bricks, const LevelArgs* args, int coll, int steps,
                                         GridBarrier* bar, uint64_t limit_ns, cudaStream_t s)
{
    if (total_bricks == 0 || steps == 0) return cudaSuccess;
    return with_coll(coll, [&](auto c) {
        return launch_persistent_t<ST, decltype(c)::value>(ent, brick_start, n_dom, total_bricks, args, steps, bar, limit_ns, s);
    });
}

template <int ST>
cudaError_t launch_step_batch(int config, const BatchEntry* ent, const int64_t* brick_start, int n_dom,
                              int64_t total_bricks, const LevelArgs* args, int coll, int parity, cudaStream_t s)
{
    switch (config) {
    case 0: return launch_step_batch_t<ST, 4, 3>(ent, brick_start, n_dom, total_bricks, args, coll, parity, s);
    case 1: return launch_step_batch_t<ST, 2, 7>(ent, brick_start, n_dom, total_bricks, args, coll, parity, s);
    case 2: return launch_step_batch_t<ST, 2, 6>(ent, brick_start, n_dom, total_bricks, args, coll, parity, s);
    case 3: return launch_step_batch_t<ST, 2, 8>(ent, brick_start, n_dom, total_bricks, args, coll, parity, s);
    default: return launch_step_batch_t<ST, 2, 10>(ent, brick_start, n_dom, total_bricks, args, coll, parity, s);
    }
}

// LBM_DEBUG: the first failed check's code since the last read (0: none), cleared on read; 0
// always in the default build
inline unsigned debug_fault()
{
#ifdef LBM_DEBUG
    unsigned h = 0u;
    const unsigned zero = 0u;
    if (cudaMemcpyFromSymbol(&h, g_debug_fault, sizeof(h)) != cudaSuccess) return 0xffffffffu;
    if (h) cudaMemcpyToSymbol(g_debug_fault, &zero, sizeof(zero));
    return h;
#else
    return 0u;
#endif
}

template <int ST>
const Launchers& make_launchers()
{
    static const Launchers L = {&launch_step<ST>,        &launch_macroscopic<ST>, &launch_init_equilibrium<ST>,
                                &launch_diagnostics<ST>, &launch_step_batch<ST>, &launch_apply_du<ST>,
                                &launch_mean_sample<ST>, &launch_probe<ST>,       &debug_fault,
                                &launch_step_batch_persistent<ST>};
    return L;
}

}  // namespace dev
}  // namespace lbm
