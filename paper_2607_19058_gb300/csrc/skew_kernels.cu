// Device kernels of libskewadam (sm_103a).
//
// One SkewAdam step (paper Sec. 3, Eq. 1, Algorithm 1) as grouped launches in stream
// order, each over an item table of (tensor, tile) pairs; a step with row-path tensors
// takes k_rowsq (and k_rowsq_wide), k_finalize, k_fallback and k_apply_rows, which also
// run its strip and flat tiles while these are few; any other takes k_sumsq, k_finalize,
// k_rms and k_apply, each after k_reset (an ordinary launch, which clears the per-step scalars), and a step
// of small tensors k_small alone:
//   k_sumsq      phase A, strip tiles: per-row and per-column sums of g^2 of a
//                factored matrix (Eq. 1), column partials per row tile (no atomics);
//   k_rowsq      phase A, whole-row tiles of factored matrices 128 to 4096 wide
//                (k_rowsq_wide: to 8192): chunks of whole rows bulk-copied into a
//                shared-memory ring; R_i formed in the tile (Eq. 1), per-column partials
//                of g^2 and of g^2 / R_i (or M^2 / R_i after the momentum update, stored
//                here), from which the finalize forms sum(U^2) by the bilinear identity;
//   k_finalize   R / C moving averages (strip path) or C (row path), 1/sqrt(C_j),
//                mean(R); on the row path also sum(U^2) and the clip factor; when the
//                1/sqrt(eps) clamp may bind, either the clip factor (provably 1; phase C
//                then sums U^2) or an entry in the queue for phase B;
//   k_rms        phase B, strip and flat tiles: momentum / exact second-moment
//                update, U up to its scalar and a compensated sum(U^2) per tile;
//                the last tile forms RMS(U) and the clip factor (Sec. 3);
//   k_fallback   phase B of the queued row-path tensors (element by element);
//   k_apply      phase C, strip and flat tiles: x = w (1 - lr*lambda) - lr*kappa*U
//                in fp32 and the dithered bf16 write-back (Philox-4x32-10);
//   k_apply_rows phase C, whole-row tiles: the same on bulk-copied rows of W and
//                G (or the new M);
//   k_small      all phases of a small tensor, one cluster of CTAs each.
// The reconstructed second moment of a factored matrix is never formed:
// 1/sqrt(max(R_i C_j / Rbar, eps)) = min(a_i * b_j, 1/sqrt(eps)) with
// a_i = 1/sqrt(R_i / Rbar) per row and b_j = 1/sqrt(C_j) per column.
//
// The per-step scalars are a kernel parameter (StepArgs, constant bank). Values
// produced by an earlier launch of the same step are read with L2-only (.cg)
// loads. When no element of a tile can reach the clamp (all but degenerate
// tiles), phase C takes a clamp-free path. Every wait on a bulk copy is bounded
// and reports a copy that does not land through the status word.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <cstddef>
#include <type_traits>
#include <stdint.h>

#include "skew_plan.h"

namespace skew {
namespace {

constexpr uint32_t kAll = 0xFFFFFFFFu;

// Resident CTAs per SM each kernel is compiled for (register budget 64K / (256 * n)).
#ifndef SKEW_MINB_SUMSQ
#define SKEW_MINB_SUMSQ 4
#endif
#ifndef SKEW_MINB_RMS
#define SKEW_MINB_RMS 2
#endif
#ifndef SKEW_MINB_APPLY
#define SKEW_MINB_APPLY 2
#endif
constexpr int kSmemFloats = kVecPerThread * kThreads;  // row scales of the tallest tile
constexpr int kStripCols = 8 * 32;                     // widest column strip

// ---------------------------------------------------------------------------
// Memory access helpers
// ---------------------------------------------------------------------------
// L2 eviction policies for 16-byte accesses (created once per thread).
struct Pol {
    uint64_t keep;  // evict_last: gradient between its first and last pass
    uint64_t drop;  // evict_first: streamed once (weights, last gradient read)
    __device__ Pol() {
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(keep));
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(drop));
    }
};

__device__ __forceinline__ uint4 ld16_hint(const void *p, uint64_t pol) {
    uint4 u;
    asm volatile("ld.global.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w)
                 : "l"(p), "l"(pol));
    return u;
}

__device__ __forceinline__ void st16_hint(void *p, uint4 u, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1,%2,%3,%4}, %5;" ::"l"(p), "r"(u.x), "r"(u.y), "r"(u.z),
                 "r"(u.w), "l"(pol));
}

__device__ __forceinline__ float bf16_to_f32(uint16_t h) { return __uint_as_float(uint32_t(h) << 16); }

__device__ __forceinline__ void unpack_bf8(uint4 u, float (&o)[8]) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        o[2 * q] = __uint_as_float(w[q] << 16);
        o[2 * q + 1] = __uint_as_float(w[q] & 0xFFFF0000u);
    }
}

// The same eight values as four (even, odd) pairs for the packed FP32x2 unit.
__device__ __forceinline__ void unpack_bf8x2(uint4 u, float2 (&o)[4]) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q] = make_float2(__uint_as_float(w[q] << 16), __uint_as_float(w[q] & 0xFFFF0000u));
}

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// Elements e0 .. e0 + 7 of a weight or gradient array (elements >= valid read as 0): bf16, or fp32
// for a tensor kept in fp32 (its array pointer then addresses floats). `wide`: the address is on
// the boundary that 16-byte loads need. Loaded as they are, and converted where they are used: a conversion
// beside the load would make each of several such loads wait for the one before (k_sumsq, 28160 x 4095 bf16:
// 124 us so, 97 with one row's loads at a time, 86 now).
struct Raw8 {
    uint32_t w[8];
    bool packed;  // two bf16 to a word
};

__device__ __forceinline__ void load8_raw(const uint16_t *base, bool f32, bool wide, int64_t e0, int valid, Raw8 &r,
                                          const Pol &pol) {
    r.packed = !f32 && wide && valid == 8;
    if (f32) {
        const uint32_t *p = reinterpret_cast<const uint32_t *>(base) + e0;
        if (wide && valid == 8) {
            const uint4 a = ld16_hint(p, pol.drop), b = ld16_hint(p + 4, pol.drop);
            r.w[0] = a.x; r.w[1] = a.y; r.w[2] = a.z; r.w[3] = a.w;
            r.w[4] = b.x; r.w[5] = b.y; r.w[6] = b.z; r.w[7] = b.w;
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) r.w[c] = c < valid ? p[c] : 0u;
        }
    } else if (r.packed) {
        const uint4 a = ld16_hint(base + e0, pol.drop);
        r.w[0] = a.x; r.w[1] = a.y; r.w[2] = a.z; r.w[3] = a.w;
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) r.w[c] = c < valid ? base[e0 + c] : 0u;
    }
}

__device__ __forceinline__ void values8(const Raw8 &r, bool f32, float (&o)[8]) {
    if (r.packed) {
        unpack_bf8(make_uint4(r.w[0], r.w[1], r.w[2], r.w[3]), o);
    } else if (f32) {
#pragma unroll
        for (int c = 0; c < 8; ++c) o[c] = __uint_as_float(r.w[c]);
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) o[c] = __uint_as_float(r.w[c] << 16);
    }
}

// The same for one vector at a time, as values.
__device__ __forceinline__ void load8_elem(const uint16_t *base, bool f32, bool wide, int64_t e0, int valid,
                                           float (&o)[8], const Pol &pol) {
    if (f32) {
        const float *p = reinterpret_cast<const float *>(base) + e0;
        if (wide && valid == 8) {
            const uint4 a = ld16_hint(p, pol.drop), b = ld16_hint(p + 4, pol.drop);
            const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] = __uint_as_float(w[c]);
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) o[c] = c < valid ? p[c] : 0.f;
        }
    } else if (wide && valid == 8) {
        unpack_bf8(ld16_hint(base + e0, pol.drop), o);
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) o[c] = c < valid ? bf16_to_f32(base[e0 + c]) : 0.f;
    }
}

// Eight fp32 state values (`wide`: on a 16-byte boundary), read through L2 (an earlier launch of
// the step may have written them).
__device__ __forceinline__ void load_f8(const float *p, bool wide, int valid, float (&o)[8]) {
    if (wide && valid == 8) {
        const float4 a = __ldcg(reinterpret_cast<const float4 *>(p));
        const float4 b = __ldcg(reinterpret_cast<const float4 *>(p + 4));
        o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
        o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) o[c] = c < valid ? __ldcg(p + c) : 0.f;
    }
}

__device__ __forceinline__ void store_f8(float *p, bool wide, int valid, const float (&o)[8]) {
    if (wide && valid == 8) {
        *reinterpret_cast<float4 *>(p) = make_float4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<float4 *>(p + 4) = make_float4(o[4], o[5], o[6], o[7]);
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < valid) p[c] = o[c];
    }
}

// ---------------------------------------------------------------------------
// Dither: Philox-4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) -- ten rounds of
// two 32x32 multiplies whose high halves are xored with the other counter
// words and the round key; the key advances by two Weyl constants per round.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                               uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
        const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
        c0 = hi1 ^ c1 ^ k0;
        c1 = lo1;
        c2 = hi0 ^ c3 ^ k1;
        c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return make_uint4(c0, c1, c2, c3);
}

// Dither key of one tensor at one step: tensor id, low 32 bits of the step and
// the two halves of the seed (kept in registers by the hot loops).
struct Dith {
    uint32_t tid, step, k0, k1;
    uint64_t base;  // dither index of the tile's tensor element 0
};

__device__ __forceinline__ Dith dith_of(const StepArgs &A, const TensorDev &T) {
    return Dith{T.tid, A.step_lo, A.seed_lo, A.seed_hi, T.base};
}

// The 16-bit dithers of the eight elements idx0 .. idx0+7 (idx0 a multiple of 8):
// counter (idx0/8 lo, idx0/8 hi, tensor id, step lo), key (seed lo, seed hi);
// element k takes half (k & 1) of word k >> 1.
__device__ __forceinline__ void dither8(uint64_t idx0, const Dith &d, uint32_t (&r)[8]) {
    const uint64_t blk = (idx0 + d.base) >> 3;
    const uint4 o = philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), d.tid, d.step, d.k0, d.k1);
    const uint32_t w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        r[2 * q] = w[q] & 0xFFFFu;
        r[2 * q + 1] = w[q] >> 16;
    }
}

// The same for an idx0 whose dither index (with the tensor's base) need not be a multiple of 8:
// the eight halves start inside a Philox block and may run into the next.
__device__ __forceinline__ void dither8_any(uint64_t idx0, const Dith &d, uint32_t (&r)[8]) {
    const uint64_t i = idx0 + d.base, blk = i >> 3;
    const uint32_t s = (uint32_t)(i & 7);
    const uint4 a = philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), d.tid, d.step, d.k0, d.k1);
    uint32_t w[8] = {a.x, a.y, a.z, a.w, 0u, 0u, 0u, 0u};
    if (s) {
        const uint64_t nxt = blk + 1;
        const uint4 b = philox4x32_10((uint32_t)nxt, (uint32_t)(nxt >> 32), d.tid, d.step, d.k0, d.k1);
        w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
        if (s & 4) {
#pragma unroll
            for (int k = 0; k < 6; ++k) w[k] = w[k + 2];
        }
        if (s & 2) {
#pragma unroll
            for (int k = 0; k < 5; ++k) w[k] = w[k + 1];
        }
        if (s & 1) {
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = __funnelshift_r(w[k], w[k + 1], 16);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        r[2 * q] = w[q] & 0xFFFFu;
        r[2 * q + 1] = w[q] >> 16;
    }
}

// Dithered rounding to bf16: add the 16-bit draw to the fp32 bit pattern and
// keep the top half (unbiased stochastic rounding); NaN -> canonical quiet NaN.
__device__ __forceinline__ uint32_t sr_bf16(float x, uint32_t r) {
    const uint32_t b = __float_as_uint(x);
    if (x != x) return 0x7FC0u | ((b >> 16) & 0x8000u);
    return (b + r) >> 16;
}

// The gradient scale gamma of the step (the trainer's global gradient-norm clip, Sec. 4
// training setup, App. A Table 9): the step sees gamma * G. It enters only through the
// moving-average increments, (1 - beta2) gamma^2 on g^2 and (1 - beta1) gamma on g, and
// the update coefficient of momentum-free tensors (U = coef * gamma * g / D; set_clip),
// so no kernel reads the gradient more than without it. With gamma = 1 every product
// below is exact and the step is bit for bit the unscaled one.
struct GScale {
    float c1, c2;  // (1 - beta1) gamma, (1 - beta2) gamma^2
    float gam;
};

__device__ __forceinline__ GScale grad_scale(const StepArgs &A) {
    if (!A.gscale) return GScale{A.c1, A.c2, 1.f};
    const float g = __ldg(A.gscale);
    return GScale{A.c1 * g, A.c2 * (g * g), g};
}

// a_i = 1/sqrt(R_i / Rbar), with Rbar = rbar_s * 2^-rbar_e (rbar_s in [1,2)); +inf if Rbar == 0.
__device__ __forceinline__ float row_scale(float Ri, float rbar_s, int rbar_e) {
    if (rbar_s == 0.f) return __int_as_float(0x7F800000);
    return __frsqrt_rn(__fdiv_rn(ldexpf(Ri, rbar_e), rbar_s));
}

// ---------------------------------------------------------------------------
// Reductions
// ---------------------------------------------------------------------------
// Eight fp32 values in shared memory (16-byte aligned).
__device__ __forceinline__ void lds8(const float *p, float (&o)[8]) {
    const float4 a = reinterpret_cast<const float4 *>(p)[0], b = reinterpret_cast<const float4 *>(p)[1];
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
    o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
}

// Error-free sum (Knuth's TwoSum): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bp = s - a;
    e = (a - (s - bp)) + (b - bp);
}

// TwoSum on both lanes of a pair (packed FP32x2 adds; same results as two_sum).
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e) {
    s = __fadd2_rn(a, b);
    const float2 bp = __fadd2_rn(s, neg2(a));
    e = __fadd2_rn(__fadd2_rn(a, neg2(__fadd2_rn(s, neg2(bp)))), __fadd2_rn(b, neg2(bp)));
}

// The value of a compensated (hi, lo) pair in fp64. Once an infinite term has
// entered, TwoSum's error term is NaN (inf - inf) while hi carries the sum
// (+-inf, or NaN for inf - inf), so a non-finite hi is the value on its own.
__device__ __forceinline__ double pair_value(float hi, float lo) {
    return isfinite(hi) ? (double)hi + (double)lo : (double)hi;
}

// The same, rounded to fp32.
__device__ __forceinline__ float pair_f(float hi, float lo) { return isfinite(hi) ? hi + lo : hi; }

// Compensated accumulator: the running sum is hi + lo.
struct Acc2 {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float v) {
        float s, e;
        two_sum(hi, v, s, e);
        hi = s;
        lo += e;
    }
};

// Sum of the squares of eight values by a balanced tree (exact doubling when equal).
__device__ __forceinline__ float sumsq8(const float (&u)[8]) {
    const float p01 = fmaf(u[0], u[0], u[1] * u[1]);
    const float p23 = fmaf(u[2], u[2], u[3] * u[3]);
    const float p45 = fmaf(u[4], u[4], u[5] * u[5]);
    const float p67 = fmaf(u[6], u[6], u[7] * u[7]);
    return (p01 + p23) + (p45 + p67);
}

// CTA-wide compensated sum of (hi, lo) pairs; result valid in thread 0.
__device__ float2 block_sum2(Acc2 a, float2 *red) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const float h = __shfl_xor_sync(kAll, a.hi, o), l = __shfl_xor_sync(kAll, a.lo, o);
        float s, e;
        two_sum(a.hi, h, s, e);
        a.hi = s;
        a.lo += l + e;
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = make_float2(a.hi, a.lo);
    __syncthreads();
    Acc2 r;
    if (threadIdx.x == 0) {
        for (int k = 0; k < kThreads / 32; ++k) {
            float s, e;
            two_sum(r.hi, red[k].x, s, e);
            r.hi = s;
            r.lo += red[k].y + e;
        }
    }
    return make_float2(r.hi, r.lo);
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kAll, v, o);
    return v;
}

// Deterministic CTA-wide fp64 sum (fixed shuffle tree, then warp 0 over the 8 warp sums).
__device__ double block_sum_d(double v, double *red) {
    v = warp_sum_d(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double r = 0.0;
    if (w == 0) {
        r = l < kThreads / 32 ? red[l] : 0.0;
        r = warp_sum_d(r);
    }
    return r;  // valid in thread 0
}

// Counter increment that publishes this CTA's (barrier-ordered) writes and, for
// the CTA that sees the final count, acquires every other CTA's.
__device__ __forceinline__ uint32_t atom_add_acq_rel(uint32_t *p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// Shared scratch of a CTA.
struct Smem {
    float colred[kThreads * 8];  // column partials of a sum-of-squares tile
    float2 red2[kThreads / 32];
    double redd[3 * (kThreads / 32)];
    int last;
};

// Row scales a_i of a factored tile's rows and column scales b_j of its strip.
struct Meta {
    float rows[kSmemFloats];
    float cols[kStripCols];
    float red[2 * kThreads / 32];  // per-warp maxima of the row / column scales
};

// Geometry of a factored tile: LC lanes along a row, RG row groups, tile_rows / RG rows per thread.
struct FactTile {
    uint32_t LC, RG, lane, rg, s, rt;
    int64_t col0, row0;
    int valid;
    bool act;
    __device__ FactTile(const TensorDev &T, uint32_t tile) {
        LC = 1u << T.lcl;
        RG = kThreads >> T.lcl;
        s = tile % T.strips;
        rt = tile / T.strips;
        lane = threadIdx.x & (LC - 1);
        rg = threadIdx.x >> T.lcl;
        col0 = int64_t(s) * 8 * LC + 8 * lane;
        act = col0 < T.m;
        valid = act ? (int)min(int64_t(8), T.m - col0) : 0;
        row0 = int64_t(rt) * T.tile_rows + rg;
    }
};

// A scale for the clamp-free test: NaN counts as +inf, so that a tile holding a
// NaN scale never takes the clamp-free path.
__device__ __forceinline__ float nan_to_inf(float v) { return v == v ? v : __int_as_float(0x7F800000); }

// a_i of the tile's rows and b_j of its strip (R, 1/sqrt(C), mean(R) read from L2).
// Returns (the same value in every thread) whether no element of the tile can
// reach the clamp: max_i a_i * max_j b_j <= 1/sqrt(eps), all scales finite. Then
// min(a_i * b_j, 1/sqrt(eps)) = a_i * b_j for every element (rounding is monotone).
__device__ bool fill_meta(const TensorDev &T, const TensorScal &S, uint32_t tile, float ce, Meta &meta) {
    const uint32_t s = tile % T.strips, rt = tile / T.strips, width = 8u << T.lcl;
    const float rbar_s = __ldcg(&S.rbar_s);
    const int rbar_e = __ldcg(&S.rbar_e);
    // (held apart from the descriptor, which the stores to shared memory may alias)
    const float *R = T.R, *bsc = T.bsc;
    const int64_t n = T.n, m = T.m;
    const uint32_t tile_rows = T.tile_rows;
    float ma = 0.f, mb = 0.f;
    for (uint32_t r = threadIdx.x; r < tile_rows; r += kThreads) {
        const int64_t i = int64_t(rt) * tile_rows + r;
        const float a = i < n ? row_scale(__ldcg(R + i), rbar_s, rbar_e) : 0.f;
        meta.rows[r] = a;
        ma = fmaxf(ma, nan_to_inf(a));
    }
    for (uint32_t c = threadIdx.x; c < width; c += kThreads) {
        const int64_t j = int64_t(s) * width + c;
        const float b = j < m ? __ldcg(bsc + j) : 0.f;
        meta.cols[c] = b;
        mb = fmaxf(mb, nan_to_inf(b));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        ma = fmaxf(ma, __shfl_xor_sync(kAll, ma, o));
        mb = fmaxf(mb, __shfl_xor_sync(kAll, mb, o));
    }
    if ((threadIdx.x & 31) == 0) {
        meta.red[threadIdx.x >> 5] = ma;
        meta.red[kThreads / 32 + (threadIdx.x >> 5)] = mb;
    }
    __syncthreads();
    ma = mb = 0.f;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        ma = fmaxf(ma, meta.red[w]);
        mb = fmaxf(mb, meta.red[kThreads / 32 + w]);
    }
    return ma * mb <= ce;
}

// ---------------------------------------------------------------------------
// Phase A: per-row / per-column sums of g^2 (Eq. 1).
// ---------------------------------------------------------------------------
// Adds the squares of one row-vector to the column partials; returns the row's
// sum over the LC lanes that share the row.
__device__ __forceinline__ float sumsq_row(const float (&g)[8], float (&col)[8], uint32_t LC) {
    float rs = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float q = g[c] * g[c];
        col[c] += q;
        rs += q;
    }
    for (uint32_t o = LC >> 1; o; o >>= 1) rs += __shfl_xor_sync(kAll, rs, o);
    return rs;
}

template <bool VEC>
__device__ void sumsq_tile(const TensorDev &T, uint32_t tile, Smem &sm, const Pol &pol) {
    const FactTile F(T, tile);
    const uint16_t *__restrict__ g_ = T.g;
    float *__restrict__ rowp = T.rowp + int64_t(F.s) * T.n;
    const int64_t n = T.n, m = T.m, row0 = F.row0, RG = F.RG, col0 = F.col0;
    const uint32_t LC = F.LC;
    const bool act = F.act, lane0 = F.lane == 0;
    const int vpt = (int)(T.tile_rows / F.RG);  // rows per thread (strip_rows)
    float col[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if constexpr (VEC) {
        constexpr int KCH = 8;  // row-vectors requested before the first is used
#pragma unroll 1
        for (int k0 = 0; k0 < vpt; k0 += KCH) {
            uint4 raw[KCH];
#pragma unroll
            for (int q = 0; q < KCH; ++q) {
                const int64_t i = row0 + (k0 + q) * RG;
                raw[q] = (act && i < n) ? ld16_hint(g_ + i * m + col0, pol.keep) : make_uint4(0, 0, 0, 0);
            }
            if (LC == 32) {
                // each lane holds partial sums of 8 rows; a transposed butterfly leaves
                // lane L with the full sum of row 4*b4 + 2*b3 + b2 (bits of L)
                float rs[KCH];
#pragma unroll
                for (int q = 0; q < KCH; ++q) {
                    float g[8];
                    unpack_bf8(raw[q], g);
                    float acc = 0.f;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const float sq = g[c] * g[c];
                        col[c] += sq;
                        acc += sq;
                    }
                    rs[q] = acc;
                }
                const uint32_t ln = threadIdx.x & 31;
                const bool b4 = ln & 16, b3 = ln & 8, b2 = ln & 4;
                float v4[4], v2[2];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float keep = b4 ? rs[q + 4] : rs[q], send = b4 ? rs[q] : rs[q + 4];
                    v4[q] = keep + __shfl_xor_sync(kAll, send, 16);
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float keep = b3 ? v4[q + 2] : v4[q], send = b3 ? v4[q] : v4[q + 2];
                    v2[q] = keep + __shfl_xor_sync(kAll, send, 8);
                }
                float v1 = (b2 ? v2[1] : v2[0]) + __shfl_xor_sync(kAll, b2 ? v2[0] : v2[1], 4);
                v1 += __shfl_xor_sync(kAll, v1, 2);
                v1 += __shfl_xor_sync(kAll, v1, 1);
                const int qs = (b4 ? 4 : 0) + (b3 ? 2 : 0) + (b2 ? 1 : 0);
                const int64_t i = row0 + (k0 + qs) * RG;
                if ((ln & 3) == 0 && i < n) rowp[i] = v1;
            } else {
#pragma unroll
                for (int q = 0; q < KCH; ++q) {
                    const int64_t i = row0 + (k0 + q) * RG;
                    float g[8];
                    unpack_bf8(raw[q], g);
                    const float rs = sumsq_row(g, col, LC);
                    if (lane0 && i < n) rowp[i] = rs;
                }
            }
        }
    } else {
        constexpr int KCH = 4;  // rows requested before the first is used
        // a row starts on a 16-byte boundary only where the width keeps it there (fp32 rows)
        const bool f32 = T.f32, wide = T.wal && (m & (f32 ? 3 : 7)) == 0;
#pragma unroll 1
        for (int k0 = 0; k0 < vpt; k0 += KCH) {
            if (int64_t(F.rt) * T.tile_rows + k0 * RG >= n) break;  // past the last row for every thread
            Raw8 raw[KCH];
#pragma unroll
            for (int q = 0; q < KCH; ++q) {
                const int64_t i = row0 + (k0 + q) * RG;
                load8_raw(g_, f32, wide, i * m + col0, act && i < n ? F.valid : 0, raw[q], pol);
            }
#pragma unroll
            for (int q = 0; q < KCH; ++q) {
                const int64_t i = row0 + (k0 + q) * RG;
                float g[8];
                values8(raw[q], f32, g);
                const float rs = sumsq_row(g, col, LC);
                if (lane0 && i < n) rowp[i] = rs;
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) sm.colred[threadIdx.x * 8 + c] = col[c];
    __syncthreads();
    const uint32_t width = 8 * LC;
    for (uint32_t cc = threadIdx.x; cc < width; cc += kThreads) {
        float acc = 0.f;
        for (uint32_t r = 0; r < F.RG; ++r) acc += sm.colred[r * width + cc];
        const int64_t j = int64_t(F.s) * width + cc;
        if (j < m) T.colp[int64_t(F.rt) * m + j] = acc;
    }
}

// ---------------------------------------------------------------------------
// Row path, phase A (k_rowsq): whole-row tiles of a momentum-free factored
// matrix. With a_i = sqrt(Rbar / R_i) and b_j = 1/sqrt(C_j), and no element at
// the clamp, sum_ij (g_ij a_i b_j)^2 = Rbar * sum_j (1 / C_j) * P_j with
// P_j = sum_i g_ij^2 / R_i. A tile holds whole rows, so it forms R_i (Eq. 1)
// itself and adds g_ij^2 / R_i into per-column partials of P; the column
// finalize then gives C_j and sum(U^2) without phase B re-reading G.
// Each chunk (kRowChunkBytes of consecutive rows, contiguous in memory) is
// brought to shared memory by one bulk copy completing on an mbarrier; the
// CTA keeps kRowStages chunks in flight.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

// One poll; the thread may be suspended for up to about kMbarSuspendNs while the
// phase is incomplete (a hint to the hardware).
constexpr uint32_t kMbarSuspendNs = 2000;

__device__ __forceinline__ bool mbar_try_wait(uint64_t *b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity), "n"(kMbarSuspendNs)
        : "memory");
    return ok != 0;
}

// Polls of one mbarrier wait before it gives up (about two seconds at the
// suspend hint): a copy that never lands ends the tile with a status word
// instead of hanging the GPU.
constexpr uint32_t kMbarPolls = 1u << 20;

__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity) {
    for (uint32_t i = 0; i < kMbarPolls; ++i)
        if (mbar_try_wait(b, parity)) return true;
    return false;
}

// After a wait gave up (status bit 2): one thread waits for chunks [c, issued_end) of a
// ring of `stages` slots that are still in flight, so that the CTA does not leave while
// a bulk copy may still write into its shared memory. Each gets up to eight more
// rounds of polls (about sixteen seconds); a copy still outstanding after that is
// recorded as status bit 4 and the CTA leaves anyway.
__device__ __noinline__ void drain_copies(uint32_t *err, uint64_t *full, uint32_t stages, uint32_t c,
                                          uint32_t issued_end) {
    atomicOr(err, 2u);
    for (uint32_t k = c; k < issued_end; ++k) {
        bool landed = false;
        for (int round = 0; round < 8 && !landed; ++round) landed = mbar_wait(&full[k % stages], (k / stages) & 1u);
        if (!landed) atomicOr(err, 4u);
    }
}

// Bulk copy global -> shared of `bytes` (multiple of 16, both ends 16-byte
// aligned), completing on mbarrier `bar`, with an L2 eviction policy.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}

// Orders this thread's earlier generic-proxy accesses of shared memory before
// its later async-proxy (bulk copy) accesses.
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// L2 policy of a bulk-copied read: kept for the next phase, or passing through.
__device__ __forceinline__ uint64_t read_policy(bool keep) {
    uint64_t p;
    if (keep)
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    else
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

struct RowSmem {
    uint4 buf[kRowStages][kRowChunkBytes / 16];  // the chunk ring (first member: 16-byte aligned)
    uint64_t full[kRowStages];                   // one mbarrier per ring slot
    float part[kThreads / 32][8];             // per-warp row partial sums of the chunk
    float inv[32];                               // 1 / R_i of the chunk's rows (0: no contribution)
};

// Rows `i` of chunk `c` of row tile `tile`: [i0, i0 + rows).
struct RowChunk {
    int64_t i0;
    uint32_t rows;
};

__device__ __forceinline__ RowChunk row_chunk(const TensorDev &T, uint32_t tile, uint32_t c) {
    const int64_t i0 = int64_t(tile) * T.rt_rows + int64_t(c) * T.cr;
    const int64_t left = T.n - i0;
    return RowChunk{i0, left <= 0 ? 0u : (uint32_t)min(left, (int64_t)T.cr)};
}

// Sum of N values p[0], p[stride], ..., p[(N - 1) stride] (N a power of two) by a
// balanced tree.
template <int N>
__device__ __forceinline__ float tree_sum(const float *p, int stride) {
    if constexpr (N == 1) {
        return p[0];
    } else {
        return tree_sum<N / 2>(p, stride) + tree_sum<N / 2>(p + (N / 2) * stride, stride);
    }
}

// Sum over a warp of K per-lane values, transposed: lane L ends with the total
// of value j(L) (K = 8: j = 4*b4 + 2*b3 + b2 of L's bits; K = 4: j = 2*b4 + b3;
// K = 2: j = b4), held by the lanes whose low 2, 3 or 4 bits are zero.
template <int K>
__device__ __forceinline__ float warp_sum_transposed(const float (&x)[K], int &j) {
    const uint32_t ln = threadIdx.x & 31;
    const bool b4 = ln & 16, b3 = ln & 8, b2 = ln & 4;
    if constexpr (K == 8) {
        float v4[4], v2[2];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float keep = b4 ? x[q + 4] : x[q], send = b4 ? x[q] : x[q + 4];
            v4[q] = keep + __shfl_xor_sync(kAll, send, 16);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float keep = b3 ? v4[q + 2] : v4[q], send = b3 ? v4[q] : v4[q + 2];
            v2[q] = keep + __shfl_xor_sync(kAll, send, 8);
        }
        float v1 = (b2 ? v2[1] : v2[0]) + __shfl_xor_sync(kAll, b2 ? v2[0] : v2[1], 4);
        v1 += __shfl_xor_sync(kAll, v1, 2);
        v1 += __shfl_xor_sync(kAll, v1, 1);
        j = (b4 ? 4 : 0) + (b3 ? 2 : 0) + (b2 ? 1 : 0);
        return v1;
    } else if constexpr (K == 2) {
        float v1 = (b4 ? x[1] : x[0]) + __shfl_xor_sync(kAll, b4 ? x[0] : x[1], 16);
        v1 += __shfl_xor_sync(kAll, v1, 8);
        v1 += __shfl_xor_sync(kAll, v1, 4);
        v1 += __shfl_xor_sync(kAll, v1, 2);
        v1 += __shfl_xor_sync(kAll, v1, 1);
        j = b4 ? 1 : 0;
        return v1;
    } else {
        float v2[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float keep = b4 ? x[q + 2] : x[q], send = b4 ? x[q] : x[q + 2];
            v2[q] = keep + __shfl_xor_sync(kAll, send, 16);
        }
        float v1 = (b3 ? v2[1] : v2[0]) + __shfl_xor_sync(kAll, b3 ? v2[0] : v2[1], 8);
        v1 += __shfl_xor_sync(kAll, v1, 4);
        v1 += __shfl_xor_sync(kAll, v1, 2);
        v1 += __shfl_xor_sync(kAll, v1, 1);
        j = (b4 ? 2 : 0) + (b3 ? 1 : 0);
        return v1;
    }
}

// Issues the bulk copy of chunk c of the tile into ring slot c % kRowStages.
__device__ __forceinline__ void row_issue(const TensorDev &T, uint32_t tile, uint32_t c, RowSmem &sm, uint64_t pol) {
    const RowChunk ch = row_chunk(T, tile, c);
    const uint32_t bytes = ch.rows * (uint32_t)T.m * 2u;
    const int st = c % kRowStages;
    mbar_expect_tx(&sm.full[st], bytes);
    bulk_g2s(sm.buf[st], T.g + ch.i0 * T.m, bytes, &sm.full[st], pol);
}

// Thread layout of a row-path kernel with TPB threads on rows of V = m / 8
// 16-byte vectors: NV vectors per thread per row (V > TPB), or RPP rows side by side
// (V < TPB); a thread owns vectors vi, vi + TPB, ... of row-in-pass rp.
template <int TPB, int V>
struct RowLayout {
    static constexpr int NV = V > TPB ? V / TPB : 1;
    static constexpr int RPP = V < TPB ? TPB / V : 1;
    static constexpr int WPR = (V < TPB ? V : TPB) / 32;  // warps per row-in-pass
    int rp, vi;
    __device__ RowLayout() : rp(threadIdx.x / (V < TPB ? V : TPB)), vi(threadIdx.x % (V < TPB ? V : TPB)) {}
};

// k_rowsq on TPB threads, rows of m = 8 V: chunks of CS = 2048 / V rows (32 KB),
// K = CS / RPP rows per thread per chunk.
template <int TPB, int V>
__device__ void rowsq_tile(const StepArgs &A, const TensorDev &T, TensorScal &S, uint32_t tile, RowSmem &sm) {
    using L = RowLayout<TPB, V>;
    constexpr int NV = L::NV, RPP = L::RPP, WPR = L::WPR;
    constexpr int CS = 2048 / V;
    constexpr int K = CS / RPP;
    static_assert(K == 4 || K == 8, "rows per thread per chunk");
    static_assert(CS <= 32, "chunk rows");
    const L lay;
    const uint64_t pol = read_policy(T.keep);
    const uint32_t nch = (uint32_t)min((int64_t)(T.rt_rows / T.cr), (T.n - int64_t(tile) * T.rt_rows + T.cr - 1) / T.cr);
    if (threadIdx.x == 0) {
        for (int st = 0; st < kRowStages; ++st) mbar_init(&sm.full[st], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (uint32_t c = 0; c < nch && c < (uint32_t)kRowStages; ++c) row_issue(T, tile, c, sm, pol);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float b2 = A.b2, c2 = grad_scale(A).c2, inv_m = 1.0f / (float)(8 * V);  // m is a power of two: exact
    // per column pair: sums of g^2, the compensated (hi, lo) sum of g^2 / R_i and its open fp32 part
    float2 cs[NV][4], ph[NV][4], pl[NV][4], t[NV][4];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int q = 0; q < 4; ++q) cs[v][q] = ph[v][q] = pl[v][q] = t[v][q] = make_float2(0.f, 0.f);
    double rsum = 0.0;                       // threads < CS: sum of the R of this chunk-row position
    float rmin = __int_as_float(0x7F800000);  // threads < CS: smallest positive R of it
    bool zero_row = false;

    // the tile's rows and R, held in registers (the stores to R in the loop could
    // otherwise make the compiler reload them from the descriptor every chunk)
    const int64_t row0 = int64_t(tile) * T.rt_rows, n = T.n;
    const uint32_t cr = T.cr;
    float *__restrict__ Rg = T.R;
    uint32_t c = 0;
    for (; c < nch; ++c) {
        const int st = c % kRowStages;
        const uint32_t par = (c / kRowStages) & 1u;
        const int64_t ci0 = row0 + int64_t(c) * cr;
        const RowChunk ch{ci0, (uint32_t)min(n - ci0, (int64_t)cr)};
        float rp = 0.f;
        if (tid < (int)ch.rows) rp = __ldcg(Rg + ch.i0 + tid);
        const bool ok = mbar_wait(&sm.full[st], par);
        const uint4 *buf = sm.buf[st];
        // a full chunk (every chunk but a tensor's last) needs no row bound checks
        const bool full = ch.rows == (uint32_t)CS;
        // pass 1: row sums and column sums of g^2 (rows lay.rp + RPP k of the chunk)
        float rs[K];
        auto pass1 = [&](auto full_c) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int r = lay.rp + RPP * k;
                float2 r2 = make_float2(0.f, 0.f);
                if (decltype(full_c)::value || r < (int)ch.rows) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        float2 g[4];
                        unpack_bf8x2(buf[r * V + v * TPB + lay.vi], g);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {  // g^2 into the column and row sums, one rounding each
                            cs[v][q] = __ffma2_rn(g[q], g[q], cs[v][q]);
                            r2 = __ffma2_rn(g[q], g[q], r2);
                        }
                    }
                }
                rs[k] = r2.x + r2.y;
            }
        };
        if (full)
            pass1(std::true_type{});
        else
            pass1(std::false_type{});
        int j;
        const float tot = warp_sum_transposed<K>(rs, j);
        if ((lane & (K == 8 ? 3 : 7)) == 0) sm.part[warp][j] = tot;
        if (__syncthreads_or(!ok)) break;  // every slot before this one has landed
        // slot of chunk c - 1 is free (its pass 2 preceded this barrier): refill it
        // (from warp 1: warp 0 forms the chunk's row scales, which the CTA waits for)
        if (tid == 32 && c >= 1 && c - 1 + kRowStages < nch) {
            fence_proxy_async_smem();
            row_issue(T, tile, c - 1 + kRowStages, sm, pol);
        }
        float Rn = 0.f, sum = 0.f;
        if (tid < (int)ch.rows) {  // chunk row r = tid: row-in-pass r % RPP, its k = r / RPP
            const int w0 = (tid % RPP) * WPR, kr = tid / RPP;
            sum = tree_sum<WPR>(&sm.part[w0][kr], 8);
            Rn = fmaf(b2, rp, c2 * (sum * inv_m));
            sm.inv[tid] = Rn > 0.f && Rn < __int_as_float(0x7F800000) ? __frcp_rn(Rn) : 0.f;
        }
        __syncthreads();
        if (tid < (int)ch.rows) {  // the row's R and the tile's statistics, off the barrier's path
            Rg[ch.i0 + tid] = Rn;
            rsum += (double)Rn;
            if (Rn > 0.f && Rn < __int_as_float(0x7F800000))
                rmin = fminf(rmin, Rn);
            else if (!(Rn == 0.f && sum == 0.f))
                zero_row = true;  // content in a row with R_i == 0, or a non-finite R_i
        }
        // pass 2: P_j += g^2 / R_i, summed in fp32 over four chunks (at most 4 K rows)
        // per column, then folded into (hi, lo)
        auto pass2 = [&](auto full_c) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int r = lay.rp + RPP * k;
                if (decltype(full_c)::value || r < (int)ch.rows) {
                    const float iv = sm.inv[r];
                    const float2 iv2 = make_float2(iv, iv);
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        float2 g[4];
                        unpack_bf8x2(buf[r * V + v * TPB + lay.vi], g);
#pragma unroll
                        for (int q = 0; q < 4; ++q) t[v][q] = __ffma2_rn(__fmul2_rn(g[q], g[q]), iv2, t[v][q]);
                    }
                }
            }
        };
        if (full)
            pass2(std::true_type{});
        else
            pass2(std::false_type{});
        if ((c & 3u) == 3u || c + 1 == nch) {
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float2 s2, e2;
                    two_sum2(ph[v][q], t[v][q], s2, e2);
                    ph[v][q] = s2;
                    pl[v][q] = __fadd2_rn(pl[v][q], e2);
                    t[v][q] = make_float2(0.f, 0.f);
                }
        }
    }
    if (c < nch) {
        // A chunk did not land in time: record it, wait (bounded) for the copies in
        // flight and drop the tile. Issued so far: chunks [0, kRowStages) by the
        // prologue and chunk k - 1 + kRowStages at each iteration k in [1, c); chunks
        // before c have landed.
        if (tid == 0)
            drain_copies(A.err, sm.full, kRowStages, c, min(nch, c == 0 ? (uint32_t)kRowStages : c + kRowStages - 1));
        return;
    }
    // per-tile partials, (sum of g^2, sum of g^2 / R_i) per column (the RPP threads that
    // share a column vector are added in row-in-pass order; the compensated sum of
    // g^2 / R_i is rounded to fp32 once), the tile's sum and smallest positive R
    const int64_t base = int64_t(tile) * 8 * V;
    if constexpr (RPP == 1) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int64_t col = 8 * int64_t(v * TPB + lay.vi);
            float4 *pp4 = reinterpret_cast<float4 *>(T.pp + base + col);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                pp4[q] = make_float4(cs[v][q].x, pair_f(ph[v][q].x, pl[v][q].x), cs[v][q].y,
                                     pair_f(ph[v][q].y, pl[v][q].y));
        }
    } else {
        // the ring is free (every chunk consumed before the last barrier): stage there
        float *mcs = reinterpret_cast<float *>(sm.buf[0]);        // [TPB][8]
        float2 *mpp = reinterpret_cast<float2 *>(sm.buf[1]);      // [TPB][8] (hi, lo)
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            mcs[tid * 8 + 2 * q] = cs[0][q].x;
            mcs[tid * 8 + 2 * q + 1] = cs[0][q].y;
            mpp[tid * 8 + 2 * q] = make_float2(ph[0][q].x, pl[0][q].x);
            mpp[tid * 8 + 2 * q + 1] = make_float2(ph[0][q].y, pl[0][q].y);
        }
        __syncthreads();
        for (int e = tid; e < 8 * V; e += TPB) {  // column e = 8 vi + q
            const int vi = e >> 3, q = e & 7;
            float cc = 0.f;
            Acc2 pq;
#pragma unroll
            for (int r = 0; r < RPP; ++r) {
                cc += mcs[(r * V + vi) * 8 + q];
                const float2 h = mpp[(r * V + vi) * 8 + q];
                pq.add(h.x);
                pq.lo += h.y;
            }
            T.pp[base + e] = make_float2(cc, pair_f(pq.hi, pq.lo));
        }
    }
    if (zero_row) atomicOr(&S.zflag, 1u);
    if (warp == 0) {  // CS <= 32: the chunk-row positions are lanes of warp 0
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            rsum += __shfl_xor_sync(kAll, rsum, o);
            rmin = fminf(rmin, __shfl_xor_sync(kAll, rmin, o));
        }
        if (lane == 0) {
            T.rsum[tile] = rsum;
            T.rmin[tile] = rmin;
        }
    }
}

// sum_{r < cnt} p[r * stride] (values an earlier launch wrote), added in order
// r = 0, 1, ...; the loads are issued eight at a time ahead of the adds.
template <typename V>
__device__ __forceinline__ V strided_sum(const V *p, int64_t stride, uint32_t cnt) {
    V s = V(0);
    uint32_t r = 0;
    for (; r < cnt; r += 8) {
        V v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = r + q < cnt ? __ldcg(p + int64_t(r + q) * stride) : V(0);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (r + q < cnt) s += v[q];
    }
    return s;
}

// mean(R) and its [1, 2) mantissa / exponent split (used by the row scales).
__device__ void set_rbar(TensorScal &S, double rbar) {
    S.rbar = rbar;
    if (rbar > 0.0) {
        int e;
        const double fr = frexp(rbar, &e);  // rbar = fr * 2^e, fr in [0.5, 1)
        S.rbar_s = (float)(2.0 * fr);       // in [1, 2]
        S.rbar_e = 1 - e;                   // rbar * 2^(1-e) = 2 fr
    } else {
        S.rbar_s = 0.f;
        S.rbar_e = 0;
    }
}

// The exponent of gamma (floor of its log2; 0 where that has no value), within an fp32 factor's range.
__device__ __forceinline__ int gamma_exponent(float gam) {
    if (!(gam > 0.f && gam < __int_as_float(0x7F800000))) return 0;
    int e;
    frexpf(gam, &e);
    return min(max(e - 1, -126), 126);
}

// U = coef * y / D: a momentum-free tensor's y is g, so its coef carries gamma (M already does).
__device__ __forceinline__ double update_coef(const StepArgs &A, const TensorDev &T) {
    return T.momentum ? A.coef_mom : A.coef_plain * (double)grad_scale(A).gam;
}

// From s = sum of (U / coef)^2: sum(U^2), RMS(U), the clip factor
// kappa = 1 / max(1, RMS / d) (Sec. 3 update clipping) and lr * kappa * coef.
__device__ void set_clip(const StepArgs &A, const TensorDev &T, TensorScal &S, double s) {
    const double coef = update_coef(A, T);
    const double su2 = s * coef * coef;
    const double rms = sqrt(su2 * T.inv_numel);
    const double d = (double)A.clip_d;
    const double kappa = rms > d ? d / rms : 1.0;  // a NaN RMS clips nothing, as fmax(1, NaN) = 1
    S.sumsq = su2;
    S.rms = rms;
    S.kappa = kappa;
    S.coefC = (float)((double)A.lr * kappa * coef);
}

// Row path, finalize item `local` (kFinChunk columns): C_j, 1/sqrt(C_j) and the
// chunk's sum of P_j / C_j. The last item of the tensor forms mean(R) and, when
// no element can reach the clamp (max_i a_i^2 * max_j b_j^2 <= 1/eps over rows and
// columns that hold gradient), sum(U^2) = coef^2 * mean(R) * sum_j P_j / C_j and
// the clip factor; otherwise, unless a bound on sum(U^2) already makes the clip factor 1
// (phase C then adds it up), it queues the tensor for phase B. P_j and the sums
// of P_j / C_j are compensated fp32 (hi, lo) pairs: fp64 arithmetic runs at a
// small fraction of the fp32 rate here, and every term is non-negative, so a
// pair keeps the sum to about fp64 accuracy and each quotient to one fp32 rounding.
__device__ void phase_F_row(const StepArgs &A, const TensorDev &T, uint32_t t, uint32_t local, Smem &sm) {
    TensorScal &S = A.scal[t];
    const float inf = __int_as_float(0x7F800000);
    // the item's fci columns, kFinChunk / fci threads per column: thread tid adds the
    // tiles r = sl, sl + tpc, ... of column cix (consecutive threads, consecutive columns)
    const int fci = (int)T.fci, tpc = kFinChunk / fci;
    const int cix = threadIdx.x % fci, sl = threadIdx.x / fci;
    const int64_t j = int64_t(local) * fci + cix;
    float cs = 0.f;  // this thread's tiles: sum of g^2 (in tile order) and, compensated, of g^2 / R_i
    Acc2 pa;
    if (j < T.m) {
        const float2 *p = T.pp + j;
        uint32_t r = sl;
        // loads issued 32 at a time ahead of the adds, which go in tile order
        for (; r + 31 * tpc < T.rtiles; r += 32 * tpc) {
            float2 v[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = __ldcg(p + int64_t(r + q * tpc) * T.m);
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                cs += v[q].x;
                pa.add(v[q].y);
            }
        }
        // the rest eight at a time (one at a time each tile would cost a trip to L2)
        for (; r < T.rtiles; r += 8 * tpc) {
            float2 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (r + q * tpc < T.rtiles) v[q] = __ldcg(p + int64_t(r + q * tpc) * T.m);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (r + q * tpc < T.rtiles) {
                    cs += v[q].x;
                    pa.add(v[q].y);
                }
        }
    }
    // without momentum P_j grows with 1 / gamma^2, and P_j / C_j with more than that: P_j is taken times 2^2e for
    // gamma's exponent e, which is exact, and the sum in fp64 divided by it (a gamma of 2^-45 overflowed, to a clip
    // factor of 0)
    const int ge = T.momentum ? 0 : gamma_exponent(grad_scale(A).gam);
    const float pscale = __int_as_float((ge + 127) << 23);
    // the column's tpc parts in slice order
    float *red = sm.colred;  // [3][kFinChunk]: sum g^2, hi, lo
    red[threadIdx.x] = cs;
    red[kFinChunk + threadIdx.x] = pa.hi;
    red[2 * kFinChunk + threadIdx.x] = pa.lo;
    __syncthreads();
    Acc2 contrib;
    float cmin = inf, gsum = 0.f;
    if (sl == 0 && j < T.m) {
        const float Cold = __ldcg(T.C + j);
        for (int k = 1; k < tpc; ++k) {
            cs += red[k * fci + cix];
            pa.add(red[kFinChunk + k * fci + cix]);
            pa.lo += red[2 * kFinChunk + k * fci + cix];
        }
        const float P = pair_f(pa.hi, pa.lo);
        gsum = cs;
        const float mean = __fdiv_rn(cs, (float)T.n);
        const float Cn = fmaf(A.b2, Cold, grad_scale(A).c2 * mean);
        T.C[j] = Cn;
        T.bsc[j] = __frsqrt_rn(Cn);
        if (P > 0.f) {
            if (Cn > 0.f && Cn < inf) {
                contrib.add(__fdiv_rn(P * pscale * pscale, Cn));
                cmin = Cn;
            } else {
                atomicOr(&S.zflag, 1u);  // gradient in a column whose C_j is 0 or not finite
            }
        } else if (!(P == 0.f)) {
            atomicOr(&S.zflag, 1u);  // NaN
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        cmin = fminf(cmin, __shfl_xor_sync(kAll, cmin, o));
        gsum += __shfl_xor_sync(kAll, gsum, o);
    }
    __syncthreads();  // the column parts in colred are consumed
    if ((threadIdx.x & 31) == 0) {
        sm.colred[threadIdx.x >> 5] = cmin;
        sm.colred[kThreads / 32 + (threadIdx.x >> 5)] = gsum;
    }
    const float2 cs2 = block_sum2(contrib, sm.red2);  // its barriers also publish colred
    if (threadIdx.x == 0) {
        gsum = 0.f;
        for (int w = 0; w < kThreads / 32; ++w) {
            cmin = fminf(cmin, sm.colred[w]);
            gsum += sm.colred[kThreads / 32 + w];
        }
        T.fsum[local] = pair_value(cs2.x, cs2.y);
        T.fmin[local] = cmin;
        T.pp[int64_t(local) * fci].x = gsum;  // the item's partials are consumed
        sm.last = (atom_add_acq_rel(&S.cntF, 1u) == T.nfc - 1);
    }
    __syncthreads();
    if (!sm.last) return;
    // Last item of the tensor: the whole CTA sums the row tiles' R sums and minima and
    // the items' sums and minima (thread k takes entries k, k + kThreads, ...; then a
    // fixed shuffle tree: the same order every step).
    double rs = 0.0, fs = 0.0, gs = 0.0;
    float rmn = inf, cmn = inf;
    for (uint32_t r = threadIdx.x; r < T.rtiles; r += kThreads) {
        rs += __ldcg(T.rsum + r);
        rmn = fminf(rmn, __ldcg(T.rmin + r));
    }
    for (uint32_t f = threadIdx.x; f < T.nfc; f += kThreads) {
        fs += __ldcg(T.fsum + f);
        gs += (double)__ldcg(&T.pp[int64_t(f) * fci].x);
        cmn = fminf(cmn, __ldcg(T.fmin + f));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        rmn = fminf(rmn, __shfl_xor_sync(kAll, rmn, o));
        cmn = fminf(cmn, __shfl_xor_sync(kAll, cmn, o));
        rs += __shfl_xor_sync(kAll, rs, o);
        fs += __shfl_xor_sync(kAll, fs, o);
        gs += __shfl_xor_sync(kAll, gs, o);
    }
    if ((threadIdx.x & 31) == 0) {  // colred was last read before the barrier above
        const int w = threadIdx.x >> 5;
        sm.colred[w] = rmn;
        sm.colred[kThreads / 32 + w] = cmn;
        sm.redd[w] = rs;
        sm.redd[kThreads / 32 + w] = fs;
        sm.redd[2 * (kThreads / 32) + w] = gs;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        rs = fs = gs = 0.0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            rmn = fminf(rmn, sm.colred[w]);
            cmn = fminf(cmn, sm.colred[kThreads / 32 + w]);
            rs += sm.redd[w];
            fs += sm.redd[kThreads / 32 + w];
            gs += sm.redd[2 * (kThreads / 32) + w];
        }
        const double rbar = rs * T.inv_n;
        set_rbar(S, rbar);
        const double sum = fs * rbar * __hiloint2double((1023 - 2 * ge) << 20, 0);
        // max_i a_i^2 = Rbar / min R_i over rows with R_i > 0; max_j b_j^2 = 1 / min C_j over columns
        // holding gradient (0 without any). Multiplied out: fp64 divides are slow here.
        const bool some = rmn < inf && cmn < inf;
        const double ce2 = (double)A.ce * (double)A.ce;
        // (a sum that overflowed fp32, from gradients of 1e-16 with a lower eps still: phase B or phase C adds it up)
        if (__ldcg(&S.zflag) == 0u && isfinite(sum) && (!some || rbar <= ce2 * (1.0 - 1e-6) * ((double)rmn * (double)cmn))) {
            set_clip(A, T, S, sum);
        } else {
            // A clamp may bind, and it only lowers |U|: no element is above its unclamped value or
            // coef |y| / sqrt(eps), so sum(U^2) is at most the bilinear sum, and (without momentum,
            // whose sum of y^2 is not at hand) coef^2 sum(g^2) / eps. Where the lower of the two
            // leaves RMS(U) below d, by more than the fp32 sums can be off, the clip factor is 1
            // whatever sum(U^2) is, and phase C, which forms every U anyway, adds it up: at the
            // paper's hyper-parameters (eps 1e-8 above most g^2) that saves every tensor's phase B,
            // 850M parameters 1724 -> 1205 us (phase B 572 us, the sums 32 us of phase C).
            const double ub = T.momentum ? sum : fmin(sum, gs * ce2);
            const double coef = update_coef(A, T);
            if (__ldcg(&S.zflag) == 0u && ub * coef * coef * T.inv_numel <= (double)A.clip_d * (double)A.clip_d * (1.0 - 1e-4)) {
                S.kappa = 1.0;
                S.coefC = (float)((double)A.lr * coef);
                S.fallback = kSumInC;
            } else {
                S.fallback = kPhaseB;
                const uint32_t q = atomicAdd(A.fb, 1u);
                A.fb[1 + q] = t;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Phase F: factor EMAs, 1/sqrt(C_j), mean(R) (Eq. 1).
// ---------------------------------------------------------------------------
__device__ void phase_F(const StepArgs &A, const TensorDev &T, uint32_t t, uint32_t local, Smem &sm) {
    TensorScal &S = A.scal[t];
    if (T.rowpath) {
        phase_F_row(A, T, t, local, sm);
        return;
    }
    if (local < T.nfr) {
        const int64_t i = int64_t(local) * kFinChunk + threadIdx.x;
        double rd = 0.0;
        if (threadIdx.x < kFinChunk && i < T.n) {
            const float rs = strided_sum(T.rowp + i, T.n, T.strips);
            const float mean = __fdiv_rn(rs, (float)T.m);
            const float Rn = fmaf(A.b2, T.R[i], grad_scale(A).c2 * mean);
            T.R[i] = Rn;
            rd = (double)Rn;
        }
        rd = block_sum_d(rd, sm.redd);
        if (threadIdx.x == 0) T.rsum[local] = rd;
    } else {
        // fci columns per item, kFinChunk / fci threads per column, each with every (kFinChunk / fci)-th tile
        const int fci = (int)T.fci, tpc = kFinChunk / fci, cix = threadIdx.x % fci, sl = threadIdx.x / fci;
        const int64_t j = int64_t(local - T.nfr) * fci + cix;
        float cs = 0.f;
        if (j < T.m && sl < (int)T.rowtiles)
            cs = strided_sum(T.colp + int64_t(sl) * T.m + j, T.m * tpc, (T.rowtiles - sl + tpc - 1) / tpc);
        sm.colred[threadIdx.x] = cs;
        __syncthreads();
        if (sl == 0 && j < T.m) {
            for (int k = 1; k < tpc; ++k) cs += sm.colred[k * fci + cix];
            const float mean = __fdiv_rn(cs, (float)T.n);
            const float Cn = fmaf(A.b2, T.C[j], grad_scale(A).c2 * mean);
            T.C[j] = Cn;
            T.bsc[j] = __frsqrt_rn(Cn);
        }
    }
    // The last finalize item of the tensor forms mean(R) from the row items' partial sums.
    __syncthreads();
    if (threadIdx.x == 0) sm.last = (atom_add_acq_rel(&S.cntF, 1u) == T.nfr + T.nfc - 1);
    __syncthreads();
    if (!sm.last) return;
    double s = 0.0;  // the CTA sums the row items' partials (fixed partition and tree)
    for (uint32_t f = threadIdx.x; f < T.nfr; f += kThreads) s += __ldcg(T.rsum + f);
    s = block_sum_d(s, sm.redd);
    if (threadIdx.x == 0) set_rbar(S, s * T.inv_n);
}

// ---------------------------------------------------------------------------
// Phase B: second moment / momentum update and sum(U^2) (Algorithm 1).
// ---------------------------------------------------------------------------
// U (up to its scalar) of one row-vector of a factored tile, squared and summed into acc.
__device__ __forceinline__ void rms_row(const float (&y)[8], float a, const float (&b)[8], int valid, float ce,
                                        Acc2 &acc) {
    float u[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) u[c] = c < valid ? y[c] * fminf(a * b[c], ce) : 0.f;
    acc.add(sumsq8(u));
}

template <bool MOM>
__device__ Acc2 rms_fact_tile(const StepArgs &A, const TensorDev &T, uint32_t tile, const Meta &meta,
                              const Pol &pol) {
    const FactTile F(T, tile);
    Acc2 acc;
    if (!F.act) return acc;
    const uint16_t *__restrict__ g_ = T.g;
    float *__restrict__ M_ = T.M;
    const int64_t n = T.n, m = T.m, row0 = F.row0, RG = F.RG, col0 = F.col0;
    const float b1 = A.b1, c1 = grad_scale(A).c1, ce = A.ce;
    const float *rows = meta.rows + F.rg;
    const int vpt = (int)(T.tile_rows / F.RG);
    float b[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) b[c] = meta.cols[F.lane * 8 + c];
    {
        // row-vectors requested together: eight when only g streams, four with the momentum
        constexpr int KCH = MOM ? 4 : 8;
#pragma unroll 1
        for (int k0 = 0; k0 < vpt; k0 += KCH) {
            uint4 graw[KCH];
            float4 mraw[MOM ? KCH : 1][2];
#pragma unroll
            for (int q = 0; q < KCH; ++q) {
                const int64_t i = row0 + (k0 + q) * RG;
                const int64_t e0 = (i < n ? i : 0) * m + col0;
                if (i < n) graw[q] = ld16_hint(g_ + e0, MOM ? pol.drop : pol.keep);
                if (MOM && i < n) {
                    mraw[MOM ? q : 0][0] = *reinterpret_cast<const float4 *>(M_ + e0);
                    mraw[MOM ? q : 0][1] = *reinterpret_cast<const float4 *>(M_ + e0 + 4);
                }
            }
#pragma unroll
            for (int q = 0; q < KCH; ++q) {
                const int64_t i = row0 + (k0 + q) * RG;
                if (i < n) {
                    float y[8];
                    unpack_bf8(graw[q], y);
                    if (MOM) {
                        const float4 m0 = mraw[MOM ? q : 0][0], m1 = mraw[MOM ? q : 0][1];
                        const float mm[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
                        for (int c = 0; c < 8; ++c) y[c] = fmaf(b1, mm[c], c1 * y[c]);
                        store_f8(M_ + i * m + col0, true, 8, y);
                    }
                    rms_row(y, rows[(k0 + q) * RG], b, 8, ce, acc);
                }
            }
        }
    }
    return acc;
}

// ---------------------------------------------------------------------------
// Phases B and C of factored tensors without 16-byte row-vectors (fp32, widths that are not a
// multiple of 8, unaligned pointers): flat tiles of 8 consecutive elements per thread and round, which
// are loaded wide wherever the arrays start on a 16-byte boundary and draw one Philox block, whatever
// the width. Bound by latency; the row-vectors' layout had 8 narrow loads per row, a Philox block per
// element and 32 rows per thread one after another (k_apply, 42829 x 58 bf16: 103 -> 18 us; 3467 x
// 1072 fp32 with momentum: 45 -> 20; 24 ragged tensors of 13M elements in all: a step 215 -> 102).
// ---------------------------------------------------------------------------
// The scales of a tile (a_i of its rows, b_j of its columns) stay in shared memory, and a round is one
// vector per thread; FlatTile says which, FlatScales what its elements are scaled by. The b_j of columns 8
// apart lie side by side, so that the lanes of a warp, 8 columns apart, read different banks: column k + s is at
// [s][k / 8] for every k that is a multiple of 8 and s below 15, so that a vector from any column on
// reads one word of 8 consecutive of these 15 lists, and 7 columns more than the tile has repeat the first, which
// a vector may run on into. (With the b_j in column order every load was an 8-way bank conflict: a step of 28160 x
// 4096 bf16 off a 16-byte boundary, converted beside its loads too, 926 us, 958 with momentum, and on strip tiles of
// narrow loads 747 and 938; 624 and 690 so.)
struct FlatVec {
    int64_t e;  // its first element; at or past numel: none in this round
    int r, j;   // row and column, from the tile's first
};

template <bool WIDE>
struct FlatScales {
    const float *a, *b;
    int pitch;  // of the lists
    int end;    // the column at which the next row begins
    static constexpr int kLists = 15;
    // room for `cols` + 7 columns, 4 words past a multiple of 32 (the lanes that fill the lists: different banks)
    static __host__ __device__ constexpr int pitch_for(int cols) { return ((cols + 14) / 8 + 27) / 32 * 32 + 4; }
    static __device__ __forceinline__ void put(float *pool, int pitch, int k, float bk) {
        const int s = k & 7, q = k >> 3;
        pool[s * pitch + q] = bk;
        if (s < 7 && q > 0) pool[(s + 8) * pitch + q - 1] = bk;
    }
    // min(a_i b_j, 1/sqrt(eps)) of the vector's `valid` elements, some finite value past them
    __device__ __forceinline__ void operator()(const FlatVec &v, int valid, float ce, float (&sc)[8]) const {
        if (!WIDE && end < 8) {  // rows shorter than a vector: b_j in order
            int r = v.r, j = v.j;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                sc[c] = c < valid ? fminf(a[r] * b[j], ce) : 0.f;
                const bool wrap = ++j == end;
                j = wrap ? 0 : j;
                r += wrap;
            }
            return;
        }
        const float *p = b + (v.j & 7) * pitch + (v.j >> 3);
        const int here = end - v.j;  // elements in this row
        const float ar = a[v.r], an = here < valid ? a[v.r + 1] : 0.f;
        if (!WIDE && end < 8 * 32) {  // a warp holds the end of a row
#pragma unroll
            for (int c = 0; c < 8; ++c) sc[c] = fminf((c < here ? ar : an) * p[c * pitch], ce);
            return;
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) sc[c] = fminf(ar * p[c * pitch], ce);
        if (here < valid) {
#pragma unroll
            for (int c = 1; c < 8; ++c)
                if (c >= here) sc[c] = fminf(an * p[c * pitch], ce);
        }
    }
};

// Matrices of at most kFlatCols columns: 2048 fvpt consecutive elements, and b_j of all columns.
template <bool WIDE>
struct FlatTile {
    FlatScales<WIDE> scales;
    int64_t e0;
    int at, r, j;   // of the next round's vector: elements from e0, row, column
    int dq, dr, m;  // one round of the CTA, 8 kThreads elements, in rows and columns
    __device__ FlatTile(const TensorDev &T, const TensorScal &S, uint32_t tile, Meta &meta) {
        const int64_t elems = int64_t(8 * kThreads) * T.fvpt;
        e0 = int64_t(tile) * elems;
        const int count = (int)min(elems, T.numel - e0);
        m = (int)T.m;
        // (64-bit divides are long here)
        const int64_t row0 = T.numel < (int64_t(1) << 31) ? (uint32_t)e0 / (uint32_t)m : e0 / m;
        const int col0 = (int)(e0 - row0 * m), rows = (int)((uint32_t)(col0 + count - 1) / (uint32_t)m) + 1;
        const float rbar_s = __ldcg(&S.rbar_s);
        const int rbar_e = __ldcg(&S.rbar_e);
        const int pitch = m < 8 ? 1 : FlatScales<WIDE>::pitch_for(m);
        float *pool = reinterpret_cast<float *>(&meta), *pa = pool + FlatScales<WIDE>::kLists * pitch;
        __builtin_assume(__isShared(pool));
        scales = FlatScales<WIDE>{pa, pool, pitch, m};
        // (pointers held apart from the descriptor, which the stores to shared memory may alias)
        const float *R = T.R + row0, *bsc = T.bsc;
        for (int k = threadIdx.x; k < rows; k += kThreads) pa[k] = row_scale(__ldcg(R + k), rbar_s, rbar_e);
        for (int k = threadIdx.x; k < m; k += kThreads) {
            const float bj = __ldcg(bsc + k);
            FlatScales<WIDE>::put(pool, pitch, k, bj);
            if (k < 7 && m >= 8) FlatScales<WIDE>::put(pool, pitch, m + k, bj);
        }
        __syncthreads();
        at = 8 * threadIdx.x;
        r = (int)((uint32_t)(col0 + at) / (uint32_t)m);
        j = col0 + at - r * m;
        dq = 8 * kThreads / m;
        dr = 8 * kThreads - dq * m;
    }
    __device__ __forceinline__ FlatVec next() {
        const FlatVec v{e0 + at, r, j};
        at += 8 * kThreads;
        r += dq;
        j += dr;
        if (j >= m) {
            j -= m;
            ++r;
        }
        return v;
    }
};

// Wider ones: kFlatStrip columns, 2 rows to a round, so that a tile needs kFlatStrip + 7 column
// scales whatever the width. A vector starts at a multiple of 8 of the matrix and belongs to the strip that its
// first element lies in; from the last strip it may run on into the next row. Reading every b_j from L2 instead
// (tiles of consecutive elements), a step of 2295 x 50257 bf16 took 1400 us, 1433 with momentum, and on strip tiles
// of narrow loads 925 and 1088; 461 and 557 so.
template <>
struct FlatTile<true> {
    FlatScales<true> scales;
    static constexpr int kLanes = kFlatStrip / 8, kRows = kThreads / kLanes;  // threads of a row; rows of a round
    int64_t first, m, numel;  // the first element, in the strip, of the thread's row of the next round
    int width, r, rows;       // columns of the strip; that row; rows of the tile
    __device__ FlatTile(const TensorDev &T, const TensorScal &S, uint32_t tile, Meta &meta) {
        const uint32_t strips = (uint32_t)((T.m + kFlatStrip - 1) / kFlatStrip), rt = tile / strips;
        const int64_t c0 = int64_t(tile - rt * strips) * kFlatStrip, i0 = int64_t(rt) * kRows * T.fvpt;
        m = T.m;
        numel = T.numel;
        width = (int)min(m - c0, int64_t(kFlatStrip));
        rows = (int)min(int64_t(kRows) * T.fvpt, T.n - i0);
        r = (int)threadIdx.x / kLanes;
        first = (i0 + r) * m + c0;
        const float rbar_s = __ldcg(&S.rbar_s);
        const int rbar_e = __ldcg(&S.rbar_e);
        constexpr int kPitch = FlatScales<true>::pitch_for(kFlatStrip), kWords = FlatScales<true>::kLists * kPitch;
        static_assert(kWords + kRows * kVecPerThread + 1 <= kSmemFloats && kRows * kVecPerThread < kThreads, "the scales fit");
        float *pool = reinterpret_cast<float *>(&meta), *pa = pool + kWords;
        __builtin_assume(__isShared(pool));
        scales = FlatScales<true>{pa, pool, kPitch, (int)min(m - c0, int64_t(2 * kFlatStrip))};
        const float *R = T.R + i0, *bsc = T.bsc;
        // (and of the row that the tile's last vector may run into)
        if (threadIdx.x <= rows && i0 + threadIdx.x < T.n) pa[threadIdx.x] = row_scale(__ldcg(R + threadIdx.x), rbar_s, rbar_e);
        for (int k = threadIdx.x; k < width + 7; k += kThreads)
            FlatScales<true>::put(pool, kPitch, k, __ldcg(bsc + (c0 + k < m ? c0 + k : c0 + k - m)));
        __syncthreads();
    }
    __device__ __forceinline__ FlatVec next() {
        const int j = (-(int)first & 7) + 8 * (int)(threadIdx.x % kLanes);  // from the strip's first column
        const FlatVec v{r < rows && j < width ? first + j : numel, r, j};
        first += kRows * m;
        r += kRows;
        return v;
    }
};
constexpr uint32_t kFlatAhead = 2;  // rounds of a flat tile whose loads are issued together

template <bool WIDE>
__device__ Acc2 rms_flat_tile(const StepArgs &A, const TensorDev &T, const TensorScal &S, uint32_t tile, Meta &meta,
                              const Pol &pol) {
    const GScale gsc = grad_scale(A);
    FlatTile<WIDE> F(T, S, tile, meta);
    Acc2 acc;
    const int64_t numel = T.numel;
    for (uint32_t k = 0; k < T.fvpt; k += kFlatAhead) {
        Raw8 g[kFlatAhead];
        float mm[kFlatAhead][8];
        FlatVec Q[kFlatAhead];
#pragma unroll
        for (uint32_t h = 0; h < kFlatAhead; ++h) {
            Q[h] = F.next();
            const int64_t e = Q[h].e;
            if (e < numel) {
                const int valid = (int)min(int64_t(8), numel - e);
                load8_raw(T.g, T.f32, T.wal, e, valid, g[h], pol);
                if (T.momentum) load_f8(T.M + e, T.sal, valid, mm[h]);
            }
        }
#pragma unroll
        for (uint32_t h = 0; h < kFlatAhead; ++h) {
            const int64_t e = Q[h].e;
            if (e < numel) {
                const int valid = (int)min(int64_t(8), numel - e);
                float y[8], sc[8], u[8];
                values8(g[h], T.f32, y);
                if (T.momentum) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) y[c] = fmaf(A.b1, mm[h][c], gsc.c1 * y[c]);
                    store_f8(T.M + e, T.sal, valid, y);
                }
                F.scales(Q[h], valid, A.ce, sc);
#pragma unroll
                for (int c = 0; c < 8; ++c) u[c] = y[c] * sc[c];  // 0 past the end
                acc.add(sumsq8(u));
            }
        }
    }
    return acc;
}

__device__ Acc2 rms_full_tile(const StepArgs &A, const TensorDev &T, uint32_t tile, const Pol &pol) {
    const GScale gsc = grad_scale(A);
    const int64_t numel = T.numel;
    Acc2 acc;
    int64_t e0 = 8 * (int64_t(tile) * kThreads * T.fvpt + threadIdx.x);
    for (uint32_t k = 0; k < T.fvpt && e0 < numel; k += kFlatAhead) {
        Raw8 raw[kFlatAhead];
        float v[kFlatAhead][8], mm[kFlatAhead][8];
#pragma unroll
        for (uint32_t h = 0; h < kFlatAhead; ++h) {
            const int64_t e = e0 + h * 8 * kThreads;
            if (k + h < T.fvpt && e < numel) {
                const int valid = (int)min(int64_t(8), numel - e);
                load8_raw(T.g, T.f32, T.wal, e, valid, raw[h], pol);
                load_f8(T.v + e, T.sal, valid, v[h]);
                if (T.momentum) load_f8(T.M + e, T.sal, valid, mm[h]);
            }
        }
#pragma unroll
        for (uint32_t h = 0; h < kFlatAhead; ++h) {
            const int64_t e = e0 + h * 8 * kThreads;
            if (k + h < T.fvpt && e < numel) {
                const int valid = (int)min(int64_t(8), numel - e);
                float g[8], u[8];
                values8(raw[h], T.f32, g);
#pragma unroll
                for (int c = 0; c < 8; ++c) v[h][c] = fmaf(A.b2, v[h][c], gsc.c2 * (g[c] * g[c]));
                store_f8(T.v + e, T.sal, valid, v[h]);
                if (T.momentum) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) g[c] = fmaf(A.b1, mm[h][c], gsc.c1 * g[c]);
                    store_f8(T.M + e, T.sal, valid, g);
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) u[c] = c < valid ? g[c] * fminf(__frsqrt_rn(v[h][c]), A.ce) : 0.f;
                acc.add(sumsq8(u));
            }
        }
        e0 += kFlatAhead * 8 * kThreads;
    }
    return acc;
}

// Stores a phase-B tile's sum of (U / coef)^2; the last tile of the tensor forms sum(U^2), RMS and
// the clip factor (fixed summation order).
__device__ void finish_B(const StepArgs &A, const TensorDev &T, uint32_t t, uint32_t local, const Acc2 &acc, Smem &sm) {
    TensorScal &S = A.scal[t];
    const float2 tsum = block_sum2(acc, sm.red2);
    if (threadIdx.x == 0) {
        T.u2[local] = tsum;
        sm.last = (atom_add_acq_rel(&S.cntB, 1u) == T.nbc - 1);
    }
    __syncthreads();
    if (!sm.last) return;
    double s = 0.0;
    for (uint32_t k = threadIdx.x; k < T.nbc; k += kThreads) {
        const float2 p = __ldcg(T.u2 + k);
        s += pair_value(p.x, p.y);
    }
    s = block_sum_d(s, sm.redd);
    if (threadIdx.x == 0) set_clip(A, T, S, s);
}

__device__ void phase_B_full(const StepArgs &A, const TensorDev &T, uint32_t t, uint32_t local, Smem &sm, const Pol &pol) {
    const Acc2 acc = rms_full_tile(A, T, local, pol);
    finish_B(A, T, t, local, acc, sm);
}

__device__ void phase_B_strip(const StepArgs &A, const TensorDev &T, uint32_t t, uint32_t local, Smem &sm, Meta &meta, const Pol &pol) {
    (void)fill_meta(T, A.scal[t], local, A.ce, meta);
    finish_B(A, T, t, local,
             T.momentum ? rms_fact_tile<true>(A, T, local, meta, pol) : rms_fact_tile<false>(A, T, local, meta, pol), sm);
}

__device__ void phase_B_flat(const StepArgs &A, const TensorDev &T, uint32_t t, uint32_t local, Smem &sm, Meta &meta, const Pol &pol) {
    finish_B(A, T, t, local,
             T.m > kFlatCols ? rms_flat_tile<true>(A, T, A.scal[t], local, meta, pol)
                             : rms_flat_tile<false>(A, T, A.scal[t], local, meta, pol), sm);
}

__device__ void phase_B_fact(const StepArgs &A, const TensorDev &T, uint32_t t, uint32_t local, Smem &sm, Meta &meta, const Pol &pol) {
    if (T.vec)
        phase_B_strip(A, T, t, local, sm, meta, pol);
    else
        phase_B_flat(A, T, t, local, sm, meta, pol);
}

// ---------------------------------------------------------------------------
// Phase C: decoupled decay, clipped update, dithered bf16 write-back.
// ---------------------------------------------------------------------------
// The dithered bf16 values of eight elements whose first has index e0 (a multiple of 8 with the
// tensor's base).
__device__ __forceinline__ void round8(const float (&x)[8], const Dith &d, uint64_t e0, uint4 &out) {
    uint32_t r[8], o[4];
    dither8(e0, d, r);
    // a NaN anywhere makes the sum NaN (so does Inf - Inf): only then test per element
    const float any = ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
    if (any == any) {
#pragma unroll
        for (int q = 0; q < 4; ++q)  // top halves of (bits + draw) of the two elements
            o[q] = __byte_perm(__float_as_uint(x[2 * q]) + r[2 * q], __float_as_uint(x[2 * q + 1]) + r[2 * q + 1],
                               0x7632);
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q] = sr_bf16(x[2 * q], r[2 * q]) | (sr_bf16(x[2 * q + 1], r[2 * q + 1]) << 16);
    }
    out = make_uint4(o[0], o[1], o[2], o[3]);
}

// x of eight elements -> dithered bf16, one 16-byte store at w + e0.
__device__ __forceinline__ void write8(uint16_t *__restrict__ w, const Dith &d, int64_t e0, const float (&x)[8],
                                       const Pol &pol) {
    uint4 o;
    round8(x, d, (uint64_t)e0, o);
    st16_hint(w + e0, o, pol.drop);
}

// Write-back of elements e0 .. e0 + valid - 1 at any alignment: the dithered bf16 rounding, or for a
// tensor kept in fp32 the fp32 value x itself.
__device__ __forceinline__ void store8_elem(const TensorDev &T, const Dith &d, int64_t e0, int valid, const float (&x)[8],
                                            const Pol &pol) {
    if (T.f32) {
        store_f8(reinterpret_cast<float *>(T.w) + e0, T.wal, valid, x);
        return;
    }
    uint32_t r[8];
    dither8_any((uint64_t)e0, d, r);
    uint32_t h[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) h[c] = sr_bf16(x[c], r[c]);
    if (T.wal && valid == 8) {
        st16_hint(T.w + e0, make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16)),
                  pol.drop);
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < valid) T.w[e0 + c] = (uint16_t)h[c];
    }
}

// FAST: no element of the tile reaches the clamp (fill_meta), so the update is
// (-lr*kappa*coef * a_i) * b_j * y, one multiply and one fma per element.
template <bool MOM, bool FAST>
__device__ void apply_fact_tile(const StepArgs &A, const TensorDev &T, const TensorScal &S, uint32_t tile,
                                const Meta &meta, const Pol &pol) {
    const FactTile F(T, tile);
    if (!F.act) return;
    const uint16_t *__restrict__ g_ = T.g;
    const float *__restrict__ M_ = T.M;
    uint16_t *__restrict__ w_ = T.w;
    const int64_t n = T.n, m = T.m, row0 = F.row0, RG = F.RG, col0 = F.col0;
    const int vpt = (int)(T.tile_rows / F.RG);
    const Dith d = dith_of(A, T);
    const float coefC = __ldcg(&S.coefC);
    const float wdf = T.decay ? A.wdf : 1.0f;
    const float ce = A.ce;
    const float *rows = meta.rows + F.rg;
    float b[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) b[c] = meta.cols[F.lane * 8 + c];
    {
        constexpr int KCH = 4;  // row-vectors (with their weights) requested together
#pragma unroll 1
        for (int k0 = 0; k0 < vpt; k0 += KCH) {
            uint4 wraw[KCH], graw[MOM ? 1 : KCH];
            float4 mraw[MOM ? KCH : 1][2];
#pragma unroll
            for (int q = 0; q < KCH; ++q) {
                const int64_t i = row0 + (k0 + q) * RG;
                const int64_t e0 = (i < n ? i : 0) * m + col0;
                if (i < n) {
                    if (MOM) {
                        mraw[MOM ? q : 0][0] = __ldcg(reinterpret_cast<const float4 *>(M_ + e0));
                        mraw[MOM ? q : 0][1] = __ldcg(reinterpret_cast<const float4 *>(M_ + e0 + 4));
                    } else {
                        graw[MOM ? 0 : q] = ld16_hint(g_ + e0, pol.drop);
                    }
                    wraw[q] = ld16_hint(w_ + e0, pol.drop);
                }
            }
#pragma unroll
            for (int q = 0; q < KCH; ++q) {
                const int64_t i = row0 + (k0 + q) * RG;
                if (i < n) {
                    float y[8], w[8], x[8];
                    if (MOM) {
                        const float4 m0 = mraw[MOM ? q : 0][0], m1 = mraw[MOM ? q : 0][1];
                        y[0] = m0.x; y[1] = m0.y; y[2] = m0.z; y[3] = m0.w;
                        y[4] = m1.x; y[5] = m1.y; y[6] = m1.z; y[7] = m1.w;
                    } else {
                        unpack_bf8(graw[MOM ? 0 : q], y);
                    }
                    unpack_bf8(wraw[q], w);
                    const float a = rows[(k0 + q) * RG];
                    if constexpr (FAST) {
                        const float ca = -coefC * a;
                        const float2 ca2 = make_float2(ca, ca), wdf2 = make_float2(wdf, wdf);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float2 xx = __ffma2_rn(__fmul2_rn(ca2, make_float2(b[2 * q], b[2 * q + 1])),
                                                         make_float2(y[2 * q], y[2 * q + 1]),
                                                         __fmul2_rn(make_float2(w[2 * q], w[2 * q + 1]), wdf2));
                            x[2 * q] = xx.x;
                            x[2 * q + 1] = xx.y;
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 8; ++c) x[c] = fmaf(-coefC, y[c] * fminf(a * b[c], ce), w[c] * wdf);
                    }
                    write8(w_, d, i * m + col0, x, pol);
                }
            }
        }
    }
}

template <bool WIDE>
__device__ void apply_flat_any(const StepArgs &A, const TensorDev &T, const TensorScal &S, uint32_t tile, Meta &meta,
                               const Pol &pol) {
    FlatTile<WIDE> F(T, S, tile, meta);
    const float coefC = __ldcg(&S.coefC);
    const float wdf = T.decay ? A.wdf : 1.0f;
    const Dith d = dith_of(A, T);
    const int64_t numel = T.numel;
    for (uint32_t k = 0; k < T.fvpt; k += kFlatAhead) {
        Raw8 g[kFlatAhead], w[kFlatAhead];
        float mm[kFlatAhead][8];
        FlatVec Q[kFlatAhead];
#pragma unroll
        for (uint32_t h = 0; h < kFlatAhead; ++h) {
            Q[h] = F.next();
            const int64_t e = Q[h].e;
            if (e < numel) {
                const int valid = (int)min(int64_t(8), numel - e);
                if (T.momentum)
                    load_f8(T.M + e, T.sal, valid, mm[h]);
                else
                    load8_raw(T.g, T.f32, T.wal, e, valid, g[h], pol);
                load8_raw(T.w, T.f32, T.wal, e, valid, w[h], pol);
            }
        }
#pragma unroll
        for (uint32_t h = 0; h < kFlatAhead; ++h) {
            const int64_t e = Q[h].e;
            if (e < numel) {
                const int valid = (int)min(int64_t(8), numel - e);
                float y[8], v[8], sc[8], x[8];
                if (T.momentum) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) y[c] = mm[h][c];
                } else {
                    values8(g[h], T.f32, y);
                }
                values8(w[h], T.f32, v);
                F.scales(Q[h], valid, A.ce, sc);
#pragma unroll
                for (int c = 0; c < 8; ++c) x[c] = fmaf(-coefC, y[c] * sc[c], v[c] * wdf);
                store8_elem(T, d, e, valid, x, pol);
            }
        }
    }
}

__device__ void apply_full_tile(const StepArgs &A, const TensorDev &T, const TensorScal &S, uint32_t tile,
                                const Pol &pol) {
    const float coefC = __ldcg(&S.coefC);
    const float wdf = T.decay ? A.wdf : 1.0f;
    const Dith d = dith_of(A, T);
    const int64_t numel = T.numel;
    int64_t e0 = 8 * (int64_t(tile) * kThreads * T.fvpt + threadIdx.x);
    for (uint32_t k = 0; k < T.fvpt && e0 < numel; k += kFlatAhead) {
        Raw8 g[kFlatAhead], w[kFlatAhead];
        float mm[kFlatAhead][8], v[kFlatAhead][8];
#pragma unroll
        for (uint32_t h = 0; h < kFlatAhead; ++h) {
            const int64_t e = e0 + h * 8 * kThreads;
            if (k + h < T.fvpt && e < numel) {
                const int valid = (int)min(int64_t(8), numel - e);
                if (T.momentum)
                    load_f8(T.M + e, T.sal, valid, mm[h]);
                else
                    load8_raw(T.g, T.f32, T.wal, e, valid, g[h], pol);
                load_f8(T.v + e, T.sal, valid, v[h]);
                load8_raw(T.w, T.f32, T.wal, e, valid, w[h], pol);
            }
        }
#pragma unroll
        for (uint32_t h = 0; h < kFlatAhead; ++h) {
            const int64_t e = e0 + h * 8 * kThreads;
            if (k + h < T.fvpt && e < numel) {
                const int valid = (int)min(int64_t(8), numel - e);
                float y[8], wv[8], x[8];
                if (T.momentum) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) y[c] = mm[h][c];
                } else {
                    values8(g[h], T.f32, y);
                }
                values8(w[h], T.f32, wv);
#pragma unroll
                for (int c = 0; c < 8; ++c) x[c] = fmaf(-coefC, y[c] * fminf(__frsqrt_rn(v[h][c]), A.ce), wv[c] * wdf);
                store8_elem(T, d, e, valid, x, pol);
            }
        }
        e0 += kFlatAhead * 8 * kThreads;
    }
}

// Phase C of a tensor whose clip factor the finalize proved to be 1 (kSumInC): stores the tile's
// sum of (U / coef)^2 (entry 2 tile + half of u2; a whole tile clears the other), counts its rows,
// and the tile that completes the tensor forms sum(U^2) and RMS(U) as phase B does.
struct SumSmem {
    float2 red2[kThreads / 32];
    double redd[kThreads / 32];
    int last;
};

__device__ void publish_sum(const StepArgs &A, const TensorDev &T, TensorScal &S, uint32_t item, uint32_t rows,
                            const Acc2 &acc, SumSmem &sm) {
    const float2 tsum = block_sum2(acc, sm.red2);
    if (threadIdx.x == 0) {
        float2 *e = T.u2 + 2 * size_t(item & kTileMask) + ((item & kSecondHalf) ? 1 : 0);
        e[0] = tsum;
        // the entry of a half that does not exist: of a whole tile, or past the matrix's end
        const int64_t r1 = int64_t(item & kTileMask) * T.at_rows + T.at_rows / 2;
        if (!(item & kHalfTile) || (!(item & kSecondHalf) && r1 >= T.n)) e[1] = make_float2(0.f, 0.f);
        sm.last = (int64_t)atom_add_acq_rel(&S.cntB, rows) + rows == T.n;
    }
    __syncthreads();
    if (!sm.last) return;
    double s = 0.0;
    for (uint32_t k = threadIdx.x; k < 2 * T.atiles; k += kThreads) {
        const float2 p = __ldcg(T.u2 + k);
        s += pair_value(p.x, p.y);
    }
    s = block_sum_d(s, sm.redd);
    if (threadIdx.x == 0) set_clip(A, T, S, s);
}

// ---------------------------------------------------------------------------
// Row path, phase C (k_apply_rows): the row tiles of k_rowsq. A chunk is CA
// whole rows of W and the same rows of G, one bulk copy each into a ring slot
// (W in the first half, G in the second); the column scales b_j of a thread's
// 8*NV columns stay in registers and the tile's row scales a_i in shared memory.
// Per element the arithmetic, the dither index and the rounding are those of
// apply_fact_tile, so the result is the same bit for bit.
// ---------------------------------------------------------------------------
struct ApplyRowSmem {
    uint4 buf[kRowStages][kRowChunkBytes / 16];  // [W rows | G rows] per slot
    uint64_t full[kRowStages];
    float a[kRowChunks * 32];                    // row scales a_i of the tile (at_rows <= 1024)
    float red[2 * kThreads / 32];
    SumSmem sum;
};

// Chunk c of the phase-C tile (or half tile) whose first row is r0. A half tile is 16 of
// the phase-A chunks' rows, i.e. whole phase-C chunks, so only the matrix's end cuts one.
__device__ __forceinline__ void apply_row_issue(const TensorDev &T, int64_t r0, uint32_t c, uint32_t ca,
                                                ApplyRowSmem &sm, uint64_t pol) {
    const int64_t i0 = r0 + int64_t(c) * ca;
    const uint32_t rows = (uint32_t)min((int64_t)ca, T.n - i0);
    const uint32_t bytes = rows * (uint32_t)T.m * 2u;
    const int st = c % kRowStages;
    mbar_expect_tx(&sm.full[st], 2u * bytes);
    bulk_g2s(sm.buf[st], T.w + i0 * T.m, bytes, &sm.full[st], pol);
    bulk_g2s(sm.buf[st] + kRowChunkBytes / 32, T.g + i0 * T.m, bytes, &sm.full[st], pol);
}

// CA = 1024 / V rows per chunk (16 KB of W, 16 KB of G), KA = CA / RPP rows per thread.
template <int TPB, int V, bool FAST>
__device__ bool apply_rows_body(const StepArgs &A, const TensorDev &T, int64_t r0,
                                const float (&b)[RowLayout<TPB, V>::NV][8], float coefC, ApplyRowSmem &sm,
                                uint32_t nch, uint64_t pol, Acc2 &acc) {
    using L = RowLayout<TPB, V>;
    constexpr int NV = L::NV, RPP = L::RPP;
    constexpr int CA = 1024 / V, KA = CA / RPP;
    const L lay;
    const int tid = threadIdx.x;
    const int64_t m = 8 * V;
    uint16_t *__restrict__ w_ = T.w;
    const Dith d = dith_of(A, T);
    const float wdf = T.decay ? A.wdf : 1.0f;
    const float ce = A.ce;
    const float2 wdf2 = make_float2(wdf, wdf);
    const Pol sp;
    for (uint32_t c = 0; c < nch; ++c) {
        const int st = c % kRowStages;
        const int64_t i0 = r0 + int64_t(c) * CA;
        const int rows = (int)min((int64_t)CA, T.n - i0);
        const bool ok = mbar_wait(&sm.full[st], (c / kRowStages) & 1u);
        const uint4 *bw = sm.buf[st];
        const uint4 *bg = sm.buf[st] + kRowChunkBytes / 32;
#pragma unroll
        for (int k = 0; k < KA; ++k) {
            const int r = lay.rp + RPP * k;
            if (r < rows) {
                const float a = sm.a[c * CA + r];
                const float cr = -coefC * a;
                const float2 cr2 = make_float2(cr, cr);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    float y[8], w[8], x[8];
                    unpack_bf8(bg[r * V + v * TPB + lay.vi], y);
                    unpack_bf8(bw[r * V + v * TPB + lay.vi], w);
                    if constexpr (FAST) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float2 xx =
                                __ffma2_rn(__fmul2_rn(cr2, make_float2(b[v][2 * q], b[v][2 * q + 1])),
                                           make_float2(y[2 * q], y[2 * q + 1]),
                                           __fmul2_rn(make_float2(w[2 * q], w[2 * q + 1]), wdf2));
                            x[2 * q] = xx.x;
                            x[2 * q + 1] = xx.y;
                        }
                    } else {
                        float u[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            u[q] = y[q] * fminf(a * b[v][q], ce);
                            x[q] = fmaf(-coefC, u[q], w[q] * wdf);
                        }
                        acc.add(sumsq8(u));
                    }
                    write8(w_, d, (i0 + r) * m + 8 * (v * TPB + lay.vi), x, sp);
                }
            }
        }
        // every thread is done with slot st: refill it with chunk c + kRowStages
        if (__syncthreads_or(!ok)) {
            if (tid == 0)  // chunks [0, c + kRowStages) were issued
                drain_copies(A.err, sm.full, kRowStages, c, min(nch, c + kRowStages));
            return false;
        }
        if (tid == 0 && c + kRowStages < nch) {
            fence_proxy_async_smem();
            apply_row_issue(T, r0, c + kRowStages, CA, sm, pol);
        }
    }
    return true;
}

template <int TPB, int V>
__device__ void apply_rows_tile(const StepArgs &A, const TensorDev &T, TensorScal &S, uint32_t item,
                                ApplyRowSmem &sm) {
    using L = RowLayout<TPB, V>;
    constexpr int NV = L::NV;
    constexpr int CA = 1024 / V;
    const L lay;
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    // a whole tile, or one half of it (the step's last tiles run as halves)
    const uint32_t trows = (item & kHalfTile) ? T.at_rows / 2 : T.at_rows;
    const int64_t r0 = int64_t(item & kTileMask) * T.at_rows + ((item & kSecondHalf) ? trows : 0);
    if (r0 >= T.n) return;  // the second half of a matrix's short last tile
    const uint32_t rows_t = (uint32_t)min((int64_t)trows, T.n - r0);
    const uint32_t nch = (rows_t + CA - 1) / CA;
    if (threadIdx.x == 0) {
        for (int st = 0; st < kRowStages; ++st) mbar_init(&sm.full[st], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (uint32_t c = 0; c < nch && c < (uint32_t)kRowStages; ++c) apply_row_issue(T, r0, c, CA, sm, pol);
    // row scales of the tile, column scales of this thread's columns, and the clamp test
    const float rbar_s = __ldcg(&S.rbar_s);
    const int rbar_e = __ldcg(&S.rbar_e);
    float ma = 0.f, mb = 0.f;
    const float *R = T.R + r0;  // (the stores may alias the descriptor)
    for (uint32_t r = threadIdx.x; r < rows_t; r += TPB) {
        const float a = row_scale(__ldcg(R + r), rbar_s, rbar_e);
        sm.a[r] = a;
        ma = fmaxf(ma, nan_to_inf(a));
    }
    float b[NV][8];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const float *p = T.bsc + 8 * (v * TPB + lay.vi);
        const float4 b0 = __ldcg(reinterpret_cast<const float4 *>(p));
        const float4 b1 = __ldcg(reinterpret_cast<const float4 *>(p + 4));
        b[v][0] = b0.x; b[v][1] = b0.y; b[v][2] = b0.z; b[v][3] = b0.w;
        b[v][4] = b1.x; b[v][5] = b1.y; b[v][6] = b1.z; b[v][7] = b1.w;
#pragma unroll
        for (int k = 0; k < 8; ++k) mb = fmaxf(mb, nan_to_inf(b[v][k]));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        ma = fmaxf(ma, __shfl_xor_sync(kAll, ma, o));
        mb = fmaxf(mb, __shfl_xor_sync(kAll, mb, o));
    }
    if ((threadIdx.x & 31) == 0) {
        sm.red[threadIdx.x >> 5] = ma;
        sm.red[TPB / 32 + (threadIdx.x >> 5)] = mb;
    }
    __syncthreads();
    ma = mb = 0.f;
#pragma unroll
    for (int w = 0; w < TPB / 32; ++w) {
        ma = fmaxf(ma, sm.red[w]);
        mb = fmaxf(mb, sm.red[TPB / 32 + w]);
    }
    const float coefC = __ldcg(&S.coefC);
    const bool sum = __ldcg(&S.fallback) == kSumInC;
    Acc2 acc;
    bool done;
    if (!sum && ma * mb <= A.ce)
        done = apply_rows_body<TPB, V, true>(A, T, r0, b, coefC, sm, nch, pol, acc);
    else
        done = apply_rows_body<TPB, V, false>(A, T, r0, b, coefC, sm, nch, pol, acc);
    if (sum && done) publish_sum(A, T, S, item, rows_t, acc, sm.sum);
}

// ---------------------------------------------------------------------------
// Row path with momentum (backbone matrices, and experts under the momentum
// variants). Phase A runs on whole rows as in k_rowsq and, in the same pass,
// applies Algorithm 1's momentum update M <- b1 M + (1 - b1) g to a copy of the
// rows of M made beside those of G, storing the new M. With U_ij = coef M_ij a_i b_j
// and no element at the clamp, sum(U^2) = coef^2 * mean(R) * sum_j Q_j / C_j with
// Q_j = sum_i M_ij^2 / R_i, accumulated here where the momentum-free path
// accumulates P_j. Phase C then reads the new M where it would read G. A chunk
// is CS = kMomGBytes / (2 m) rows: 16 KB of G (or W in phase C) and the same rows
// of M (32 KB) in one slot of a 2-slot ring, one bulk copy each. A row whose R_i
// is 0 or not finite sends the tensor to phase B (its momentum may still be
// nonzero), where M is used as already updated.
// ---------------------------------------------------------------------------
constexpr int kMomStages = 2;
constexpr int kMomSlot16 = 3 * kMomGBytes / 16;  // 16-byte words per slot: 16 KB bf16 | 32 KB fp32

struct MomRowSmem {
    uint4 buf[kMomStages][kMomSlot16];  // [G rows | M rows] per slot
    uint64_t full[kMomStages];
    float part[kThreads / 32][8];
    float inv[32];
};

// Issues the bulk copies of chunk c of the tile whose first row is r0 (rows of x = G in phase A,
// W in phase C, and the same rows of M) into ring slot c % kMomStages.
__device__ __forceinline__ void mom_issue(const TensorDev &T, const uint16_t *x, int64_t r0, uint32_t c,
                                          uint4 (*buf)[kMomSlot16], uint64_t *full, uint64_t pol) {
    const int64_t i0 = r0 + int64_t(c) * T.cr;
    const uint32_t bx = (uint32_t)min(T.n - i0, (int64_t)T.cr) * (uint32_t)T.m * 2u;
    const int st = c % kMomStages;
    mbar_expect_tx(&full[st], 3u * bx);
    bulk_g2s(buf[st], x + i0 * T.m, bx, &full[st], pol);
    bulk_g2s(buf[st] + kMomGBytes / 16, T.M + i0 * T.m, 2u * bx, &full[st], pol);
}

// k_rowsq for momentum tensors on TPB threads, rows of m = 8 V: chunks of CS = 1024 / V
// rows, K = CS / RPP rows per thread per chunk.
template <int TPB, int V>
__device__ void rowsq_mom_tile(const StepArgs &A, const TensorDev &T, TensorScal &S, uint32_t tile, MomRowSmem &sm) {
    using L = RowLayout<TPB, V>;
    constexpr int NV = L::NV, RPP = L::RPP, WPR = L::WPR;
    constexpr int CS = 1024 / V;
    constexpr int K = CS / RPP;
    static_assert(K == 2 || K == 4, "rows per thread per chunk");
    const L lay;
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    const uint32_t nch = (uint32_t)min((int64_t)(T.rt_rows / T.cr), (T.n - int64_t(tile) * T.rt_rows + T.cr - 1) / T.cr);
    if (threadIdx.x == 0) {
        for (int st = 0; st < kMomStages; ++st) mbar_init(&sm.full[st], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (uint32_t c = 0; c < nch && c < (uint32_t)kMomStages; ++c) mom_issue(T, T.g, int64_t(tile) * T.rt_rows, c, sm.buf, sm.full, pol);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const GScale gsc = grad_scale(A);
    const float b1 = A.b1, c1 = gsc.c1, b2 = A.b2, c2 = gsc.c2, inv_m = 1.0f / (float)(8 * V);  // exact
    const float2 b12 = make_float2(b1, b1), c12 = make_float2(c1, c1);
    // per column pair: sums of g^2, the compensated (hi, lo) sum of M^2 / R_i and its open fp32 part
    float2 cs[NV][4], ph[NV][4], pl[NV][4], t[NV][4];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int q = 0; q < 4; ++q) cs[v][q] = ph[v][q] = pl[v][q] = t[v][q] = make_float2(0.f, 0.f);
    double rsum = 0.0;
    float rmin = __int_as_float(0x7F800000);
    bool zero_row = false;

    uint32_t c = 0;
    for (; c < nch; ++c) {
        const int st = c % kMomStages;
        const uint32_t par = (c / kMomStages) & 1u;
        const RowChunk ch = row_chunk(T, tile, c);
        float rp = 0.f;
        if (tid < (int)ch.rows) rp = __ldcg(T.R + ch.i0 + tid);
        const bool ok = mbar_wait(&sm.full[st], par);
        const uint4 *bg = sm.buf[st];
        const float4 *bm = reinterpret_cast<const float4 *>(sm.buf[st] + kMomGBytes / 16);
        // pass 1: row sums and column sums of g^2
        float rs[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int r = lay.rp + RPP * k;
            float2 r2 = make_float2(0.f, 0.f);
            if (r < (int)ch.rows) {
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    float2 g[4];
                    unpack_bf8x2(bg[r * V + v * TPB + lay.vi], g);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        cs[v][q] = __ffma2_rn(g[q], g[q], cs[v][q]);
                        r2 = __ffma2_rn(g[q], g[q], r2);
                    }
                }
            }
            rs[k] = r2.x + r2.y;
        }
        int j;
        const float tot = warp_sum_transposed<K>(rs, j);
        if ((lane & (K == 4 ? 7 : 15)) == 0) sm.part[warp][j] = tot;
        if (__syncthreads_or(!ok)) break;  // every slot before this one has landed
        // refill from warp 1: warp 0 forms the chunk's row scales, which the CTA waits for
        if (tid == 32 && c >= 1 && c - 1 + kMomStages < nch) {
            fence_proxy_async_smem();
            mom_issue(T, T.g, int64_t(tile) * T.rt_rows, c - 1 + kMomStages, sm.buf, sm.full, pol);
        }
        float Rn = 0.f;
        if (tid < (int)ch.rows) {
            const int w0 = (tid % RPP) * WPR, kr = tid / RPP;
            Rn = fmaf(b2, rp, c2 * (tree_sum<WPR>(&sm.part[w0][kr], 8) * inv_m));
            sm.inv[tid] = Rn > 0.f && Rn < __int_as_float(0x7F800000) ? __frcp_rn(Rn) : 0.f;
        }
        __syncthreads();
        if (tid < (int)ch.rows) {  // the row's R and the tile's statistics, off the barrier's path
            T.R[ch.i0 + tid] = Rn;
            rsum += (double)Rn;
            if (Rn > 0.f && Rn < __int_as_float(0x7F800000))
                rmin = fminf(rmin, Rn);
            else
                zero_row = true;  // R_i == 0 or not finite: its momentum may still be nonzero
        }
        // pass 2: M <- b1 M + (1 - b1) g (stored), Q_j += M^2 / R_i
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int r = lay.rp + RPP * k;
            if (r < (int)ch.rows) {
                const float iv = sm.inv[r];
                const float2 iv2 = make_float2(iv, iv);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const int vec = v * TPB + lay.vi;
                    float2 g[4];
                    unpack_bf8x2(bg[r * V + vec], g);
                    const float4 m0 = bm[2 * (r * V + vec)], m1 = bm[2 * (r * V + vec) + 1];
                    const float2 mo[4] = {make_float2(m0.x, m0.y), make_float2(m0.z, m0.w), make_float2(m1.x, m1.y),
                                          make_float2(m1.z, m1.w)};
                    float2 mn[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        mn[q] = __ffma2_rn(b12, mo[q], __fmul2_rn(c12, g[q]));
                        t[v][q] = __ffma2_rn(__fmul2_rn(mn[q], mn[q]), iv2, t[v][q]);
                    }
                    float4 *dst = reinterpret_cast<float4 *>(T.M + (ch.i0 + r) * T.m + 8 * vec);
                    dst[0] = make_float4(mn[0].x, mn[0].y, mn[1].x, mn[1].y);
                    dst[1] = make_float4(mn[2].x, mn[2].y, mn[3].x, mn[3].y);
                }
            }
        }
        if ((c & 3u) == 3u || c + 1 == nch) {
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float2 s2, e2;
                    two_sum2(ph[v][q], t[v][q], s2, e2);
                    ph[v][q] = s2;
                    pl[v][q] = __fadd2_rn(pl[v][q], e2);
                    t[v][q] = make_float2(0.f, 0.f);
                }
        }
    }
    if (c < nch) {
        // a chunk did not land in time: as in rowsq_tile
        if (tid == 0)
            drain_copies(A.err, sm.full, kMomStages, c, min(nch, c == 0 ? (uint32_t)kMomStages : c + kMomStages - 1));
        return;
    }
    const int64_t base = int64_t(tile) * 8 * V;
    if constexpr (RPP == 1) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int64_t col = 8 * int64_t(v * TPB + lay.vi);
            float4 *pp4 = reinterpret_cast<float4 *>(T.pp + base + col);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                pp4[q] = make_float4(cs[v][q].x, pair_f(ph[v][q].x, pl[v][q].x), cs[v][q].y,
                                     pair_f(ph[v][q].y, pl[v][q].y));
        }
    } else {
        // the ring is free (every chunk consumed before the last barrier): stage there
        float *mcs = reinterpret_cast<float *>(sm.buf[0]);    // [TPB][8]
        float2 *mpp = reinterpret_cast<float2 *>(sm.buf[1]);  // [TPB][8] (hi, lo)
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            mcs[tid * 8 + 2 * q] = cs[0][q].x;
            mcs[tid * 8 + 2 * q + 1] = cs[0][q].y;
            mpp[tid * 8 + 2 * q] = make_float2(ph[0][q].x, pl[0][q].x);
            mpp[tid * 8 + 2 * q + 1] = make_float2(ph[0][q].y, pl[0][q].y);
        }
        __syncthreads();
        for (int e = tid; e < 8 * V; e += TPB) {  // column e = 8 vi + q
            const int vi = e >> 3, q = e & 7;
            float cc = 0.f;
            Acc2 pq;
#pragma unroll
            for (int r = 0; r < RPP; ++r) {
                cc += mcs[(r * V + vi) * 8 + q];
                const float2 h = mpp[(r * V + vi) * 8 + q];
                pq.add(h.x);
                pq.lo += h.y;
            }
            T.pp[base + e] = make_float2(cc, pair_f(pq.hi, pq.lo));
        }
    }
    if (zero_row) atomicOr(&S.zflag, 1u);
    if (warp == 0) {  // CS <= 32: the chunk-row positions are lanes of warp 0
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            rsum += __shfl_xor_sync(kAll, rsum, o);
            rmin = fminf(rmin, __shfl_xor_sync(kAll, rmin, o));
        }
        if (lane == 0) {
            T.rsum[tile] = rsum;
            T.rmin[tile] = rmin;
        }
    }
}

struct MomApplySmem {
    uint4 buf[kMomStages][kMomSlot16];  // [W rows | M rows] per slot
    uint64_t full[kMomStages];
    float a[kRowChunks * 32];           // row scales a_i of the tile (at_rows <= 1024)
    float red[2 * kThreads / 32];
    SumSmem sum;
};

// Phase C of a momentum row tile: as apply_rows_body with y = the new M (Algorithm 1,
// backbone branch: U = coef M / D).
template <int TPB, int V, bool FAST>
__device__ bool apply_rows_mom_body(const StepArgs &A, const TensorDev &T, int64_t r0,
                                    const float (&b)[RowLayout<TPB, V>::NV][8], float coefC, MomApplySmem &sm,
                                    uint32_t nch, uint64_t pol, Acc2 &acc) {
    using L = RowLayout<TPB, V>;
    constexpr int NV = L::NV, RPP = L::RPP;
    constexpr int CA = 1024 / V, KA = CA / RPP;
    const L lay;
    const int tid = threadIdx.x;
    const int64_t m = 8 * V;
    uint16_t *__restrict__ w_ = T.w;
    const Dith d = dith_of(A, T);
    const float wdf = T.decay ? A.wdf : 1.0f;
    const float ce = A.ce;
    const float2 wdf2 = make_float2(wdf, wdf);
    const Pol sp;
    for (uint32_t c = 0; c < nch; ++c) {
        const int st = c % kMomStages;
        const int64_t i0 = r0 + int64_t(c) * CA;
        const int rows = (int)min((int64_t)CA, T.n - i0);
        const bool ok = mbar_wait(&sm.full[st], (c / kMomStages) & 1u);
        const uint4 *bw = sm.buf[st];
        const float4 *bm = reinterpret_cast<const float4 *>(sm.buf[st] + kMomGBytes / 16);
#pragma unroll
        for (int k = 0; k < KA; ++k) {
            const int r = lay.rp + RPP * k;
            if (r < rows) {
                const float a = sm.a[c * CA + r];
                const float cr = -coefC * a;
                const float2 cr2 = make_float2(cr, cr);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const int vec = v * TPB + lay.vi;
                    float w[8], x[8];
                    unpack_bf8(bw[r * V + vec], w);
                    const float4 m0 = bm[2 * (r * V + vec)], m1 = bm[2 * (r * V + vec) + 1];
                    const float y[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                    if constexpr (FAST) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float2 xx =
                                __ffma2_rn(__fmul2_rn(cr2, make_float2(b[v][2 * q], b[v][2 * q + 1])),
                                           make_float2(y[2 * q], y[2 * q + 1]),
                                           __fmul2_rn(make_float2(w[2 * q], w[2 * q + 1]), wdf2));
                            x[2 * q] = xx.x;
                            x[2 * q + 1] = xx.y;
                        }
                    } else {
                        float u[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            u[q] = y[q] * fminf(a * b[v][q], ce);
                            x[q] = fmaf(-coefC, u[q], w[q] * wdf);
                        }
                        acc.add(sumsq8(u));
                    }
                    write8(w_, d, (i0 + r) * m + 8 * vec, x, sp);
                }
            }
        }
        // every thread is done with slot st: refill it with chunk c + kMomStages
        if (__syncthreads_or(!ok)) {
            if (tid == 0) drain_copies(A.err, sm.full, kMomStages, c, min(nch, c + kMomStages));
            return false;
        }
        if (tid == 0 && c + kMomStages < nch) {
            fence_proxy_async_smem();
            mom_issue(T, T.w, r0, c + kMomStages, sm.buf, sm.full, pol);
        }
    }
    return true;
}

template <int TPB, int V>
__device__ void apply_rows_mom_tile(const StepArgs &A, const TensorDev &T, TensorScal &S, uint32_t item,
                                    MomApplySmem &sm) {
    using L = RowLayout<TPB, V>;
    constexpr int NV = L::NV;
    const L lay;
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    const uint32_t trows = (item & kHalfTile) ? T.at_rows / 2 : T.at_rows;
    const int64_t r0 = int64_t(item & kTileMask) * T.at_rows + ((item & kSecondHalf) ? trows : 0);
    if (r0 >= T.n) return;  // the second half of a matrix's short last tile
    const uint32_t rows_t = (uint32_t)min((int64_t)trows, T.n - r0);
    const uint32_t nch = (rows_t + T.cr - 1) / T.cr;
    if (threadIdx.x == 0) {
        for (int st = 0; st < kMomStages; ++st) mbar_init(&sm.full[st], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (uint32_t c = 0; c < nch && c < (uint32_t)kMomStages; ++c) mom_issue(T, T.w, r0, c, sm.buf, sm.full, pol);
    const float rbar_s = __ldcg(&S.rbar_s);
    const int rbar_e = __ldcg(&S.rbar_e);
    float ma = 0.f, mb = 0.f;
    const float *R = T.R + r0;  // (the stores may alias the descriptor)
    for (uint32_t r = threadIdx.x; r < rows_t; r += TPB) {
        const float a = row_scale(__ldcg(R + r), rbar_s, rbar_e);
        sm.a[r] = a;
        ma = fmaxf(ma, nan_to_inf(a));
    }
    float b[NV][8];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const float *p = T.bsc + 8 * (v * TPB + lay.vi);
        const float4 b0 = __ldcg(reinterpret_cast<const float4 *>(p));
        const float4 b1 = __ldcg(reinterpret_cast<const float4 *>(p + 4));
        b[v][0] = b0.x; b[v][1] = b0.y; b[v][2] = b0.z; b[v][3] = b0.w;
        b[v][4] = b1.x; b[v][5] = b1.y; b[v][6] = b1.z; b[v][7] = b1.w;
#pragma unroll
        for (int k = 0; k < 8; ++k) mb = fmaxf(mb, nan_to_inf(b[v][k]));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        ma = fmaxf(ma, __shfl_xor_sync(kAll, ma, o));
        mb = fmaxf(mb, __shfl_xor_sync(kAll, mb, o));
    }
    if ((threadIdx.x & 31) == 0) {
        sm.red[threadIdx.x >> 5] = ma;
        sm.red[TPB / 32 + (threadIdx.x >> 5)] = mb;
    }
    __syncthreads();
    ma = mb = 0.f;
#pragma unroll
    for (int w = 0; w < TPB / 32; ++w) {
        ma = fmaxf(ma, sm.red[w]);
        mb = fmaxf(mb, sm.red[TPB / 32 + w]);
    }
    const float coefC = __ldcg(&S.coefC);
    const bool sum = __ldcg(&S.fallback) == kSumInC;
    Acc2 acc;
    bool done;
    if (!sum && ma * mb <= A.ce)
        done = apply_rows_mom_body<TPB, V, true>(A, T, r0, b, coefC, sm, nch, pol, acc);
    else
        done = apply_rows_mom_body<TPB, V, false>(A, T, r0, b, coefC, sm, nch, pol, acc);
    if (sum && done) publish_sum(A, T, S, item, rows_t, acc, sm.sum);
}

// ---------------------------------------------------------------------------
// Row path for any other width m = 8 V in [128, 8192] (phase A; phase C is
// apply_flat_tile). The same algorithm as rowsq_tile / rowsq_mom_tile on a layout
// formed at run time: a row belongs to wpr = ceil(V / (32 NV)) warps, of which a
// thread owns vectors vi, vi + 32 wpr, ... (columns stay in its registers), and
// rpp = 8 / wpr rows go side by side; warps past rpp * wpr, and lanes past the row's
// end, only keep the barriers (at worst 3 of 8 warps, m = 1032 to 1280). A chunk is
// K rpp whole rows (at most 32 KB of G, or 48 KB of G and M), in as many ring slots
// as 96 KB holds. What bounds it: the chain of two passes and two barriers per chunk, as
// for the fixed widths (ncu: barrier stalls first), with fewer of the eight warps working.
// 512 MiB of G: m = 1536 117 us (4.6 TB/s, after a write-back of the last launch's dirty
// L2), 768 120, 1408 124, 3072 127, against 105 to 110 us at the fixed widths; with momentum
// 210 to 219 us (6.2 TB/s of G and M) at every width. Branches on the lanes past a row's end made
// it 536 us where reading zeros instead takes 405 (930M parameters in 3072 x 1536 experts).
// Widths above 4096 have CTAs of W = 16 warps, one per SM, and a ring of twice the size:
// 512 MiB of G at m = 5120 147 us, 7168 129, 8192 124; a step of 1.16B parameters of 4864
// and 7128 columns 2314 us on strip tiles and 1653 so.
// ---------------------------------------------------------------------------
constexpr int kGenStages = 8;
constexpr int kGenRingBytes = 3 * 32768;  // of the 8-warp tile

// W warps: 8, or 16 for the widths above 4096.
template <int W>
struct GenSmem {
    uint4 ring[W / 8 * kGenRingBytes / 16];
    uint4 zero[2];      // what the lanes past a row's end (and rows past the matrix) read
    uint64_t full[kGenStages];
    float part[W][8];   // per-warp row partial sums of the chunk
    float inv[64];      // 1 / R_i of the chunk's rows (0: no contribution)
    double rsum[2];
    float rmin[2];
    uint32_t first;     // 1: the layout starts with the third warp
};
static_assert(offsetof(GenSmem<8>, zero) == kGenRingBytes, "zero follows the ring");
static_assert(offsetof(GenSmem<16>, zero) == 2 * kGenRingBytes, "zero follows the ring");

template <int W, int NV, bool MOM>
__device__ void rowsq_gen_tile(const StepArgs &A, const TensorDev &T, TensorScal &S, uint32_t tile, GenSmem<W> &sm) {
    constexpr uint32_t kGenZero = W / 8 * kGenRingBytes / 16;  // index of `zero` from `ring`
    constexpr int TPB = 32 * W;
    constexpr int K = gen_rows_per_thread(NV, MOM);
    // with one vector per thread and row the chunk stays in registers from pass 1 to pass 2, as in
    // rowsq_tile: its squares, or with momentum g (M is still read from the slot)
    constexpr bool kHold = NV == 1, kEarly = kHold && !MOM;
    const uint32_t V = (uint32_t)T.m / 8u, m = (uint32_t)T.m;
    const uint32_t wpr = (V + 32 * NV - 1) / (32 * NV), rpp = W / wpr, lpr = 32 * wpr;
    const uint32_t cr = T.cr, gbytes = cr * m * 2u, slot = MOM ? 3u * gbytes : gbytes;
    const uint32_t stages = min((uint32_t)kGenStages, 16u * kGenZero / slot);
    const int64_t row0 = int64_t(tile) * T.rt_rows, n = T.n;
    const uint32_t rows_t = (uint32_t)min((int64_t)T.rt_rows, n - row0);
    const uint32_t nch = (rows_t + cr - 1) / cr;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float *__restrict__ Mt = MOM ? T.M + row0 * T.m : nullptr;
    float *__restrict__ Rt = T.R + row0;
    char *ring = reinterpret_cast<char *>(sm.ring);
    // (the issuing thread reads its addresses from the descriptor each time: they would cost
    // every thread registers)
    auto issue = [&](uint32_t c, uint32_t st) {
        const uint32_t rows = min(cr, rows_t - c * cr), bx = rows * m * 2u;
        const int64_t e0 = (int64_t(tile) * T.rt_rows + c * cr) * T.m;
        const uint64_t pol = read_policy(!MOM && T.keep);
        mbar_expect_tx(&sm.full[st], MOM ? 3u * bx : bx);
        bulk_g2s(ring + st * slot, T.g + e0, bx, &sm.full[st], pol);
        if (MOM) bulk_g2s(ring + st * slot + gbytes, T.M + e0, 2u * bx, &sm.full[st], pol);
    };
    if (tid == 0) {
        for (uint32_t st = 0; st < stages; ++st) mbar_init(&sm.full[st], 1);
        fence_mbar_init();
        // the warps left idle sit on the same two of the SM's four schedulers in every CTA: the CTAs in
        // the SM's second half of warp slots start with the third warp (a hint; any value is right).
        // 512 MiB of G, before: 126 us at m = 1536, 129 at 768, 133 at 1408
        uint32_t slot;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
        sm.first = W == 8 ? (slot >> 3) & 1u : 0u;
    }
    if (tid < 8) reinterpret_cast<uint32_t *>(sm.zero)[tid] = 0u;
    __syncthreads();
    if (tid == 0)
        for (uint32_t c = 0; c < nch && c < stages; ++c) issue(c, c);

    const uint32_t lw = (warp + 2 * sm.first) & (W - 1u);  // the warp's place in the layout
    const uint32_t rp = lw / wpr, vi = (lw - rp * wpr) * 32u + lane;
    const bool on = rp < rpp;  // the warp has rows (the same for its lanes)
    bool act[NV];              // the thread has vector vi + v lpr
    uint32_t step[NV];         // vectors from one of its rows to the next
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        act[v] = on && vi + v * lpr < V;
        step[v] = act[v] ? rpp * V : 0u;
    }
    const uint32_t kr = tid / rpp, w0 = (tid - kr * rpp) * wpr;  // threads < cr: chunk row tid is k = kr of row-in-pass tid % rpp
    const GScale gsc = grad_scale(A);
    // c2 / m, without a step into the subnormals that c2 itself does not take (a tiny gamma): c2 over m times kLead, at
    // most 2, and the row's sum times kLead
    constexpr float kLead = W == 16 ? 1.f / 4096.f : NV == 2 ? 1.f / 2048.f : 1.f / 1024.f;
    const float b2 = A.b2, c2m = __fdiv_rn(gsc.c2, (float)m * kLead);
    const float2 b12 = make_float2(A.b1, A.b1), c12 = make_float2(gsc.c1, gsc.c1);
    // per column pair: sums of g^2, the compensated (hi, lo) sum of y^2 / R_i (y = g, or the new
    // M with momentum) and its open fp32 part
    float2 cs[NV][4], ph[NV][4], pl[NV][4], t[NV][4];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int q = 0; q < 4; ++q) cs[v][q] = ph[v][q] = pl[v][q] = t[v][q] = make_float2(0.f, 0.f);
    const float inf = __int_as_float(0x7F800000);
    double rsum = 0.0;  // threads < cr: sum and smallest positive R of this chunk-row position
    float rmin = inf;
    bool zero_row = false;

    uint32_t c = 0, st = 0, par = 0;
    for (; c < nch; ++c) {
        const uint32_t rows = min(cr, rows_t - c * cr);
        float rold = 0.f;
        if (tid < (int)rows) rold = __ldcg(Rt + c * cr + tid);
        const bool ok = mbar_wait(&sm.full[st], par);
        // the thread's first vector of the chunk's G, and of its M (indices from the ring's start);
        // a lane without a vector reads zeros, so that the passes need no branches
        uint32_t ig[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) ig[v] = act[v] ? st * (slot / 16) + rp * V + vi + v * lpr : kGenZero;
        const bool full = rows == cr;  // every chunk but the tile's last needs no row bound checks
        // pass 1: row and column sums of g^2
        float rs[K];
        float2 hold[kHold ? K : 1][4];
        auto pass1 = [&](auto full_c) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                float2 r2 = make_float2(0.f, 0.f);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const bool in = decltype(full_c)::value || rp + rpp * k < rows;
                    float2 g[4];
                    unpack_bf8x2(sm.ring[in ? ig[v] + k * step[v] : kGenZero], g);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 g2 = __fmul2_rn(g[q], g[q]);  // exact
                        cs[v][q] = __fadd2_rn(cs[v][q], g2);
                        r2 = __fadd2_rn(r2, g2);
                        if constexpr (kHold) hold[k][q] = MOM ? g[q] : g2;
                    }
                }
                rs[k] = r2.x + r2.y;
            }
        };
        if (on) {
            if (full)
                pass1(std::true_type{});
            else
                pass1(std::false_type{});
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) rs[k] = 0.f;
        }
        int j;
        const float tot = warp_sum_transposed<K>(rs, j);
        if ((lane & (K == 8 ? 3 : K == 4 ? 7 : 15)) == 0) sm.part[lw][j] = tot;
        if (__syncthreads_or(!ok)) break;  // every slot before this one has landed
        // the slot of chunk c (when its values are held), or else of chunk c - 1, is free: refill it
        // (from the last warp: the first ones form the chunk's row scales, which the CTA waits for)
        if (tid == TPB - 32 && (kEarly || c >= 1) && c - (kEarly ? 0 : 1) + stages < nch) {
            fence_proxy_async_smem();
            issue(c - (kEarly ? 0 : 1) + stages, kEarly ? st : st == 0 ? stages - 1 : st - 1);
        }
        float Rn = 0.f, sum = 0.f;
        if (tid < (int)rows) {
            float p[W];
#pragma unroll
            for (int w = 0; w < W; ++w) p[w] = w < (int)wpr ? sm.part[w0 + w][kr] : 0.f;
#pragma unroll
            for (int h = W / 2; h; h >>= 1)
#pragma unroll
                for (int w = 0; w < W / 2; ++w)
                    if (w < h) p[w] += p[w + h];
            sum = p[0];
            Rn = fmaf(b2, rold, c2m * (sum * kLead));  // c2 / m, rounded once
            sm.inv[tid] = Rn > 0.f && Rn < inf ? __frcp_rn(Rn) : 0.f;
        }
        __syncthreads();
        if (tid < (int)rows) {  // the row's R and the tile's statistics, off the barrier's path
            Rt[c * cr + tid] = Rn;
            rsum += (double)Rn;
            if (Rn > 0.f && Rn < inf)
                rmin = fminf(rmin, Rn);
            else if (MOM || !(Rn == 0.f && sum == 0.f))
                zero_row = true;  // content (or, with momentum, perhaps an old M) in a row with R_i == 0, or a non-finite R_i
        }
        // pass 2: y^2 / R_i, summed in fp32 over four chunks per column, then folded into (hi, lo);
        // with momentum M <- b1 M + (1 - b1) g, stored here
        auto pass2 = [&](auto full_c) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const uint32_t r = rp + rpp * k;
                const bool in = decltype(full_c)::value || r < rows;
                const float iv = in ? sm.inv[r] : 0.f;
                const float2 iv2 = make_float2(iv, iv);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    float2 y[4];
                    if constexpr (kHold) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) y[q] = hold[k][q];
                    } else {
                        unpack_bf8x2(sm.ring[in ? ig[v] + k * step[v] : kGenZero], y);
                    }
                    if constexpr (MOM) {
                        // M's vector: twice G's distance from the slot's start, past its G
                        const uint32_t im = gbytes / 16 - st * (slot / 16) + 2 * (ig[v] + k * step[v]);
                        const float4 *bm = reinterpret_cast<const float4 *>(sm.ring + (in && act[v] ? im : kGenZero));
                        const float4 m0 = bm[0], m1 = bm[1];
                        y[0] = __ffma2_rn(b12, make_float2(m0.x, m0.y), __fmul2_rn(c12, y[0]));
                        y[1] = __ffma2_rn(b12, make_float2(m0.z, m0.w), __fmul2_rn(c12, y[1]));
                        y[2] = __ffma2_rn(b12, make_float2(m1.x, m1.y), __fmul2_rn(c12, y[2]));
                        y[3] = __ffma2_rn(b12, make_float2(m1.z, m1.w), __fmul2_rn(c12, y[3]));
                        if (act[v] && in) {
                            float4 *dst = reinterpret_cast<float4 *>(Mt + uint64_t(c * cr + r) * m + 8 * (vi + v * lpr));
                            dst[0] = make_float4(y[0].x, y[0].y, y[1].x, y[1].y);
                            dst[1] = make_float4(y[2].x, y[2].y, y[3].x, y[3].y);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        t[v][q] = __ffma2_rn(kEarly ? y[q] : __fmul2_rn(y[q], y[q]), iv2, t[v][q]);
                }
            }
        };
        if (on) {
            if (full)
                pass2(std::true_type{});
            else
                pass2(std::false_type{});
        }
        if ((c & 3u) == 3u || c + 1 == nch) {
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float2 s2, e2;
                    two_sum2(ph[v][q], t[v][q], s2, e2);
                    ph[v][q] = s2;
                    pl[v][q] = __fadd2_rn(pl[v][q], e2);
                    t[v][q] = make_float2(0.f, 0.f);
                }
        }
        if (++st == stages) {
            st = 0;
            par ^= 1u;
        }
    }
    if (c < nch) {
        // a chunk did not land in time: as in rowsq_tile
        if (tid == 0) drain_copies(A.err, sm.full, stages, c, min(nch, kEarly || c == 0 ? c + stages : c + stages - 1));
        return;
    }
    // per-tile partials, as rowsq_tile's
    float2 *pp = T.pp + int64_t(tile) * m;
    if (rpp == 1) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            if (act[v]) {
                float4 *pp4 = reinterpret_cast<float4 *>(pp + 8 * (vi + v * lpr));
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    pp4[q] = make_float4(cs[v][q].x, pair_f(ph[v][q].x, pl[v][q].x), cs[v][q].y,
                                         pair_f(ph[v][q].y, pl[v][q].y));
            }
        }
    } else {  // NV == 1: rpp rows of at most 128 vectors side by side
        float *mcs = reinterpret_cast<float *>(sm.ring);          // [256][8]
        float2 *mpp = reinterpret_cast<float2 *>(sm.ring + 512);  // [256][8] (hi, lo)
        __syncthreads();  // the ring is free: every chunk is consumed
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t o = (lw * 32 + lane) * 8 + 2 * q;
            mcs[o] = cs[0][q].x;
            mcs[o + 1] = cs[0][q].y;
            mpp[o] = make_float2(ph[0][q].x, pl[0][q].x);
            mpp[o + 1] = make_float2(ph[0][q].y, pl[0][q].y);
        }
        __syncthreads();
        for (uint32_t e = tid; e < m; e += TPB) {
            float cc = 0.f;
            Acc2 pq;
            for (uint32_t r = 0; r < rpp; ++r) {
                cc += mcs[r * lpr * 8 + e];
                const float2 h = mpp[r * lpr * 8 + e];
                pq.add(h.x);
                pq.lo += h.y;
            }
            pp[e] = make_float2(cc, pair_f(pq.hi, pq.lo));
        }
    }
    if (zero_row) atomicOr(&S.zflag, 1u);
    if (warp < 2) {  // at most 64 rows per chunk: the chunk-row positions are lanes of warps 0 and 1
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            rsum += __shfl_xor_sync(kAll, rsum, o);
            rmin = fminf(rmin, __shfl_xor_sync(kAll, rmin, o));
        }
        if (lane == 0) {
            sm.rsum[warp] = rsum;
            sm.rmin[warp] = rmin;
        }
    }
    __syncthreads();
    if (tid == 0) {
        T.rsum[tile] = sm.rsum[0] + sm.rsum[1];
        T.rmin[tile] = fminf(sm.rmin[0], sm.rmin[1]);
    }
}

// Phase C of these widths: given the step's scalars it is elementwise, so the tile's rows are one
// run of 16-byte vectors, cut into chunks of 1024 (16 KB of W, and 16 KB of G or 32 KB of M) that
// need not end with a row, and every thread works whatever the width. Row scales and all m column
// scales sit in shared memory; a thread steps its row and column by 256 vectors without dividing.
// Per element the arithmetic is apply_fact_tile's, bit for bit. Bound by HBM: 930M parameters in
// 3072 x 1536 experts 994 us on strip tiles, 826 us (6.75 TB/s) here.
// Above 4096 columns the column scales take 16 to 32 KB, and the ring's chunks are half as long.
struct FlatSmem {
    uint64_t full[4];
    float red[2 * kThreads / 32];
    SumSmem sum;
    uint4 data[kFlatBytes / 16];  // the ring, then b_j [m] and a_i of the tile's rows
};

template <bool MOM, bool WIDE>
struct FlatRing {
    static constexpr uint32_t kChunk = WIDE ? 512 : 1024;                       // vectors
    static constexpr uint32_t kSlot16 = (MOM ? 3 : 2) * kChunk;                 // [W | G] or [W | M]
    static constexpr uint32_t kStages = (MOM ? 2 : 3) + (WIDE ? 1 : 0);
    static constexpr uint32_t kWords = kSlot16 * kStages;
    static constexpr int kScales = (int)(kFlatBytes / 4 - 4 * kWords);          // floats left
    static __device__ float *scales(FlatSmem &sm) { return reinterpret_cast<float *>(sm.data + kWords); }
};
static_assert(FlatRing<false, false>::kScales >= kFlatScales && FlatRing<true, false>::kScales >= kFlatScales &&
                  FlatRing<false, true>::kScales >= kFlatWideScales && FlatRing<true, true>::kScales >= kFlatWideScales,
              "the planner's rows fit");

// Issues the copies of chunk c of the tile (vectors of rows r0, ...) into slot st.
template <bool MOM, bool WIDE>
__device__ __forceinline__ void flat_issue(const TensorDev &T, int64_t r0, uint32_t total, uint32_t c, uint32_t st,
                                           FlatSmem &sm, uint64_t pol) {
    using F = FlatRing<MOM, WIDE>;
    constexpr uint32_t kFlatChunk = F::kChunk, kSlot16 = F::kSlot16;
    const uint32_t bytes = min(kFlatChunk, total - c * kFlatChunk) * 16u;
    const uint64_t e0 = uint64_t(r0) * (uint64_t)T.m + uint64_t(c) * kFlatChunk * 8u;
    uint4 *dst = sm.data + st * kSlot16;
    mbar_expect_tx(&sm.full[st], MOM ? 3u * bytes : 2u * bytes);
    bulk_g2s(dst, T.w + e0, bytes, &sm.full[st], pol);
    if (MOM)
        bulk_g2s(dst + kFlatChunk, T.M + e0, 2u * bytes, &sm.full[st], pol);
    else
        bulk_g2s(dst + kFlatChunk, T.g + e0, bytes, &sm.full[st], pol);
}

template <bool MOM, bool WIDE, bool FAST>
__device__ bool apply_flat_body(const StepArgs &A, const TensorDev &T, int64_t r0, uint32_t total, float coefC,
                                FlatSmem &sm, uint64_t pol, Acc2 &acc) {
    using F = FlatRing<MOM, WIDE>;
    constexpr uint32_t kStages = F::kStages, kSlot16 = F::kSlot16, kFlatChunk = F::kChunk;
    const uint32_t V = (uint32_t)T.m / 8u, nch = (total + kFlatChunk - 1) / kFlatChunk;
    const int tid = threadIdx.x;
    uint16_t *__restrict__ w_ = T.w + r0 * T.m;
    const Dith d = dith_of(A, T);
    const uint64_t el0 = uint64_t(r0) * (uint64_t)T.m;
    const float wdf = T.decay ? A.wdf : 1.0f, ce = A.ce;
    const float2 wdf2 = make_float2(wdf, wdf);
    const Pol sp;
    const float *__restrict__ sb = F::scales(sm), *__restrict__ sa = sb + 8 * V;
    uint32_t row = tid / V, col = tid - row * V;  // of vector tid of the tile
    const uint32_t dq = kThreads / V, dr = kThreads - dq * V;
    uint32_t st = 0, par = 0;
    for (uint32_t c = 0; c < nch; ++c) {
        const uint32_t cnt = min(kFlatChunk, total - c * kFlatChunk);
        const bool ok = mbar_wait(&sm.full[st], par);
        const uint4 *bw = sm.data + st * kSlot16, *by = bw + kFlatChunk;
#pragma unroll
        for (uint32_t k = 0; k < kFlatChunk / kThreads; ++k) {
            const uint32_t f = k * kThreads + tid;
            if (f < cnt) {
                const float a = sa[row];
                const float4 b0 = *reinterpret_cast<const float4 *>(sb + 8 * col);
                const float4 b1 = *reinterpret_cast<const float4 *>(sb + 8 * col + 4);
                const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
                float y[8], w[8], x[8];
                if constexpr (MOM) {
                    const float4 m0 = reinterpret_cast<const float4 *>(by)[2 * f];
                    const float4 m1 = reinterpret_cast<const float4 *>(by)[2 * f + 1];
                    y[0] = m0.x; y[1] = m0.y; y[2] = m0.z; y[3] = m0.w;
                    y[4] = m1.x; y[5] = m1.y; y[6] = m1.z; y[7] = m1.w;
                } else {
                    unpack_bf8(by[f], y);
                }
                unpack_bf8(bw[f], w);
                if constexpr (FAST) {
                    const float cr = -coefC * a;
                    const float2 cr2 = make_float2(cr, cr);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 xx = __ffma2_rn(__fmul2_rn(cr2, make_float2(b[2 * q], b[2 * q + 1])),
                                                     make_float2(y[2 * q], y[2 * q + 1]),
                                                     __fmul2_rn(make_float2(w[2 * q], w[2 * q + 1]), wdf2));
                        x[2 * q] = xx.x;
                        x[2 * q + 1] = xx.y;
                    }
                } else {
                    float u[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        u[q] = y[q] * fminf(a * b[q], ce);
                        x[q] = fmaf(-coefC, u[q], w[q] * wdf);
                    }
                    acc.add(sumsq8(u));
                }
                const uint64_t e0 = uint64_t(c * kFlatChunk + f) * 8u;
                uint4 o;
                round8(x, d, el0 + e0, o);
                st16_hint(w_ + e0, o, sp.drop);
            }
            row += dq;
            col += dr;
            if (col >= V) {
                col -= V;
                ++row;
            }
        }
        // every thread is done with the slot: refill it
        if (__syncthreads_or(!ok)) {
            if (tid == 0) drain_copies(A.err, sm.full, kStages, c, min(nch, c + kStages));
            return false;
        }
        if (tid == 0 && c + kStages < nch) {
            fence_proxy_async_smem();
            flat_issue<MOM, WIDE>(T, r0, total, c + kStages, st, sm, pol);
        }
        if (++st == kStages) {
            st = 0;
            par ^= 1u;
        }
    }
    return true;
}

template <bool MOM, bool WIDE>
__device__ void apply_flat_tile(const StepArgs &A, const TensorDev &T, TensorScal &S, uint32_t item, FlatSmem &sm) {
    using F = FlatRing<MOM, WIDE>;
    constexpr uint32_t kStages = F::kStages, kFlatChunk = F::kChunk;
    float *ab = F::scales(sm);
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    const uint32_t trows = (item & kHalfTile) ? T.at_rows / 2 : T.at_rows;
    const int64_t r0 = int64_t(item & kTileMask) * T.at_rows + ((item & kSecondHalf) ? trows : 0);
    if (r0 >= T.n) return;  // the second half of a matrix's short last tile
    const uint32_t m = (uint32_t)T.m, rows_t = (uint32_t)min((int64_t)trows, T.n - r0), total = rows_t * (m / 8u);
    const uint32_t nch = (total + kFlatChunk - 1) / kFlatChunk;
    if (threadIdx.x == 0) {
        for (uint32_t st = 0; st < kStages; ++st) mbar_init(&sm.full[st], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (uint32_t c = 0; c < nch && c < kStages; ++c) flat_issue<MOM, WIDE>(T, r0, total, c, c, sm, pol);
    const float rbar_s = __ldcg(&S.rbar_s);
    const int rbar_e = __ldcg(&S.rbar_e);
    float ma = 0.f, mb = 0.f;
    const float4 *bsc = reinterpret_cast<const float4 *>(T.bsc);  // (the stores may alias the descriptor)
    const float *R = T.R + r0;
    for (uint32_t j = threadIdx.x; j < m / 4; j += kThreads) {
        const float4 b = __ldcg(bsc + j);
        reinterpret_cast<float4 *>(ab)[j] = b;
        mb = fmaxf(fmaxf(mb, fmaxf(nan_to_inf(b.x), nan_to_inf(b.y))), fmaxf(nan_to_inf(b.z), nan_to_inf(b.w)));
    }
    for (uint32_t r = threadIdx.x; r < rows_t; r += kThreads) {
        const float a = row_scale(__ldcg(R + r), rbar_s, rbar_e);
        ab[m + r] = a;
        ma = fmaxf(ma, nan_to_inf(a));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        ma = fmaxf(ma, __shfl_xor_sync(kAll, ma, o));
        mb = fmaxf(mb, __shfl_xor_sync(kAll, mb, o));
    }
    if ((threadIdx.x & 31) == 0) {
        sm.red[threadIdx.x >> 5] = ma;
        sm.red[kThreads / 32 + (threadIdx.x >> 5)] = mb;
    }
    __syncthreads();
    ma = mb = 0.f;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        ma = fmaxf(ma, sm.red[w]);
        mb = fmaxf(mb, sm.red[kThreads / 32 + w]);
    }
    const float coefC = __ldcg(&S.coefC);
    const bool sum = __ldcg(&S.fallback) == kSumInC;
    Acc2 acc;
    bool done;
    if (!sum && ma * mb <= A.ce)
        done = apply_flat_body<MOM, WIDE, true>(A, T, r0, total, coefC, sm, pol, acc);
    else
        done = apply_flat_body<MOM, WIDE, false>(A, T, r0, total, coefC, sm, pol, acc);
    if (sum && done) publish_sum(A, T, S, item, rows_t, acc, sm.sum);
}

// Phase B of a queued row-path tensor: sum(U^2) over the rows of a phase-C tile, from a ring of G (or the
// new M, which phase A stored) alone. Chunks run on from tile to tile (`turn` counts them), so that the
// barriers keep their phases. With all of 65M parameters in 173 matrices of 768 x 488 queued a step takes 188 us,
// 119 with none (118M in 354 of 816 x 408: 304 and 191).
template <bool MOM>
struct SumRing {
    static constexpr uint32_t kChunk = MOM ? 512 : 1024, kSlot16 = 1024, kStages = 4;  // vectors; 16 KB slots
    static constexpr uint32_t kWords = kSlot16 * kStages;
};
// What k_fallback has read of the queue of such tensors.
struct alignas(16) QueueSmem {
    uint32_t id[kThreads], end[kThreads];  // queued tensors, and the tiles up to and with each
    uint32_t warp[kThreads / 32];
};
constexpr int kSumScales = (kFlatBytes - (int)sizeof(QueueSmem)) / 4 - 4 * (int)SumRing<false>::kWords;
static_assert(kSumScales >= kFlatWideScales && kSumScales >= 4096 + 128, "the planner's rows fit");

template <bool MOM>
__device__ bool sum_tile(const StepArgs &A, const TensorDev &T, TensorScal &S, uint32_t tile, uint32_t &turn, FlatSmem &sm) {
    using F = SumRing<MOM>;
    const int tid = threadIdx.x;
    const int64_t r0 = int64_t(tile) * T.at_rows;
    const uint32_t m = (uint32_t)T.m, V = m / 8u, rows_t = (uint32_t)min((int64_t)T.at_rows, T.n - r0), total = rows_t * V;
    const uint32_t nch = (total + F::kChunk - 1) / F::kChunk;
    const uint64_t pol = read_policy(false);
    const char *src = MOM ? reinterpret_cast<const char *>(T.M + r0 * T.m) : reinterpret_cast<const char *>(T.g + r0 * T.m);
    const uint32_t t0 = turn;
    auto issue = [&](uint32_t c) {
        const uint32_t st = (t0 + c) % F::kStages, bytes = min(F::kChunk, total - c * F::kChunk) * (MOM ? 32u : 16u);
        mbar_expect_tx(&sm.full[st], bytes);
        bulk_g2s(sm.data + st * F::kSlot16, src + uint64_t(c) * F::kChunk * (MOM ? 32u : 16u), bytes, &sm.full[st], pol);
    };
    if (tid == 0) {
        fence_proxy_async_smem();
        for (uint32_t c = 0; c < nch && c < F::kStages; ++c) issue(c);
    }
    float *ab = reinterpret_cast<float *>(sm.data + F::kWords);
    const float rbar_s = __ldcg(&S.rbar_s), ce = A.ce;
    const int rbar_e = __ldcg(&S.rbar_e);
    for (uint32_t j = tid; j < m / 4; j += kThreads)
        reinterpret_cast<float4 *>(ab)[j] = __ldcg(reinterpret_cast<const float4 *>(T.bsc) + j);
    for (uint32_t r = tid; r < rows_t; r += kThreads) ab[m + r] = row_scale(__ldcg(T.R + r0 + r), rbar_s, rbar_e);
    __syncthreads();
    const float *sb = ab, *sa = ab + m;
    uint32_t row = tid / V, col = tid - row * V;
    const uint32_t dq = kThreads / V, dr = kThreads - dq * V;
    Acc2 acc;
    for (uint32_t c = 0; c < nch; ++c) {
        const uint32_t cnt = min(F::kChunk, total - c * F::kChunk), st = (t0 + c) % F::kStages;
        const bool ok = mbar_wait(&sm.full[st], ((t0 + c) / F::kStages) & 1u);
        const uint4 *by = sm.data + st * F::kSlot16;
#pragma unroll
        for (uint32_t k = 0; k < F::kChunk / kThreads; ++k) {
            const uint32_t f = k * kThreads + tid;
            if (f < cnt) {
                const float a = sa[row];
                const float4 b0 = *reinterpret_cast<const float4 *>(sb + 8 * col);
                const float4 b1 = *reinterpret_cast<const float4 *>(sb + 8 * col + 4);
                const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
                float y[8], u[8];
                if constexpr (MOM)
                    lds8(reinterpret_cast<const float *>(by) + 8 * f, y);
                else
                    unpack_bf8(by[f], y);
#pragma unroll
                for (int q = 0; q < 8; ++q) u[q] = y[q] * fminf(a * b[q], ce);
                acc.add(sumsq8(u));
            }
            row += dq;
            col += dr;
            if (col >= V) {
                col -= V;
                ++row;
            }
        }
        if (__syncthreads_or(!ok)) {  // every thread is done with the slot: refill it
            if (tid == 0) drain_copies(A.err, sm.full, F::kStages, t0 + c, t0 + min(nch, c + F::kStages));
            return false;
        }
        if (tid == 0 && c + F::kStages < nch) {
            fence_proxy_async_smem();
            issue(c + F::kStages);
        }
    }
    turn = t0 + nch;
    publish_sum(A, T, S, tile, rows_t, acc, sm.sum);
    __syncthreads();  // the scales and sums are free for the next tile
    return true;
}

// ---------------------------------------------------------------------------
// A step of small tensors only (k_small): a cluster of CTAs takes one tensor through the whole step.
// Each CTA keeps a slice of it (whole rows of a factored tensor) in shared memory as fp32, so G is read
// once and nothing goes through the workspace; the CTAs exchange column sums, sum of R and sum of U^2
// through distributed shared memory, three cluster barriers in all. Bound by latency: one launch with
// three trips to memory (G; M or v; W) instead of the four launches of the strip tiles.
// Toy MoE (296K elements in 39 tensors), in L2: 28 us as four launches, 17 us so; a 141 x 208 matrix
// through the no-alloc entry point 24 and 15 us. A cluster spends 10 us: 1 on G, 2 on its sums, 2
// on C and the scales, 1 on U, 2 on the scalars (fp64 is slow here), 1 on W, the rest in barriers.
// ---------------------------------------------------------------------------
struct SmallSmem {
    float2 rsum, u2;   // this CTA's sums of R and of (U / coef)^2, (hi, lo), read by the cluster
    TensorScal scal;   // the tensor's scalars (the same in every CTA of the cluster)
    float2 red2[kSmallThreads / 32];
    float part[kSmallThreads];
};

// The CTA's slice: rows [r0, r1) of a factored tensor, elements [e0, e1).
struct SmallSlice {
    int64_t r0, r1, e0, e1;
    __device__ SmallSlice(const TensorDev &T, uint32_t rank) {
        r0 = min(int64_t(rank) * T.srows, T.n);
        r1 = min(r0 + (int64_t)T.srows, T.n);
        e0 = r0 * T.m;
        e1 = r1 * T.m;
    }
};

// Eight fp32 values to shared memory (16-byte aligned).
__device__ __forceinline__ void sts8(float *p, const float (&o)[8]) {
    reinterpret_cast<float4 *>(p)[0] = make_float4(o[0], o[1], o[2], o[3]);
    reinterpret_cast<float4 *>(p)[1] = make_float4(o[4], o[5], o[6], o[7]);
}

// CTA-wide compensated sum; the result (hi, lo) is valid in warp 0.
__device__ __forceinline__ Acc2 small_sum(Acc2 a, float2 *red) {
    auto fold = [&](int o) {
        const float h = __shfl_xor_sync(kAll, a.hi, o), l = __shfl_xor_sync(kAll, a.lo, o);
        float s, e;
        two_sum(a.hi, h, s, e);
        a.hi = s;
        a.lo += l + e;
    };
#pragma unroll
    for (int o = 16; o; o >>= 1) fold(o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(a.hi, a.lo);
    __syncthreads();
    if (threadIdx.x < 32) {
        const float2 p = red[threadIdx.x & (kSmallThreads / 32 - 1)];
        a.hi = p.x;
        a.lo = p.y;
#pragma unroll
        for (int o = kSmallThreads / 64; o; o >>= 1) fold(o);
    }
    return a;
}

// Every CTA's value at `p` (the same place in each), all loads in flight together; zeros past the cluster.
template <typename V>
__device__ __forceinline__ void cluster_values(cooperative_groups::cluster_group &cl, V *p, uint32_t ranks, V (&v)[8]) {
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) v[k] = k < ranks ? *cl.map_shared_rank(p, k) : V{};
}

// The sum of the cluster's (hi, lo) pairs at `p`, in rank order.
__device__ __forceinline__ double cluster_pairs(cooperative_groups::cluster_group &cl, float2 *p, uint32_t ranks) {
    float2 v[8];
    cluster_values(cl, p, ranks, v);
    double s = 0.0;
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k)
        if (k < ranks) s += pair_value(v[k].x, v[k].y);
    return s;
}

// (The descriptor by value: its fields stay in registers across the stores.)
__device__ void small_step(const StepArgs &A, const TensorDev T, TensorScal *out, float *mem) {
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const uint32_t rank = cl.block_rank(), ranks = cl.num_blocks();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int TPB = kSmallThreads;
    const SmallSlice L(T, rank);
    const int rows = (int)(L.r1 - L.r0), m = (int)T.m, cnt = (int)(L.e1 - L.e0);
    const bool fact = T.kind == kKindFactored, mom = T.momentum != 0;
    SmallSmem &sm = *reinterpret_cast<SmallSmem *>(mem);
    float *y = mem + (sizeof(SmallSmem) + 15) / 16 * 4;  // [srows m]: g, then U / coef (zeros to a multiple of 8)
    float *a = y + size_t(T.srows) * m;                  // [srows] R, then a_i (srows is a multiple of 8)
    float *cp = a + T.srows;                             // [m] this CTA's column sums, read by the cluster
    float *b = cp + m;                                   // [m] old C, then b_j
    const Pol pol;
    const GScale gsc = grad_scale(A);
    const Dith d = dith_of(A, T);
    // G into y; the lines of M or v and of W are asked for in the same trip
    for (int i = 8 * tid; i < cnt; i += 8 * TPB) {
        const int64_t e = L.e0 + i;
        const int valid = min(8, cnt - i);
        float g[8];
        load8_elem(T.g, T.f32, T.wal, e, valid, g, pol);
        if (mom) asm volatile("prefetch.global.L2 [%0];" ::"l"(T.M + e));
        if (!fact) asm volatile("prefetch.global.L2 [%0];" ::"l"(T.v + e));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char *>(T.w) + (T.f32 ? 4 : 2) * e));
        sts8(y + i, g);
    }
    if (fact) {
        for (int j = tid; j < m; j += TPB) b[j] = __ldcg(T.C + j);
        for (int r = tid; r < rows; r += TPB) a[r] = __ldcg(T.R + L.r0 + r);
    }
    __syncthreads();
    if (fact) {
        // row sums: 2^lg lanes per row, about 16 elements each; R_i of the CTA's rows
        Acc2 rd;
        int lg = 0;
        while (lg < 5 && (16 << lg) < m) ++lg;
        const int g = 1 << lg, gl = lane & (g - 1), rpw = 32 >> lg;
        for (int r0 = warp * rpw; r0 < rows; r0 += rpw * (TPB / 32)) {
            const int r = r0 + (lane >> lg);
            float sum = 0.f;
            if (r < rows)
                for (int j = gl; j < m; j += g) sum = fmaf(y[r * m + j], y[r * m + j], sum);
            for (int o = g >> 1; o; o >>= 1) sum += __shfl_xor_sync(kAll, sum, o);
            if (gl == 0 && r < rows) {
                const float Rn = fmaf(A.b2, a[r], gsc.c2 * __fdiv_rn(sum, (float)m));
                a[r] = Rn;
                T.R[L.r0 + r] = Rn;
                rd.add(Rn);
            }
        }
        // column sums: a thread per column and run of rows
        const int runs = m < TPB ? TPB / m : 1;
        if (runs > 1) {
            const int j = tid % m, q = tid / m, per = (rows + runs - 1) / runs;
            float sum = 0.f;
            if (q < runs)
                for (int r = q * per; r < min(rows, (q + 1) * per); ++r) sum = fmaf(y[r * m + j], y[r * m + j], sum);
            sm.part[tid] = sum;
            __syncthreads();
            if (tid < m) {
                for (int k = 1; k < runs; ++k) sum += sm.part[k * m + tid];
                cp[tid] = sum;
            }
        } else {
            for (int j = tid; j < m; j += TPB) {
                float sum = 0.f;
                for (int r = 0; r < rows; ++r) sum = fmaf(y[r * m + j], y[r * m + j], sum);
                cp[j] = sum;
            }
        }
        rd = small_sum(rd, sm.red2);
        if (tid == 0) sm.rsum = make_float2(rd.hi, rd.lo);
        cl.sync();  // column sums and sums of R of the cluster; every CTA has read the old C
        for (int j = tid; j < m; j += TPB) {
            float v[8], cs = 0.f;
            cluster_values(cl, cp + j, ranks, v);
#pragma unroll
            for (int k = 0; k < 8; ++k) cs += v[k];
            const float Cn = fmaf(A.b2, b[j], gsc.c2 * __fdiv_rn(cs, (float)T.n));
            if (rank == 0) T.C[j] = Cn;
            b[j] = __frsqrt_rn(Cn);
        }
        // beside the columns of the first warps
        if (tid == TPB - 32) set_rbar(sm.scal, cluster_pairs(cl, &sm.rsum, ranks) * T.inv_n);
        __syncthreads();
        const float rbar_s = sm.scal.rbar_s;
        const int rbar_e = sm.scal.rbar_e;
        for (int r = tid; r < rows; r += TPB) a[r] = row_scale(a[r], rbar_s, rbar_e);
        __syncthreads();
    } else if (tid == 0) {
        sm.scal.rbar = 0.0;
        sm.scal.rbar_s = 0.f;
        sm.scal.rbar_e = 0;
    }
    // M, v, and U / coef into y
    Acc2 acc;
    for (int i = 8 * tid; i < cnt; i += 8 * TPB) {
        const int64_t e = L.e0 + i;
        const int valid = min(8, cnt - i);
        float g[8], mm[8], v[8], u[8];
        lds8(y + i, g);  // 0 past the slice
        if (mom) load_f8(T.M + e, T.sal, valid, mm);
        if (!fact) load_f8(T.v + e, T.sal, valid, v);
        int r = fact ? i / m : 0, j = i - r * m;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            float sc = 0.f;
            if (fact) {
                if (c < valid) sc = fminf(a[r] * b[j], A.ce);
                const bool wrap = ++j == m;
                j = wrap ? 0 : j;
                r += wrap;
            } else {
                v[c] = fmaf(A.b2, v[c], gsc.c2 * (g[c] * g[c]));
                sc = fminf(__frsqrt_rn(v[c]), A.ce);
            }
            const float yy = mom ? fmaf(A.b1, mm[c], gsc.c1 * g[c]) : g[c];
            mm[c] = yy;
            u[c] = c < valid ? yy * sc : 0.f;
        }
        sts8(y + i, u);
        if (mom) store_f8(T.M + e, T.sal, valid, mm);
        if (!fact) store_f8(T.v + e, T.sal, valid, v);
        acc.add(sumsq8(u));
    }
    acc = small_sum(acc, sm.red2);
    if (tid == 0) sm.u2 = make_float2(acc.hi, acc.lo);
    cl.sync();
    double s2 = 0.0;
    if (tid == 0) {
        s2 = cluster_pairs(cl, &sm.u2, ranks);
        // (fp64 roots are slow here: an update that is not clipped goes on without it)
        const double coef = update_coef(A, T), d = (double)A.clip_d;
        if (s2 * coef * coef * T.inv_numel > d * d)
            set_clip(A, T, sm.scal, s2);
        else
            sm.scal.coefC = (float)((double)A.lr * coef);
    }
    __syncthreads();
    const float coefC = sm.scal.coefC, wdf = T.decay ? A.wdf : 1.0f;
    for (int i = 8 * tid; i < cnt; i += 8 * TPB) {
        const int64_t e = L.e0 + i;
        const int valid = min(8, cnt - i);
        float u[8], w[8], x[8];
        load8_elem(T.w, T.f32, T.wal, e, valid, w, pol);
        lds8(y + i, u);
#pragma unroll
        for (int c = 0; c < 8; ++c) x[c] = fmaf(-coefC, u[c], w[c] * wdf);
        store8_elem(T, d, e, valid, x, pol);
    }
    if (tid == 0 && rank == 0) {
        const TensorScal &c = sm.scal;
        out->rbar = c.rbar;
        out->rbar_s = c.rbar_s;
        out->rbar_e = c.rbar_e;
        set_clip(A, T, *out, s2);
    }
    cl.sync();  // no CTA leaves while another may still read its shared memory
}

// ---------------------------------------------------------------------------
// Kernels: one tile / item per CTA. The per-step parameters are a kernel
// parameter (constant bank), so the dither keys and step scalars are uniform
// operands of every warp.
// ---------------------------------------------------------------------------
__device__ void phase_A_strip(const TensorDev &T, uint32_t tile, Smem &sm, const Pol &pol) {
    if (T.vec)
        sumsq_tile<true>(T, tile, sm, pol);
    else
        sumsq_tile<false>(T, tile, sm, pol);
}

// Phase C of a strip or flat tile.
__device__ void phase_C(const StepArgs &A, const TensorDev &T, const TensorScal &S, uint32_t tile, Meta &meta,
                        const Pol &pol) {
    if (T.kind != kKindFactored) {
        apply_full_tile(A, T, S, tile, pol);
    } else if (!T.vec) {
        if (T.m > kFlatCols)
            apply_flat_any<true>(A, T, S, tile, meta, pol);
        else
            apply_flat_any<false>(A, T, S, tile, meta, pol);
    } else {
        const bool fast = fill_meta(T, S, tile, A.ce, meta);
        if (T.momentum) {
            if (fast)
                apply_fact_tile<true, true>(A, T, S, tile, meta, pol);
            else
                apply_fact_tile<true, false>(A, T, S, tile, meta, pol);
        } else {
            if (fast)
                apply_fact_tile<false, true>(A, T, S, tile, meta, pol);
            else
                apply_fact_tile<false, false>(A, T, S, tile, meta, pol);
        }
    }
}

// The launches of a step are programmatic dependents of one another: a launch may start when every
// CTA of the one before has, so that its launch latency (and the load of its item) passes while that
// one ends, and it waits here, before it touches anything another launch writes, until that one is
// complete and its writes are visible. Each launch waits, so completion is transitive. A step's last launch
// releases nothing: the next step begins with an ordinary launch, and a programmatic dependent of the caller's
// would start while phase C still writes the weights (one that stamps its start and its wait's end: up to
// 43 us apart behind 160M parameters). `items`: the
// CTA's (tensor, tile) table, written at bind; null: tensor 0, tiles in order.
// A step of 296K elements in 39 tensors 37 -> 28 us, 2048 x 1408 alone 43 -> 35, the 6.78B set 8357 -> 8322.
__device__ __forceinline__ void wait_previous_launch() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void let_next_launch_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A CTA's item, with its tensor's descriptor copied to shared memory: one trip to L2 for all of it, where
// reading fields as they are needed, between barriers, is a chain of trips. Both come from bind and are
// read before the wait; the no-alloc step, without tables, passes its descriptor as a parameter.
// Against reading fields from L2: 24 ragged tensors 150 -> 135 us, a 432-wide model 69 -> 61, a 2048-wide
// one 378 -> 369, the 6.78B set 8349 -> 8318.
// `release`: another launch of the step follows.
__device__ __forceinline__ uint2 begin_item(const uint2 *__restrict__ items, const StepArgs &A, TensorDev &td,
                                            bool release = true) {
    constexpr uint32_t kWords = sizeof(TensorDev) / 4;
    static_assert(sizeof(TensorDev) % 4 == 0 && kWords <= kThreads, "one word per thread");
    if (release) let_next_launch_start();
    const uint2 it = items ? items[blockIdx.x] : make_uint2(0u, blockIdx.x);
    if (threadIdx.x < kWords)
        reinterpret_cast<uint32_t *>(&td)[threadIdx.x] =
            items ? __ldcg(reinterpret_cast<const uint32_t *>(A.tensors + it.x) + threadIdx.x)
                  : reinterpret_cast<const uint32_t *>(&A.one)[threadIdx.x];
    wait_previous_launch();
    __syncthreads();
    return it;
}

// Clears the per-step scalars and the length of the phase-B queue (words of 4 bytes).
__global__ void k_reset(uint32_t *p, uint32_t words) {
    let_next_launch_start();
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < words; k += gridDim.x * blockDim.x) p[k] = 0u;
}

__global__ void __launch_bounds__(kThreads, SKEW_MINB_SUMSQ)
    k_sumsq(const __grid_constant__ StepArgs A, const uint2 *__restrict__ items) {
    __shared__ Smem sm;
    __shared__ TensorDev td;
    const uint2 it = begin_item(items, A, td);
    phase_A_strip(td, it.y, sm, Pol());
}

// A step with row-path tensors runs its strip and flat tiles in the row path's launches, ahead of
// the row tiles, unless there are many of them (kRideElems): phase B of the flat tiles needs nothing from phase A or the finalize, so it comes
// with phase A. Such a step has four launches (after k_reset) instead of seven, and the light tiles' latency (a
// launch of its own took 12 to 25 us each for phases A, B and C) hides behind the row tiles.

// Row path, phase A: one row tile per CTA (dynamic shared memory: RowSmem), and before them the
// phase-A strip tiles and phase-B flat tiles.
__global__ void __launch_bounds__(kThreads, 2)
    k_rowsq(const __grid_constant__ StepArgs A, const uint2 *__restrict__ items) {
    extern __shared__ uint4 dyn_smem[];
    RowSmem &sm = *reinterpret_cast<RowSmem *>(dyn_smem);
    __shared__ TensorDev td;
    const uint2 it = begin_item(items, A, td);
    const TensorDev &T = td;
    TensorScal &S = A.scal[it.x];
    if (T.rowpath == kRowNone) {
        Smem &ss = *reinterpret_cast<Smem *>(dyn_smem);
        if (T.kind == kKindFactored)
            phase_A_strip(T, it.y, ss, Pol());
        else
            phase_B_full(A, T, it.x, it.y, ss, Pol());
        return;
    }
    if (T.rowpath == kRowAny) {
        GenSmem<8> &gs = *reinterpret_cast<GenSmem<8> *>(dyn_smem);
        const bool two = T.m > 2048;
        if (T.momentum) {
            if (two)
                rowsq_gen_tile<8, 2, true>(A, T, S, it.y, gs);
            else
                rowsq_gen_tile<8, 1, true>(A, T, S, it.y, gs);
        } else {
            if (two)
                rowsq_gen_tile<8, 2, false>(A, T, S, it.y, gs);
            else
                rowsq_gen_tile<8, 1, false>(A, T, S, it.y, gs);
        }
        return;
    }
    if (T.momentum) {
        MomRowSmem &ms = *reinterpret_cast<MomRowSmem *>(dyn_smem);
        switch (T.m) {
            case 4096: rowsq_mom_tile<kThreads, 512>(A, T, S, it.y, ms); break;
            case 2048: rowsq_mom_tile<kThreads, 256>(A, T, S, it.y, ms); break;
            case 1024: rowsq_mom_tile<kThreads, 128>(A, T, S, it.y, ms); break;
            default: rowsq_mom_tile<kThreads, 64>(A, T, S, it.y, ms); break;  // 512
        }
        return;
    }
    switch (T.m) {
        case 4096: rowsq_tile<kThreads, 512>(A, T, S, it.y, sm); break;
        case 2048: rowsq_tile<kThreads, 256>(A, T, S, it.y, sm); break;
        case 1024: rowsq_tile<kThreads, 128>(A, T, S, it.y, sm); break;
        default: rowsq_tile<kThreads, 64>(A, T, S, it.y, sm); break;  // 512
    }
}

// Row path, phase A of the widths above 4096: one row tile per CTA, one CTA per SM.
__global__ void __launch_bounds__(kWideThreads, 1)
    k_rowsq_wide(const __grid_constant__ StepArgs A, const uint2 *__restrict__ items) {
    extern __shared__ uint4 dyn_smem[];
    GenSmem<16> &gs = *reinterpret_cast<GenSmem<16> *>(dyn_smem);
    __shared__ TensorDev td;
    const uint2 it = begin_item(items, A, td);
    const TensorDev &T = td;
    if (T.momentum)
        rowsq_gen_tile<16, 2, true>(A, T, A.scal[it.x], it.y, gs);
    else
        rowsq_gen_tile<16, 2, false>(A, T, A.scal[it.x], it.y, gs);
}

// Row path, phase C: one row tile per CTA (dynamic shared memory: ApplyRowSmem), and before them
// the phase-C strip and flat tiles.
__global__ void __launch_bounds__(kThreads, 2)
    k_apply_rows(const __grid_constant__ StepArgs A, const uint2 *__restrict__ items) {
    extern __shared__ uint4 dyn_smem[];
    ApplyRowSmem &sm = *reinterpret_cast<ApplyRowSmem *>(dyn_smem);
    __shared__ TensorDev td;
    const uint2 it = begin_item(items, A, td, false);
    const TensorDev &T = td;
    TensorScal &S = A.scal[it.x];
    if (T.rowpath == kRowNone) {
        phase_C(A, T, S, it.y, *reinterpret_cast<Meta *>(dyn_smem), Pol());
        return;
    }
    if (T.rowpath == kRowAny) {
        FlatSmem &fs = *reinterpret_cast<FlatSmem *>(dyn_smem);
        const bool wide = T.m > kAnyNarrow;
        if (T.momentum) {
            if (wide)
                apply_flat_tile<true, true>(A, T, S, it.y, fs);
            else
                apply_flat_tile<true, false>(A, T, S, it.y, fs);
        } else {
            if (wide)
                apply_flat_tile<false, true>(A, T, S, it.y, fs);
            else
                apply_flat_tile<false, false>(A, T, S, it.y, fs);
        }
        return;
    }
    if (T.momentum) {
        MomApplySmem &ms = *reinterpret_cast<MomApplySmem *>(dyn_smem);
        switch (T.m) {
            case 4096: apply_rows_mom_tile<kThreads, 512>(A, T, S, it.y, ms); break;
            case 2048: apply_rows_mom_tile<kThreads, 256>(A, T, S, it.y, ms); break;
            case 1024: apply_rows_mom_tile<kThreads, 128>(A, T, S, it.y, ms); break;
            default: apply_rows_mom_tile<kThreads, 64>(A, T, S, it.y, ms); break;  // 512
        }
        return;
    }
    switch (T.m) {
        case 4096: apply_rows_tile<kThreads, 512>(A, T, S, it.y, sm); break;
        case 2048: apply_rows_tile<kThreads, 256>(A, T, S, it.y, sm); break;
        case 1024: apply_rows_tile<kThreads, 128>(A, T, S, it.y, sm); break;
        default: apply_rows_tile<kThreads, 64>(A, T, S, it.y, sm); break;  // 512
    }
}

// Phase B of the row-path tensors whose finalize found that a clamp may bind and the update be clipped
// (queued in A.fb): the CTAs of this grid share the phase-C tiles of all queued tensors, laid end to end
// (starting every tensor at CTA 0 would give the first CTAs a tile of each small one). The first nB CTAs
// run the phase-B strip and flat tiles of the other tensors.
// A CTA reads the queue kThreads tensors at a time, one per thread, and finds its tiles among the running
// sums of their tile counts: walking from tensor to tensor cost two dependent trips to L2 for each, which every
// CTA paid (82 MiB of G, 121 of its matrices queued, no momentum: k_fallback 78 us so, 45 now, the step 171 and 138).
// Loads queue entries [q0, q0 + kThreads) (ids and running tile counts); returns the tiles they hold.
__device__ uint32_t load_queue(const StepArgs &A, uint32_t q0, uint32_t cnt, QueueSmem &qs) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t t = 0, n = 0;
    if (q0 + tid < cnt) {
        t = __ldcg(A.fb + 1 + q0 + tid);
        n = A.tensors ? __ldg(&A.tensors[t].atiles) : A.one.atiles;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t p = __shfl_up_sync(kAll, n, o);
        if (lane >= o) n += p;
    }
    if (lane == 31) qs.warp[warp] = n;
    __syncthreads();
    for (int w = 0; w < warp; ++w) n += qs.warp[w];
    qs.id[tid] = t;
    qs.end[tid] = n;
    __syncthreads();
    return qs.end[kThreads - 1];
}

__global__ void __launch_bounds__(kThreads, 2)
    k_fallback(const __grid_constant__ StepArgs A, const uint2 *__restrict__ items, uint32_t nB) {
    extern __shared__ uint4 dyn_smem[];
    __shared__ TensorDev td;
    if (blockIdx.x < nB) {
        struct Own {
            Smem sm;
            Meta meta;
        };
        Own &o = *reinterpret_cast<Own *>(dyn_smem);
        static_assert(sizeof(Own) <= sizeof(FlatSmem), "k_fallback's shared memory");
        const uint2 it = begin_item(items, A, td);
        phase_B_fact(A, td, it.x, it.y, o.sm, o.meta, Pol());
        return;
    }
    let_next_launch_start();
    wait_previous_launch();
    const uint32_t cnt = __ldcg(A.fb), ctas = gridDim.x - nB;
    if (!cnt) return;
    FlatSmem &sm = *reinterpret_cast<FlatSmem *>(dyn_smem);
    QueueSmem &qs = *reinterpret_cast<QueueSmem *>(sm.data + (kFlatBytes - sizeof(QueueSmem)) / 16);  // past the scales
    if (threadIdx.x == 0) {
        for (uint32_t st = 0; st < 4; ++st) mbar_init(&sm.full[st], 1);
        fence_mbar_init();
    }
    uint32_t tile = blockIdx.x - nB, turn = 0;  // of the tensors from queue entry q0 on
    for (uint32_t q0 = 0; q0 < cnt; q0 += kThreads) {
        const uint32_t total = load_queue(A, q0, cnt, qs);
        for (; tile < total; tile += ctas) {
            uint32_t k = 0;  // the first entry whose tiles go past this one
#pragma unroll
            for (uint32_t step = kThreads / 2; step; step >>= 1)
                if (qs.end[k + step - 1] <= tile) k += step;
            const uint32_t t = qs.id[k], local = tile - (k ? qs.end[k - 1] : 0u);
            if (threadIdx.x < sizeof(TensorDev) / 4)
                reinterpret_cast<uint32_t *>(&td)[threadIdx.x] =
                    A.tensors ? __ldg(reinterpret_cast<const uint32_t *>(A.tensors + t) + threadIdx.x)
                              : reinterpret_cast<const uint32_t *>(&A.one)[threadIdx.x];
            __syncthreads();
            TensorScal &S = A.scal[t];
            if (!(td.momentum ? sum_tile<true>(A, td, S, local, turn, sm) : sum_tile<false>(A, td, S, local, turn, sm)))
                return;
        }
        tile -= total;
    }
}

__global__ void __launch_bounds__(kThreads) k_finalize(const __grid_constant__ StepArgs A, const uint2 *__restrict__ items) {
    __shared__ Smem sm;
    __shared__ TensorDev td;
    const uint2 it = begin_item(items, A, td);
    phase_F(A, td, it.x, it.y, sm);
}

__global__ void __launch_bounds__(kThreads, SKEW_MINB_RMS)
    k_rms(const __grid_constant__ StepArgs A, const uint2 *__restrict__ items) {
    __shared__ Smem sm;
    __shared__ Meta meta;
    __shared__ TensorDev td;
    const uint2 it = begin_item(items, A, td);
    const TensorDev &T = td;
    if (T.kind == kKindFactored)
        phase_B_fact(A, T, it.x, it.y, sm, meta, Pol());
    else
        phase_B_full(A, T, it.x, it.y, sm, Pol());
}

__global__ void __launch_bounds__(kThreads, SKEW_MINB_APPLY)
    k_apply(const __grid_constant__ StepArgs A, const uint2 *__restrict__ items, bool last) {
    __shared__ Meta meta;
    __shared__ TensorDev td;
    const uint2 it = begin_item(items, A, td, !last);
    phase_C(A, td, A.scal[it.x], it.y, meta, Pol());
}

// One cluster per tensor of the handle, or (tensors null) the one tensor A.one.
__global__ void __launch_bounds__(kSmallThreads, 2)
    k_small(const __grid_constant__ StepArgs A) {
    extern __shared__ uint4 dyn_smem[];
    const uint32_t t = blockIdx.x / cooperative_groups::this_cluster().num_blocks();
    small_step(A, A.tensors ? A.tensors[t] : A.one, A.scal + t, reinterpret_cast<float *>(dyn_smem));
}

// Self-test of the bounded wait: one thread waits, exactly as the row kernels wait for
// a chunk, on an mbarrier phase that nothing completes (no arrival, no transaction);
// the wait gives up after kMbarPolls polls and the timeout lands in the status word.
__global__ void k_wait_selftest(uint32_t *err) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
        if (!mbar_wait(&bar, 0u)) atomicOr(err, 2u);
    }
}

}  // namespace

int launch_wait_selftest(uint32_t *err, void *stream) {
    k_wait_selftest<<<1, 32, 0, (cudaStream_t)stream>>>(err);
    return (int)cudaGetLastError();
}

constexpr size_t max3(size_t a, size_t b, size_t c) { return a > b ? (a > c ? a : c) : (b > c ? b : c); }

namespace {

// Launches `k` as a programmatic dependent of the launch before it in the stream (k waits for it
// itself, wait_previous_launch).
template <typename... P, typename... Q>
cudaError_t launch(void (*k)(P...), uint32_t grid, uint32_t threads, size_t smem, cudaStream_t s, Q... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

}  // namespace

int launch_small(const StepArgs &A, uint32_t tensors, const SmallPlan &P, void *stream, void *const *ev) {
    cudaStream_t s = (cudaStream_t)stream;
    static_assert(kSmallHeadBytes >= (sizeof(SmallSmem) + 15) / 16 * 16, "k_small's shared memory");
    if (ev)
        for (int k = 0; k < kLaunches; ++k) cudaEventRecord((cudaEvent_t)ev[k], s);
    // (always the most that a step may take: the attribute is the process's, and other threads launch too)
    cudaError_t e = cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem);
    if (e != cudaSuccess) return (int)e;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = P.ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(tensors * P.ctas);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = P.smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_small, A);
    if (ev) cudaEventRecord((cudaEvent_t)ev[kLaunches], s);
    return (int)e;
}

int launch_reset(void *p, size_t bytes, void *stream) {
    const uint32_t words = (uint32_t)(bytes / 4), grid = (words + kThreads - 1) / kThreads;
    // An ordinary launch: with the steps chained too, no SM ever drains, and the strip kernels then keep
    // the row kernels' shared-memory carve-out and run short of L1 (1.15B elements in strip tiles: 2322
    // us with steps apart, 2657 chained).
    k_reset<<<grid < 16 ? grid : 16, kThreads, 0, (cudaStream_t)stream>>>((uint32_t *)p, words);
    return (int)cudaGetLastError();
}

int launch_phases(const StepArgs &A, const LaunchPlan &L, void *stream, void *const *ev) {
    cudaStream_t s = (cudaStream_t)stream;
    auto mark = [&](int k) {
        if (ev) cudaEventRecord((cudaEvent_t)ev[k], s);
    };
    cudaError_t e = cudaSuccess;
    auto run = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
    };
    auto past = [](const uint2 *t, uint32_t n) { return t ? t + n : t; };
    const bool rows = L.nR != 0;
    const uint32_t rA = L.ride ? L.nA : 0, rB = L.ride ? L.nB : 0, rC = L.ride ? L.nC : 0;  // with the row tiles
    mark(0);
    if (L.nA > rA) run(launch(k_sumsq, L.nA, kThreads, 0, s, A, L.itemsA));
    mark(1);
    if (rows) {
        constexpr size_t kSm = max3(sizeof(RowSmem), sizeof(MomRowSmem), sizeof(GenSmem<8>));
        run(cudaFuncSetAttribute(k_rowsq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSm));
        if (rA + L.nR > L.nRW) run(launch(k_rowsq, rA + L.nR - L.nRW, kThreads, kSm, s, A, past(L.itemsA, L.nA - rA)));
        constexpr size_t kWide = sizeof(GenSmem<16>);
        static_assert(kWide + 1024 <= 227 * 1024, "one CTA per SM");
        if (L.nRW) {
            run(cudaFuncSetAttribute(k_rowsq_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWide));
            run(launch(k_rowsq_wide, L.nRW, kWideThreads, kWide, s, A, past(L.itemsA, L.nA + L.nR - L.nRW)));
        }
    }
    mark(2);
    if (L.nF) run(launch(k_finalize, L.nF, kThreads, 0, s, A, L.itemsF));
    mark(3);
    if (L.nB > rB) run(launch(k_rms, L.nB, kThreads, 0, s, A, L.itemsB));
    mark(4);
    if (rows) {
        run(cudaFuncSetAttribute(k_fallback, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FlatSmem)));
        run(launch(k_fallback, rB + L.nFB, kThreads, sizeof(FlatSmem), s, A, L.itemsB, rB));
    }
    mark(5);
    if (L.nC > rC) run(launch(k_apply, L.nC, kThreads, 0, s, A, L.itemsC, !rows));
    mark(6);
    if (rows) {
        constexpr size_t kSm = max3(sizeof(ApplyRowSmem), sizeof(MomApplySmem), sizeof(FlatSmem));
        static_assert(2 * (kSm + 1024 + (sizeof(TensorDev) + 127) / 128 * 128) <= 228 * 1024, "two CTAs per SM");
        static_assert(sizeof(Meta) <= kSm && sizeof(Smem) <= kSm, "light tiles");
        run(cudaFuncSetAttribute(k_apply_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSm));
        run(launch(k_apply_rows, rC + L.nCR, kThreads, kSm, s, A, past(L.itemsC, L.nC - rC)));
    }
    mark(7);
    return (int)e;
}

}  // namespace skew
