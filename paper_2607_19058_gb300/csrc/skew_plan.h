// Internal layout shared by the host planner (skew_host.cpp), the no-alloc
// entry point (skew_noalloc.cu) and the device kernels (skew_kernels.cu) of
// libskewadam. Not part of the public ABI.
#pragma once

#include <math.h>
#include <stdint.h>
#include <vector_types.h>

#include "skewadam.h"

namespace skew {

// Every kernel runs 256-thread CTAs; a thread owns 8 consecutive elements (one 16-byte vector of bf16) of
// strip_rows rows (strip tiles), of flat_rounds flat vectors (flat tiles of factored tensors), or of up to
// kFlatVecPerThread (full-second-moment tiles: 8 Ki elements, so that the router and the vectors, small, spread
// over many CTAs).
constexpr int kThreads = 256;
constexpr int kVecPerThread = 32;
constexpr int64_t kFullTile = int64_t(kThreads) * 8 * kVecPerThread;  // elements

// Heights of the tiles of factored tensors off the row path, which hold `strip` elements in a step: where these
// give an SM few tiles, a tile's rounds, one after another, set the time; where they give it many, the tiles' own
// start and the partials they leave do. Measured at 8, 16 and 32 rows (4, 8, 16 and 32 rounds), one matrix without
// momentum: 768 columns 4M elements 29 31 40 us, 8M 44 38 44, 13M 63 59 56, 26M 110 95 94; 4095 columns 2M 33 38 53 72,
// 6M 63 60 63 85, 13M 113 94 98 96, 20M 164 139 135 149, 36M 271 218 189 178; 24 ragged tensors of 13M 114 102 113 125.
// (`vec`: row-vectors of 16 bytes; the others' phase A, too, gains from more tiles. `ride`: in the launches of row
// tiles, which fill what full tiles leave idle: 12M elements beside 60M, 16 and 8: 188 us, full 181; fp32 217 and 205.)
inline int strip_rows(bool vec, bool ride, int64_t strip) {
    return strip < (vec ? 76 : 38) * kFullTile ? 8 : strip < (ride ? 152 : 228) * kFullTile ? 16 : kVecPerThread;
}
inline int flat_rounds(bool ride, int64_t strip) {
    return strip < 38 * kFullTile                     ? 4
           : strip < (ride ? 152 : 228) * kFullTile   ? 8
           : strip < (ride ? 152 : 456) * kFullTile   ? 16 : kVecPerThread;
}
// A step with row tiles runs its strip and flat tiles in their launches while these hold at most
// kRideElems elements: more of them are faster in launches of their own, where four CTAs share an SM
// (1.15B elements of 4864 and 7128 columns beside one 4095 x 1000 matrix: 2316 against 2586 us).
constexpr int64_t kRideElems = int64_t(32) << 20;
constexpr int kFlatVecPerThread = 4;
constexpr int64_t kFlatTileElems = int64_t(kThreads) * kFlatVecPerThread * 8;
// Flat tiles of factored tensors with at most kFlatCols columns: consecutive elements, the scales of all columns
// and of the tile's rows in shared memory; of wider ones: kFlatStrip columns of 2 fvpt rows (as many elements).
constexpr int64_t kFlatCols = 4096;
constexpr int kFlatStrip = 1024;
constexpr int kFinChunk = 256;  // rows / columns per finalize item

// Row-tile path (phase A on whole rows, no phase B unless a clamp may bind):
// a chunk is kRowChunkBytes of consecutive whole rows of the bf16 gradient,
// copied to shared memory by one bulk copy; a phase-A row tile is kRowChunks
// chunks (kRowChunksWide for 4096-wide matrices of at least 2048 rows, whose
// tiles then pay their ring ramp and column partials half as often; shorter
// matrices keep more, smaller tiles, which measured faster); a phase-C row tile
// is always the rows of kRowChunks chunks; the CTA keeps kRowStages chunks in flight.
constexpr int kRowChunkBytes = 32768;
constexpr int kRowChunks = 32;
constexpr int kRowChunksWide = 64;
constexpr int kRowStages = 3;
// Momentum tensors on the row path: a chunk holds kMomGBytes of bf16 rows (G in
// phase A, W in phase C) and the same rows of fp32 M; a row tile is kMomChunks chunks.
// Phase C on the row path: the last kApplyTailSplit tiles of a step (two waves of the
// kernel's two CTAs per SM on GB300's 152 SMs) run as two half tiles each, so that the
// launch's last wave ends sooner. An item's tile field then carries kHalfTile, plus
// kSecondHalf for the second half (results do not depend on the split).
constexpr uint32_t kApplyTailSplit = 2u * 2u * 152u;
constexpr int64_t kSplitTileBytes = 512 << 10;  // smaller tiles (of W) stay whole
constexpr uint32_t kHalfTile = 1u << 31, kSecondHalf = 1u << 30, kTileMask = kSecondHalf - 1u;
constexpr int kMomGBytes = 16384;
constexpr int kMomChunks = 64;

// Row path of the widths m = 8 V in [kAnyMin, kAnyMax] that are not 512, 1024, 2048 or 4096
// (rowsq_gen_tile, apply_flat_tile): rows per thread and phase-A chunk at NV vectors per
// thread and row, and the floats of shared memory that hold phase C's scales.
// Below 128 columns a row fills less than half a warp (20M parameters of a 256-wide model with experts
// of 248 columns: strip tiles below 256 91 us, below 128 72 us), and above 8192 the column sums of a row do
// not fit the registers of one CTA: both stay on the strip tiles. (Above 4096, 16-warp CTAs, one per SM.) Against
// the strip tiles (three reads of G): 930M parameters in 3072 x 1536 experts 1872 -> 1259 us.
enum RowPath : uint32_t { kRowNone = 0, kRowFixed = 1, kRowAny = 2 };
constexpr int64_t kAnyMin = 128, kAnyNarrow = 4096, kAnyMax = 8192;
constexpr int kWideThreads = 512;
constexpr int64_t kAnyTileBytes = 1 << 20;  // bf16 bytes of a tile in phases A and C, as of the fixed widths
constexpr int kFlatBytes = 115072;  // phase C's ring and scales
constexpr int kFlatScales = 4184, kFlatWideScales = 10336;  // scales that fit beside the ring
__host__ __device__ constexpr int gen_rows_per_thread(int nv, bool mom) { return (nv == 1 ? 8 : 4) / (mom ? 2 : 1); }

enum Kind : uint32_t { kKindFull = 0, kKindFactored = 1 };

// Tier policy of one tensor (Sec. 3 "The tiers", Algorithm 1, the Table 3
// variants, and the Adafactor comparator of Sec. 5 / App. A): a vector keeps the exact
// second moment; the router too unless the variant factors it; every other matrix
// is factored (Eq. 1). Momentum: the backbone; experts under "+ momentum on
// experts" and "uniform"; the router under "uniform"; nothing under Adafactor.
// Weight decay: every tier but the router, unless the caller exempts the tensor.
inline void resolve_policy(int ndim, int tier, int policy, uint32_t flags, uint32_t &kind, uint32_t &momentum,
                           uint32_t &decay) {
    const bool router_factored = policy == SKEW_POLICY_FACTORED_ROUTER || policy == SKEW_POLICY_UNIFORM ||
                                 policy == SKEW_POLICY_ADAFACTOR;
    kind = (ndim == 1 || (tier == SKEW_TIER_ROUTER && !router_factored)) ? kKindFull : kKindFactored;
    if (policy == SKEW_POLICY_ADAFACTOR)
        momentum = 0;
    else if (tier == SKEW_TIER_BACKBONE)
        momentum = 1;
    else if (tier == SKEW_TIER_EXPERT)
        momentum = (policy == SKEW_POLICY_EXPERT_MOMENTUM || policy == SKEW_POLICY_UNIFORM);
    else
        momentum = (policy == SKEW_POLICY_UNIFORM);
    decay = (tier != SKEW_TIER_ROUTER) && !(flags & SKEW_F_NO_DECAY);
}

// Second-moment decay (fp32, with 1 - beta2 formed from it in fp64) and the update
// coefficients of step t: sqrt(1 - beta2^t) / (1 - beta1^t) with momentum and
// sqrt(1 - beta2^t) without (Algorithm 1's bias corrections). The Adafactor
// comparator anneals the decay, beta2_t = 1 - t^-0.8, and has no bias correction.
struct StepCoefs {
    float b2, c2;
    double coef_mom, coef_plain;
};

inline StepCoefs step_coefs(const skew_hparams_t &H, int64_t step) {
    const double t = (double)step;
    StepCoefs c;
    if (H.policy == SKEW_POLICY_ADAFACTOR) {
        c.b2 = (float)(1.0 - pow(t, -0.8));
        c.c2 = (float)(1.0 - (double)c.b2);
        c.coef_mom = c.coef_plain = 1.0;
    } else {
        const double s2 = sqrt(1.0 - pow((double)H.beta2, t));
        c.b2 = H.beta2;
        c.c2 = (float)(1.0 - (double)H.beta2);
        c.coef_mom = s2 / (1.0 - pow((double)H.beta1, t));
        c.coef_plain = s2;
    }
    return c;
}

// Tile geometry of one tensor (shared by every entry point, so that the same
// tensor is always cut the same way and results are bit-identical).
struct TileGeom {
    uint32_t lcl = 0, strips = 1, rowtiles = 1, tile_rows = 0, ntiles = 0, nfr = 0, nfc = 0;
    uint32_t nbc = 0, fvpt = 0;  // tiles of phases B and C; vectors per thread of a flat tile
    uint32_t rowpath = 0, cr = 0, rt_rows = 0, rtiles = 0;
    uint32_t at_rows = 0, atiles = 0;  // row path: phase-C row tiles
    uint32_t fci = 0;  // columns per finalize item (kFinChunk / fci threads per column)
};

// Phase C takes the matrices in the reverse of phase A's order, so that it starts with the G (with
// momentum the M) that phase A read (wrote) last, and phase A asks L2 to keep the last kKeepBytes of it
// (the L2 holds 126 MB, and R, W and the partials pass through it meanwhile), in steps whose phase C
// reads kKeepTotal bytes or more again: the 6.78B set 8316 -> 8215 us (k_apply_rows 5862 -> 5765: more
// than the kept bytes, so the rest of its stream gains too), one MoE layer 2088 -> 2066; without the hint
// 8295 and 2086. Smaller steps lose by the hint what else the L2 would hold for them (65M parameters in
// 768 x 488 experts 161 -> 168 us with it).
constexpr int64_t kKeepBytes = int64_t(64) << 20, kKeepTotal = int64_t(256) << 20;

constexpr int64_t kWholeGroup = int64_t(1) << 60;  // as `rest`: full-sized tiles

// Chunks (of `chunk` bytes) in the row tiles of a matrix of `own` bytes when the step's row-path
// matrices from it on, in launch order, hold `rest` bytes: `most` while that gives `waves` waves of
// two CTAs on each of the 152 SMs or more, then ever smaller tiles, so that the launch's last tiles
// end together and a small step still fills the chip, down to `least`. 680M parameters with momentum
// on the experts 1960 -> 1881 us (k_rowsq 1080 -> 1021, k_apply_rows 811 -> 775 us); 850M without
// 1205 -> 1172 us (k_rowsq 350 -> 321); the 6.78B set 8377 -> 8358. Phase A takes one wave without
// momentum (a second one costs the finalize more partials than it saves: k_rowsq 331, not 321) and
// two with it, phase C three. `parts`: tiles a matrix may have before its column partials would outgrow the
// no-alloc scratch; it then keeps to one wave of tiles, up to twice `most` each.
// (Tiles below kWaveTileBytes come in one wave, which saves the second wave's ramps: k_apply_rows of
// 118M parameters in 816 x 408 experts 162 -> 149 us.)
constexpr int64_t kWaveTileBytes = 128 << 10;
inline uint32_t row_tile_chunks(int64_t own, int64_t rest, int64_t waves, int64_t chunk, int64_t least, int64_t most,
                                int64_t parts) {
    const int64_t ctas = 2 * 152;
    auto per = [chunk](int64_t bytes, int64_t tiles) { return (bytes + tiles * chunk - 1) / (tiles * chunk); };
    int64_t t = per(rest, ctas), whole = kWaveTileBytes / chunk;  // a single wave of small tiles: no second ramp
    if (t > whole) t = per(rest, ctas * waves) > whole ? per(rest, ctas * waves) : whole;
    t = t < least ? least : t > most ? most : t;
    if (parts && rest < kWholeGroup && own > t * chunk * parts && own <= 2 * most * chunk * ctas) t = per(own, parts < ctas ? parts : ctas);
    return (uint32_t)t;
}

// Below this many bytes of G in all row-path matrices, those that only kRowAny serves take strip tiles: beside
// larger row tiles a 4095 x 1000 matrix of 8 MB costs 43 us more there, but alone the second read of G (much of it
// from L2) costs a step little. One matrix, strip and row tiles: 2048 x 1408 27 and 32 us, 768 columns of 16 MiB of G
// 37 and 40, 32 MiB 59 and 51, 52 MiB 91 and 73; with momentum 16 MiB 52 and 46, 32 MiB 79 and 69. Models of 256
// columns, most of it the embedding's: 20 MiB 67 and 57, 42 MiB 104 and 78; all matrices queued for phase B (below):
// 68 and 83, 107 and 116.
constexpr int64_t kAnyGroupBytes = 32 << 20;
// An eps that the clamp may bind at (kBindEps: a row's or column's mean g^2 of 1e-12 is g = 1e-6) can queue
// matrices for k_fallback, which reads them again, M included; a step of these widths alone then takes row tiles
// from twice that on. What binds is eps against g^2, which no plan knows: 768 columns, strip and row tiles, in MiB of G,
// where all is queued 32: 60 and 69 us, 52: 95 and 99, 68: 104 and 112, 100: 150 and 149, 180: 231 and 216 (momentum 82
// and 88, 132 and 158, 142 and 176, 208 and 239, 333 and 372); where the clamp does not bind 59 and 51, 91 and 73, 100
// and 80, 146 and 102, 225 and 158 (79 and 69, 129 and 118, 141 and 133, 206 and 177, 329 and 291). Where it binds in
// the first steps only, or the clip factor is provably 1, the latter holds for most of a run.
constexpr int64_t kAnyBindBytes = 64 << 20;
constexpr float kBindEps = 1e-12f;
// Beside row tiles of other widths, those above kAnyNarrow need a launch of their own, and below this
// many bytes of G the strip tiles, which ride along, are faster (260M parameters, 23 MB of them 5632
// wide: 379 us against 407; 1.16B parameters of 4864 and 7128 columns: 2314 against 1653). 5632 columns alone, as
// above: not bound 32 MiB 58 and 57, 68 MiB 104 and 93 (momentum 79 and 78, 143 and 140), queued 60 and 76, 108 and 139
// (82 and 100, 145 and 196); with momentum 7168 columns and more gain nothing to 100 MiB (8192: 80 and 91 at 32 MiB).
constexpr int64_t kWideGroupBytes = 64 << 20;

// Which widths that only kRowAny serves take row tiles in a step: `narrow` and `wide` bytes of G of its
// matrices up to and above kAnyNarrow columns, `fixed`: of those of the fixed widths; `eps`: the clamp's.
struct AnyWidths {
    bool narrow, wide;
};
inline AnyWidths any_widths(int64_t narrow, int64_t wide, int64_t fixed, float eps) {
    const int64_t least = fixed < kAnyGroupBytes && eps > kBindEps ? kAnyBindBytes : kAnyGroupBytes;
    AnyWidths w;
    w.wide = wide >= kWideGroupBytes || (fixed == 0 && narrow < least && wide >= least);
    w.narrow = narrow > 0 && (narrow + fixed >= least || w.wide);
    return w;
}

// `kind`, `momentum` as resolved by the tier policy; `wg_aligned`: weight and
// gradient pointers are 16-byte aligned; `vec`: row-vectors may be 16-byte accesses (row_vectors);
// `strip`: elements of the step's factored tensors off the row path, `ride`: whether in the row tiles' launches; `rest`, `rest_c`: bytes of G of the step's
// row-path matrices from this one on in phase A's order and in phase C's. Counts fit 32 bits for n, m <= 2^40
// and n*m <= 2^62 only when the caller has checked the tile count (planner).
inline TileGeom plan_geometry(uint32_t kind, uint32_t momentum, bool wg_aligned, bool vec, bool ride, int64_t strip, int64_t n,
                              int64_t m, int64_t numel, int64_t rest, int64_t rest_c) {
    TileGeom g;
    if (kind == kKindFactored) {
        const int64_t vecs = (m + 7) / 8;  // 8-column groups per row
        uint32_t lc = 1;
        while (lc < 32 && lc < vecs) {
            lc <<= 1;
            ++g.lcl;
        }
        g.strips = (uint32_t)((m + 8 * lc - 1) / (8 * lc));
        g.tile_rows = (uint32_t)(strip_rows(vec, ride, strip) * (kThreads / lc));
        g.rowtiles = (uint32_t)((n + g.tile_rows - 1) / g.tile_rows);
        g.ntiles = g.strips * g.rowtiles;
        g.nfc = (uint32_t)((m + kFinChunk - 1) / kFinChunk);
        // Whole-row phases A and C: factored matrices of width 512, 1024, 2048
        // or 4096 (64 to 512 16-byte vectors per row), with or without momentum, and
        // (kRowAny) every other multiple of 8 between kAnyMin and kAnyMax.
        const bool fixed = m == 512 || m == 1024 || m == 2048 || m == 4096;
        g.rowpath = !wg_aligned ? kRowNone
                    : fixed     ? kRowFixed
                    : (m % 8 == 0 && m >= kAnyMin && m <= kAnyMax) ? kRowAny : kRowNone;
        if (g.rowpath) {
            const int64_t own = 2 * numel;
            if (g.rowpath == kRowFixed) {
                const int64_t chunk = momentum ? kMomGBytes : kRowChunkBytes;
                g.cr = (uint32_t)(chunk / (2 * m));
                const int64_t most = momentum ? kMomChunks : m == 4096 && n >= 2048 ? kRowChunksWide : kRowChunks;
                g.rt_rows = g.cr * row_tile_chunks(own, rest, momentum ? 2 : 1, chunk, 65536 / chunk, most, (12 << 20) / (8 * m));
                const uint32_t at = row_tile_chunks(own, rest_c, 3, chunk, 32768 / chunk, (1 << 20) / chunk, 0);
                g.at_rows = g.cr * (momentum ? (at + 1) / 2 * 2 : at);  // a half tile is whole phase-C chunks
            } else {
                const int nv = m > 2048 ? 2 : 1, warps = m > kAnyNarrow ? 16 : 8;
                const int64_t wpr = (m / 8 + 32 * nv - 1) / (32 * nv);
                g.cr = (uint32_t)(gen_rows_per_thread(nv, momentum != 0) * (warps / wpr));
                const int64_t chunk = 2 * m * g.cr, least = 65536 / chunk;
                g.rt_rows = g.cr * row_tile_chunks(own, rest, momentum ? 2 : 1, chunk, least < 1 ? 1 : least,
                                                   (warps / 8) * kAnyTileBytes / chunk,
                                                   (12 << 20) / (8 * m));
                int64_t at = 2 * row_tile_chunks(own, rest_c, 3, 4 * m, (32768 + 4 * m - 1) / (4 * m), kAnyTileBytes / (4 * m), 0);
                const int64_t fit = (m > kAnyNarrow ? kFlatWideScales : kFlatScales) - m;
                if (at > fit) at = fit;
                g.at_rows = (uint32_t)(at / 2 * 2);
            }
            g.rtiles = (uint32_t)((n + g.rt_rows - 1) / g.rt_rows);
            g.atiles = (uint32_t)((n + g.at_rows - 1) / g.at_rows);
            g.nfr = 0;
            // tall matrices: up to 8 threads share a column, each adding every 8th tile
            uint32_t tpc = 1;
            while (tpc < 8 && g.rtiles >= 64u * tpc) tpc <<= 1;
            g.fci = (uint32_t)(kFinChunk / tpc);
            g.nfc = (uint32_t)((m + g.fci - 1) / g.fci);
        } else {
            g.nfr = (uint32_t)((n + kFinChunk - 1) / kFinChunk);
            // tall matrices: up to 32 threads share a column (one adds 8 tiles per trip to L2)
            uint32_t tpc = 1;
            while (tpc < 32 && g.rowtiles > 32u * tpc) tpc <<= 1;
            g.fci = (uint32_t)(kFinChunk / tpc);
            g.nfc = (uint32_t)((m + g.fci - 1) / g.fci);
        }
        g.nbc = g.ntiles;
        if (!g.rowpath && !vec) {
            // (with more rounds a tile of a matrix of fewer than 8 columns has more rows than room for their scales)
            g.fvpt = (uint32_t)flat_rounds(ride, strip);
            if (m < 8 && g.fvpt > kFlatVecPerThread * m) g.fvpt = (uint32_t)(kFlatVecPerThread * m);
            const int64_t tile = int64_t(kThreads) * 8 * g.fvpt;
            g.nbc = (uint32_t)(m > kFlatCols ? ((m + kFlatStrip - 1) / kFlatStrip) * ((n + 2 * g.fvpt - 1) / (2 * g.fvpt))
                                             : (numel + tile - 1) / tile);
        }
    } else {
        // one round per thread spreads a small tensor over more CTAs
        g.fvpt = numel < 2 * 152 * kFlatTileElems ? 1 : kFlatVecPerThread;
        const int64_t tile = int64_t(kThreads) * 8 * g.fvpt;
        g.rowtiles = (uint32_t)((numel + tile - 1) / tile);
        g.ntiles = g.nbc = g.rowtiles;
    }
    return g;
}

// Whether a factored tensor's row-vectors may be 16-byte accesses: bf16, every row of W, G and M on
// a 16-byte boundary.
inline bool row_vectors(bool f32, bool wg_aligned, bool m_aligned, int64_t m) {
    return !f32 && wg_aligned && m_aligned && m % 8 == 0;
}

// Entries of a tensor's sums of U^2.
inline uint32_t u2_len(const TileGeom &g) {
    return g.rowpath && 2 * g.atiles > g.nbc ? 2 * g.atiles : g.nbc;
}

// Where a row-path tensor whose clamp may bind gets its sum(U^2): phase B, or phase C (clip factor 1).
enum SumWhere : uint32_t { kPhaseB = 1, kSumInC = 2 };

// Device descriptor of one tensor (lives in the workspace).
struct TensorDev {
    uint16_t *w;        // bf16 weights, n*m, row-major (borrowed)
    const uint16_t *g;  // bf16 gradient (borrowed)
    float *M;           // momentum (numel) or null
    float *v;           // exact second moment (numel) or null
    float *R;           // row factor (n) or null
    float *C;           // column factor (m) or null
    float *rowp;        // strip path: row partials [strips][n]
    float *colp;        // strip path: column partials of g^2 [rowtiles][m]
    float *bsc;         // factored: 1/sqrt(C_j) [m]
    double *rsum;       // factored: sums of R per finalize-row item [nfr] / per row tile [rtiles]
    float2 *pp;         // row path: per row tile and column, (sum of g^2, sum of g^2 / R_i) [rtiles][m];
                        // then an item's sum of g^2 in the first entry of its columns
    float *rmin;        // row path: smallest positive R_i per row tile [rtiles]
    double *fsum;       // row path: sum of P_j / C_j per finalize item [nfc]
    float *fmin;        // row path: smallest C_j with P_j > 0 per finalize item [nfc]
    float2 *u2;         // sums of (U / coef)^2 as (hi, lo) pairs: per phase-B tile [nbc], or on the
                        // row path per half of a phase-C tile [2 atiles] (u2_len)
    int64_t n, m, numel;
    double inv_n, inv_numel;  // 1 / n, 1 / numel
    uint32_t tid;       // dither tensor id
    uint64_t base;      // dither index of element 0 (a matrix of a stacked tensor: its offset)
    uint32_t kind, momentum, decay;
    uint32_t vec;       // 1: 16-byte vector loads / stores are legal (bf16 tensors only)
    uint32_t wal, sal;  // 1: w and g (M and v) start on 16-byte boundaries
    uint32_t f32;       // 1: weights and gradient are fp32 (w, g then address floats; no dither)
    uint32_t lcl;       // factored: log2 of lanes along a row (LC)
    uint32_t strips;    // factored: column strips of 8*LC columns
    uint32_t rowtiles;  // factored: row tiles of tile_rows rows; full: flat tiles
    uint32_t tile_rows; // factored: rows per strip tile (strip_rows times its row groups)
    uint32_t ntiles;    // strip tiles (full: flat tiles) of this tensor
    uint32_t nbc, fvpt; // tiles of phases B and C; vectors per thread of a flat tile
    uint32_t nfr, nfc;  // factored: finalize items over rows / columns
    uint32_t rowpath;   // RowPath; nonzero: whole-row phase A (k_rowsq) and the bilinear sum of U^2
    uint32_t cr;        // row path: rows per chunk
    uint32_t rt_rows;   // row path: rows per phase-A row tile
    uint32_t rtiles;    // row path: phase-A row tiles
    uint32_t fci;       // columns per finalize item
    uint32_t at_rows;   // row path: rows per phase-C row tile (<= 1024 at the fixed widths)
    uint32_t atiles;    // row path: phase-C row tiles
    uint32_t keep;      // row path: phase C finds this G in L2 if phase A leaves it there
    uint32_t srows;     // k_small: rows (full: elements, m = 1) of a CTA's slice
};

// Per-tensor scalars of the current step (zeroed at the start of every step).
struct TensorScal {
    double rbar;        // mean(R)
    double sumsq;       // sum over the tensor of U^2
    double rms;         // RMS(U)
    double kappa;       // 1 / max(1, RMS / d)
    float rbar_s;       // mean(R) * 2^rbar_e, in [1, 2); 0 if mean(R) == 0
    int32_t rbar_e;
    float coefC;        // lr * kappa * coef, the factor applied to (y / D)
    uint32_t cntF;      // finalize items done
    uint32_t cntB;      // update-RMS tiles done
    uint32_t fallback;  // row path, when a clamp may bind: SumWhere of sum(U^2); else 0
    uint32_t zflag;     // row path: a row with R_i == 0 holds a nonzero gradient
    uint32_t pad;
};
static_assert(sizeof(TensorScal) == 64, "TensorScal layout");

// Per-step parameters, passed by value to every kernel (a kernel parameter).
struct StepArgs {
    const TensorDev *tensors;  // null: the one tensor `one` (the no-alloc step)
    TensorDev one;
    TensorScal *scal;
    uint32_t *err;         // sticky status word (nonzero: a bounded wait gave up)
    uint32_t *fb;          // [0]: row-path tensors that need phase B, [1..]: their ids
    float b1, b2, c1, c2;  // beta1, beta2, 1-beta1, 1-beta2 (fp32)
    float ce;              // 1 / sqrt(eps), fp32
    float wdf;             // 1 - lr * lambda, fp32
    float lr;
    float clip_d;
    double coef_mom;       // sqrt(1-beta2^t) / (1-beta1^t)
    double coef_plain;     // sqrt(1-beta2^t)
    uint32_t step_lo;
    uint32_t seed_lo, seed_hi;
    const float *gscale;   // device pointer to the step's gradient scale gamma (the trainer's
                           // global-norm clip factor), or null for gamma = 1
};

// The phases of one step: item lists (tensor, local tile / item) in device
// memory and their lengths.
//   A  strip-tile sums of squares (strip-path factored tensors); when riding, also
//      the update-RMS tiles of full tensors
//   R  row-tile sums of squares and bilinear partials (row-path tensors)
//   F  finalize items (rows and columns; columns only on the row path)
//   B  update-RMS tiles (strip-path factored tensors; unless riding, full tensors too)
//   FB phase B of the row-path tensors whose finalize asked for it (nFB CTAs)
//   C  apply strip and flat tiles (tensors not on the row path)
//   CR apply row tiles (row-path tensors)
// A null table stands for tensor 0's tiles in order. The items of R follow those of A, and those of CR those of C; `ride`: A, B and C go into the launches
// of the row tiles (R, FB and CR).
struct LaunchPlan {
    uint32_t nA, nR, nF, nB, nFB, nC, nCR;
    uint32_t nRW;  // of the nR, those of widths above kAnyNarrow (last)
    bool ride;
    const uint2 *itemsA, *itemsF, *itemsB, *itemsC;
};

// Enqueues the clearing of the per-step scalars and of the phase-B queue's length at `p` (a multiple of
// 4 bytes). Returns a cudaError_t value.
int launch_reset(void *p, size_t bytes, void *stream);

constexpr int kLaunches = 7;  // kernels a step may launch in turn

// A step of small tensors only runs as one launch, a cluster of `ctas` CTAs per tensor (k_small).
constexpr int kSmallThreads = 512;
constexpr size_t kSmallHeadBytes = 4096;                     // fixed part of its shared memory
constexpr size_t kSmallSmem = 224 * 1024;                    // most that it takes
constexpr size_t kSmallHalf = 112 * 1024;                    // up to which an SM holds two CTAs
constexpr int64_t kSmallCtas = 256;                          // CTAs of a launch
struct SmallPlan {
    uint32_t ctas = 0;  // 0: not a step for k_small
    size_t smem = 0;
};

// Rows (elements of a full tensor, stepped as n x 1) of a CTA's slice, a multiple of 8 so that a slice
// starts on a Philox block and a 16-byte boundary where the tensor does.
inline int64_t small_rows(int64_t n, uint32_t ctas) { return ((n + ctas - 1) / ctas + 7) / 8 * 8; }

// Shared memory of one CTA's slice: its elements, row scales and twice the columns as fp32.
inline int64_t small_bytes(int64_t n, int64_t m, uint32_t ctas) {
    const int64_t rows = small_rows(n, ctas);
    return (int64_t)kSmallHeadBytes + 4 * (rows * m + rows + 2 * m);
}

// Adds one tensor (full: n = numel, m = 1) to the plan of a step over `tensors` of them: the fewest CTAs
// whose shared memory holds a slice, in clusters of at most 8.
inline bool small_fits(int64_t n, int64_t m, uint32_t ctas) {
    return n <= (int64_t(1) << 22) && m <= (int64_t(1) << 16) && small_bytes(n, m, ctas) <= (int64_t)kSmallSmem;
}

// The rule: every tensor of the step fits, with at most kSmallCtas CTAs in all (two waves at one CTA per
// SM, one at two): beyond, the strip tiles' four launches are as fast. Slices are then halved while that
// holds: the toy MoE's 39 tensors take 21 us in clusters of two, 17 in clusters of four. `vec`: matrices with 16-byte
// row-vectors hold more than half of the elements. Their strip tiles are fast, so that slices too large for two CTAs
// on an SM lose to them, unless one wave of small clusters holds all (48 matrices of 256 x 776 bf16 81 us so, 51 in
// four launches; 16 of 640 x 640 79 and 35; 76 of 256 x 256, clusters of two, 30 and 30, with momentum 35 and 38).
// Tensors without row-vectors gain up to the full room (64 of 256 x 776 fp32 86 and 94, 128 of 200 x 333 bf16 64 and 74).
template <typename Each>
inline SmallPlan plan_small(int64_t tensors, bool vec, Each each) {
    SmallPlan P;
    if (tensors < 1 || tensors > kSmallCtas) return P;
    auto fits = [&](uint32_t c) { return each([c](int64_t n, int64_t m) { return small_fits(n, m, c); }); };
    uint32_t c = 1;
    while (c <= 8 && !fits(c)) c *= 2;
    if (c > 8 || tensors * c > kSmallCtas) return P;
    // smaller slices, while they still hold 4 elements per thread
    while (c < 8 && tensors * c * 2 <= kSmallCtas &&
           !each([c](int64_t n, int64_t m) { return small_rows(n, 2 * c) * m < 4 * kSmallThreads; }))
        c *= 2;
    int64_t most = 0;
    each([&](int64_t n, int64_t m) {
        const int64_t b = small_bytes(n, m, c);
        most = b > most ? b : most;
        return true;
    });
    if (vec && most > (int64_t)kSmallHalf && (c > 2 || tensors * c > 152)) return P;
    P.ctas = c;
    P.smem = size_t(most);
    return P;
}

// Enqueues the step of `tensors` small tensors as one launch; `ev` as for launch_phases (its time is that
// of the last place). Returns a cudaError_t value.
int launch_small(const StepArgs &A, uint32_t tensors, const SmallPlan &P, void *stream, void *const *ev);


// Enqueues the phases of `L` as grouped launches (A, F, B, C; with row tiles A + R, F,
// B + FB, C + CR; empty ones skipped) on `stream`, each given the step parameters by value. If `ev` is
// not null it holds kLaunches + 1 cudaEvent_t, recorded before the first launch and after
// each of the seven kernels' places (k_sumsq, k_rowsq, k_finalize, k_rms, k_fallback, k_apply,
// k_apply_rows). Returns a cudaError_t value.
int launch_phases(const StepArgs &A, const LaunchPlan &L, void *stream, void *const *ev);

// Enqueues the bounded-wait self-test (one thread waits on an mbarrier phase that
// never completes and records the timeout in *err). Returns a cudaError_t value.
int launch_wait_selftest(uint32_t *err, void *stream);

}  // namespace skew
