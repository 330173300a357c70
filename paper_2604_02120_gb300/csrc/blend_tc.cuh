// Tensor-core blending (Alg. 2, Eqs. 4-8) for sm_100-family GPUs.
//
// Persistent kernel: each CTA pulls tiles from a global queue (an atomic
// counter) until the queue is empty; the tiles of all views of the call form
// one queue.  Every 16 x 16 tile is split into an upper and a lower 16 x 8
// half; M_p (A operand, 128 x K) holds the monomials
// [xb^2, yb^2, xb yb, xb, yb, 1] of the 128 pixels of a half relative to the
// half's reference pixel and is built once per CTA.  For every chunk of CH
// splats of a tile the builder writes 2 CH coefficient rows v_g (Eq. 6):
// rows [0, CH) referred to the upper half's reference, rows [CH, 2 CH) to the
// lower half's (8 pixels further down).  One tcgen05.mma (M = 128, N = 2 CH,
// K = 16 or 32) then leaves in TMEM lane r, column j the exponent of splat j
// at upper pixel r and, at column CH + j, at lower pixel r: each epilogue
// thread owns two pixels of one lane and composites both with packed f32x2
// arithmetic.
//
// Warps: 0-3 epilogue (warp w reads TMEM lanes 32 w .. 32 w + 31; it holds an
// 8 x 4 pixel block of each half, lane_col / lane_row), 4 scanner, 5 row
// builder, MMA issue (lane 0) and TMEM owner.
//  - The scanner walks the tiles of the queue and their lists in groups of 32
//    entries, copies the splats a group ahead by cp.async (or by TMA gathers
//    of packed records), drops the entries whose alpha stays below 1/255 on
//    the whole tile (splat_reaches) and packs the others, with their list
//    positions, into chunks of CH raw splats, raw_slots ahead.
//  - The builder turns a raw chunk into a stage of the shared-memory ring
//    (SS stages: header, v_g rows, per-splat colour and position), issues its
//    MMA into one of 2 TMEM stages and drops the chunks of a tile whose pixels
//    have all stopped meanwhile.
// Both run across tile boundaries, so the next tile's lookups and gathers
// overlap the current tile's compositing.  An empty tile travels as one stage
// with n = 0, the end of the queue as n = -1.
//
// Why the lists are culled here: with full 3-sigma rectangles 50 to 72% of a
// tile's entries reach none of its pixels, and an entry dropped costs the
// scanner about 2 instructions per epilogue warp, one kept 29 (the kernel runs
// at 62 to 71% of the issue slots).  1920 x 1080, 1M clustered splats, full
// rectangles: 0.828 -> 0.339 ms; 1280 x 720, 200k: 0.119 -> 0.079 ms; 256 x 256,
// 10k: 0.036 -> 0.028 ms; opacity-aware lists, where every entry is kept:
// 0.286 -> 0.273 ms (1920 x 1080), 0.482 -> 0.470 ms (3840 x 2160, 3M).
// Skipping splats per warp (a vote on the exponents) was measured as well: 5%
// faster on those full lists, 15% slower at 3840 x 2160, where most splats
// reach most warps and the branch costs the overlap of neighbouring splats.
// All waits are bounded by opts.timeout_ns; on expiry the CTA records
// GS_ERR_TIMEOUT in the device error word, every role leaves its loop, the
// MMA thread commits to a drain barrier of its own and waits (bounded, 1 s)
// until every MMA it issued has completed; then TMEM is freed.
//
// Compositing without branches (per pixel, alpha already clamped):
//   cull = sat((1/255 - alpha) 2^36)        1 iff alpha < 1/255 (exact: one rounding)
//   a    = alpha - alpha cull
//   T'   = T - a T;  stop = sat((1e-4 - T') 2^40)   1 iff T' < 1e-4
//   T_stop += T stop;  a2 = a - a stop;  w = a2 T;  T = T' - T' stop
//   C += c w;  used = sat(a2 2^36);  last += used (index + 1 - last)
// A pixel that stops keeps T = 0 from then on (so it never contributes
// again, and T' = 0 keeps `stop` at 1 while T_stop stays put); T_final =
// T + T_stop.  Pixels outside the image start with T = 0.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "internal.h"

namespace gs {
namespace tc {

constexpr int kEpiWarps = 4;
constexpr int kThreads = 192;  // 4 epilogue warps, scanner, row builder
constexpr int kTStages = 2;
constexpr int kDoneRing = 16;  // tiles in flight between scanner and epilogue < kDoneRing
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kTMin = 1e-4f;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLog2AlphaMin = -7.9943534368588578f;    // log2(1/255)
constexpr float kLog2AlphaMax = -0.014499569695115089f;  // log2(0.99)
constexpr float kDeadPower = -200.0f;
constexpr float kCullScale = 68719476736.0f;    // 2^36
constexpr float kStopScale = 1099511627776.0f;  // 2^40

// Operand encoding of a variant.  K elements of a row: TERMS operand-type terms
// of v_g times PTERMS terms of the monomials, 6 each (every product of a v_g
// term with a monomial term gets its own K slot), zero-padded.  FP8: e4m3
// operands (tcgen05 kind::f8f6f4), each v_g row scaled by a power of two so
// that its largest coefficient lies in [128, 256), the monomials split into 2
// exact terms.
template <int V>
struct Traits {
    // CC: the exponent v_g . v_p by FP32 FMAs on the CUDA cores; the B stage
    // then holds each splat's two FP32 rows (12 floats) and no MMA runs
    static constexpr bool CC = (V == GS_BLEND_PERSISTENT_FP32);
    static constexpr bool FP8 = (V == GS_BLEND_TC_FP8_SPLIT);
    static constexpr int TERMS = FP8 ? 5 : (V == GS_BLEND_TC_FP16_SPLIT) ? 2 : (V == GS_BLEND_TC_BF16_SPLIT ? 3 : 1);
    static constexpr int PTERMS = FP8 ? 2 : 1;
    static constexpr int K = FP8 ? 64 : (V == GS_BLEND_TC_BF16_SPLIT) ? 32 : 16;
    static constexpr uint32_t FMT = (V == GS_BLEND_TC_BF16 || V == GS_BLEND_TC_BF16_SPLIT) ? 1u : 0u;  // e4m3: 0
    static constexpr bool HALF = (FMT == 0);
    static constexpr int ROW_BYTES = FP8 ? K : 2 * K;
    static constexpr int KSTEPS = ROW_BYTES / 32;               // one MMA consumes 32 bytes of every row
    static constexpr int SBO = (ROW_BYTES / 16) * 128;          // bytes between 8-row core-matrix groups
    static_assert(6 * TERMS * PTERMS <= K, "operand terms exceed K");
};

// FP8 term t of v_g is stored multiplied by 2^kFp8Shift[t] and the monomial
// slots it meets by 2^-kFp8Shift[t] (products unchanged): the small terms move
// up into e4m3's normal range, the monomials (>= 1/4) stay normal.
__device__ __forceinline__ float fp8_term_shift(int t) { return t >= 2 ? 16.0f : 1.0f; }

// e4m3 encoding (round to nearest, saturating) and its value
__device__ __forceinline__ uint8_t to_e4m3(float x) {
    return (uint8_t)__nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3);
}
__device__ __forceinline__ float from_e4m3(uint8_t b) {
    const __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)b, __NV_E4M3);
    return __half2float(__half(h));
}

template <bool HALF>
__device__ __forceinline__ uint16_t to_op(float x) {
    if constexpr (HALF) return __half_as_ushort(__float2half_rn(x));
    else return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}
template <bool HALF>
__device__ __forceinline__ float from_op(uint16_t b) {
    if constexpr (HALF) return __half2float(__ushort_as_half(b));
    else return __bfloat162float(__ushort_as_bfloat16(b));
}

// Per-splat record of the fused small-scene kernel: colour
// duplicated for both pixels of a lane and the exponent ceiling min(log2 0.99, log2 o).
// (The forward's epilogue reads (r, g, b, cap) as one float4: a warp-wide broadcast
// of 16 bytes costs four cycles of the SM's shared-memory pipe.)
struct alignas(16) Rec {
    float4 rg;  // r, r, g, g
    float4 bc;  // b, b, cap, cap
};

// Pixel of accumulator lane r within a 16 x 8 half: warp r / 32 holds an 8 x 4
// block (of both halves), so that the pixels a small splat reaches fall into
// few warps.
__host__ __device__ __forceinline__ int lane_col(int r) { return ((r >> 5) & 1) * 8 + (r & 7); }
__host__ __device__ __forceinline__ int lane_row(int r) { return (r >> 6) * 4 + ((r >> 3) & 3); }

// tcgen05.mma of the variant's operand kind (f16/bf16 or e4m3)
template <int V>
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
    if constexpr (Traits<V>::FP8)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    else
        tc_mma_f16(d_tmem, adesc, bdesc, idesc, accumulate);
}

// Chunks of raw splats between the scanner and the row builder.  Two keep the
// epilogue fed where most entries are dropped (one: 1920 x 1080, full lists 343 ->
// 356 us).  The CUDA-core variant's epilogue takes longer per splat, and what the
// scanner takes past a tile's end costs it more: one there (3840 x 2160, 3M,
// opacity-aware lists 611 -> 597 us, full lists the same).
template <int V>
constexpr int raw_slots() {
    return Traits<V>::CC ? 1 : 2;
}
constexpr int kRawFields = 10;  // mean x, y, conic A, B, C, log2 opacity, r, g, b, list position + 1
constexpr int kGroup = 32;      // list entries the scanner tests at a time
constexpr int kGeoFields = 9;   // mean (2), conic (3), opacity, colour (3)
constexpr int kGeoSlots = 4;    // groups of splats copied ahead: two of the current tile, two first ones of a tile
constexpr int kRecSlots = 4;    // TMA slots of a group's records

template <int SS, int CH, int V>
struct Layout {
    static constexpr int RAW = raw_slots<V>();
    static constexpr int A_BYTES = 128 * Traits<V>::ROW_BYTES;
    static constexpr int B_BYTES = 2 * CH * Traits<V>::ROW_BYTES;
    static constexpr int OFF_B = A_BYTES;
    static constexpr int OFF_REC = OFF_B + SS * B_BYTES;
    static constexpr int OFF_IDX = OFF_REC + SS * CH * 16;   // list positions + 1 (floats)
    static constexpr int OFF_SCL = OFF_IDX + SS * CH * 4;    // FP8: row scales (float2 per splat)
    static constexpr int OFF_RAW = OFF_SCL + (Traits<V>::FP8 ? SS * CH * 8 : 0);
    static constexpr int OFF_RECT =
        (OFF_RAW + RAW * kRawFields * CH * 4 + 255) / 256 * 256;  // TMA record slots (256-aligned)
    static constexpr int OFF_GEO = OFF_RECT;  // the same memory: a launch uses one or the other
    static_assert(kGeoSlots * kGeoFields * 4 <= kRecSlots * kRecBytes, "splat slots");
    static constexpr int OFF_BAR = OFF_RECT + kRecSlots * kGroup * kRecBytes;
    // full[SS], empty[SS], tfull, tempty, drain, raw full, raw empty, record slots
    static constexpr int NBAR = 2 * SS + 2 * kTStages + 1 + 2 * RAW + kRecSlots;
    static constexpr int OFF_HDR = OFF_BAR + NBAR * 8;
    static constexpr int OFF_RAWHDR = OFF_HDR + SS * 32;
    static constexpr int OFF_MISC = OFF_RAWHDR + RAW * 32;
    static constexpr int BYTES = OFF_MISC + 16 + 4 * kDoneRing;
    static constexpr uint32_t TCOLS_RAW = 2u * kTStages * CH;
    static constexpr uint32_t TCOLS = TCOLS_RAW <= 32 ? 32 : TCOLS_RAW <= 64 ? 64 : TCOLS_RAW <= 128 ? 128
                                      : TCOLS_RAW <= 256 ? 256 : 512;
    static_assert(TCOLS_RAW <= 512, "TMEM stages exceed 512 columns");
    static_assert(CH % 16 == 0 && 2 * CH <= 256, "chunk must be a multiple of 16 and at most 128");
};

// Store 8 consecutive K elements (one 16-byte core-matrix row) of row r.
template <int V>
__device__ __forceinline__ void store_row_chunk(uint8_t* mat, int r, int kc, const uint16_t (&e)[8]) {
    uint4 u;
    u.x = (uint32_t)e[0] | ((uint32_t)e[1] << 16);
    u.y = (uint32_t)e[2] | ((uint32_t)e[3] << 16);
    u.z = (uint32_t)e[4] | ((uint32_t)e[5] << 16);
    u.w = (uint32_t)e[6] | ((uint32_t)e[7] << 16);
    *reinterpret_cast<uint4*>(mat + (r >> 3) * Traits<V>::SBO + kc * 128 + (r & 7) * 16) = u;
}

// Maximum of q(d) = -1/2 d^T [[A, B], [B, C]] d over the box [bx0, bx1] x [by0, by1].
__device__ __forceinline__ float box_max_quadratic(float A, float B, float C, float bx0, float bx1, float by0,
                                                   float by1) {
    if (!(A > 0.f) || !(C > 0.f)) return 0.f;  // not positive definite: never skipped
    if (bx0 <= 0.f && bx1 >= 0.f && by0 <= 0.f && by1 >= 0.f) return 0.f;
    float best = -INFINITY;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float ex = e ? bx1 : bx0;
        const float dy = fminf(fmaxf(-B * ex / C, by0), by1);
        best = fmaxf(best, -0.5f * (A * ex * ex + 2.f * B * ex * dy + C * dy * dy));
        const float ey = e ? by1 : by0;
        const float dx = fminf(fmaxf(-B * ey / A, bx0), bx1);
        best = fmaxf(best, -0.5f * (A * dx * dx + 2.f * B * dx * ey + C * ey * ey));
    }
    return best;
}

// Relative error, per unit of the magnitude sum S of Eq. 3's terms, that the
// variant's exponent may have against the quadratic, with room.  The products of
// Eq. 6 add up to log2(e) S in magnitude at most, so one fp16 or bf16 term (2^-11
// or 2^-8 of each coefficient; log2 o's own share is inside box_reaches' margin)
// errs by 0.00071 S or 0.0057 S, the split operands by 2^-21 S.  The five e4m3 terms
// err by 2^-20 of a coefficient or 2^-21 of the largest, the monomials add up to 402
// at most: 0.0003 S.  Twice these bounds for one term kept so many dead entries that
// the bf16 backward of 500k splats on 64 x 64 pixels was slower than without
// culling: 1768 -> 1869 us, with these 1789; 1920 x 1080, 1M, full lists, bf16
// forward 389 -> 363 us, backward 727 -> 676.
template <int V>
constexpr float reach_rel() {
    return V == GS_BLEND_TC_FP16 ? 1.0f / 1024 : V == GS_BLEND_TC_BF16 ? 1.0f / 128
           : V == GS_BLEND_TC_FP8_SPLIT ? 1.0f / 256 : 1.0f / 131072;
}

// False only if a splat's alpha is below 1/255 at every pixel of a box; x0..x1
// and y0..y1 are the pixels' offsets from the splat's centre.  The largest
// quadratic over the box is compared with the threshold, lowered by 0.3 in
// base-2 units and by `rel` of the magnitude sum S of Eq. 3's terms (what the
// caller's arithmetic may be off).  A sum that is not finite keeps the splat.
__device__ __forceinline__ bool box_reaches(float A, float B, float C, float l2o, float x0, float x1, float y0,
                                            float y1, float S, float rel) {
    // the maximum over the box lies on the two lines nearest to the splat's centre
    // (a definite form; a nearly singular or indefinite one is kept)
    const float ex = fminf(fmaxf(0.f, x0), x1), ey = fminf(fmaxf(0.f, y0), y1);
    const float dy = fminf(fmaxf(__fdividef(-B * ex, C), y0), y1);
    const float dx = fminf(fmaxf(__fdividef(-B * ey, A), x0), x1);
    const float qx = fmaf(A * ex, ex, fmaf(2.f * B * ex, dy, C * dy * dy));
    const float qy = fmaf(A * dx, dx, fmaf(2.f * B * dx, ey, C * ey * ey));
    const float p = fmaf(-0.5f * kLog2e, fminf(qx, qy), l2o);
    const bool definite = A > 0.f && C > 0.f && A * C > B * B;
    return !(S < 1e30f && ((definite && fmaf(rel, S, p) < kLog2AlphaMin - 0.3f) || l2o < kLog2AlphaMin - 0.3f));
}

// False only if the splat's alpha, in the variant's own arithmetic, is below
// 1/255 at every pixel of the tile; such a splat changes no pixel (the skip
// rule of Alg. 1) and its MMA columns and compositing can be left out.  The
// margin (0.3 in base-2 units) is more than coeff_row's own test of far splats
// allows; S is taken at offsets enlarged by 16 px (a pixel is at most 15 from the
// upper half's reference in either direction, counted over the lower half's).
// (xh, yh): splat centre minus the upper half's reference; bx0..by1: the offsets of
// that half's pixels from it.
template <int V>
__device__ __forceinline__ bool splat_reaches(float A, float B, float C, float l2o, float xh, float yh, float bx0,
                                              float bx1, float by0, float by1) {
    const float ax = fabsf(xh) + 16.f, ay = fabsf(yh) + 16.f;
    const float S = fmaf(0.5f * fabsf(A) * ax, ax, fmaf(fabsf(B) * ax, ay, 0.5f * fabsf(C) * ay * ay));
    return box_reaches(A, B, C, l2o, xh + bx0, xh + bx1, yh + by0 - 8.0f, yh + by1, S, reach_rel<V>());
}

// Coefficient row of Eq. 6 for one splat and one reference pixel, in base-2
// units with log2(o) folded into the constant term: v . v_p = log2(e) power + log2 o.
// (xh, yh) = splat centre minus reference pixel.  fp16 operands cannot hold
// coefficients beyond 65504: if any would exceed 30000, the splat is tested
// against the half-tile's pixel-offset box (bx0..by1) and, if it cannot reach
// alpha >= 1/255 there, gets a dead row (exponent -200 everywhere); otherwise
// the coefficients are clamped (only splats far from the tile relative to
// their size reach this, and the error is stated in the design notes).
template <bool HALF>
__device__ __forceinline__ void coeff_row(float A, float B, float C, float l2o, float xh, float yh, float bx0,
                                          float bx1, float by0, float by1, float (&v)[6]) {
    const float ux = fmaf(A, xh, B * yh), uy = fmaf(B, xh, C * yh);
    const float P0 = -0.5f * fmaf(xh, ux, yh * uy);
    v[0] = -0.5f * A * kLog2e;
    v[1] = -0.5f * C * kLog2e;
    v[2] = -B * kLog2e;
    v[3] = -ux * kLog2e;
    v[4] = -uy * kLog2e;
    v[5] = fmaf(P0, kLog2e, l2o);
    if constexpr (HALF) {
        float big = 0.f;
#pragma unroll
        for (int i = 0; i < 6; ++i) big = fmaxf(big, fabsf(v[i]));
        if (big > 30000.f) {
            const float qmax = box_max_quadratic(A, B, C, xh + bx0, xh + bx1, yh + by0, yh + by1);
            if (fmaf(qmax, kLog2e, l2o) >= kLog2AlphaMin - 0.25f) {
#pragma unroll
                for (int i = 0; i < 6; ++i) v[i] = fminf(fmaxf(v[i], -30000.f), 30000.f);
            } else {
#pragma unroll
                for (int i = 0; i < 5; ++i) v[i] = 0.f;
                v[5] = kDeadPower;
            }
        }
    }
}

// Write row r of a B stage: v split into TERMS operand-type terms, each in its
// own K slots (once per monomial term), zero padding up to K.  Returns the
// factor that maps the MMA result back to v . v_p (1 unless FP8, whose rows
// are scaled by a power of two first).
template <int V>
__device__ __forceinline__ float store_coeff_row(uint8_t* mB, int r, const float (&v)[6]) {
    using TR = Traits<V>;
    if constexpr (TR::FP8) {
        float big = 0.f;
#pragma unroll
        for (int i = 0; i < 6; ++i) big = fmaxf(big, fabsf(v[i]));
        // 2^E <= big < 2^(E+1); scale 2^(7-E) puts the largest coefficient in [128, 256)
        const int E = big > 0.f ? ((__float_as_int(big) >> 23) & 0xff) - 127 : 0;
        const int sh = max(-100, min(100, 7 - E));
        const float scale = __int_as_float((127 + sh) << 23), inv = __int_as_float((127 - sh) << 23);
        uint8_t terms[TR::TERMS][6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            float rem = v[i] * scale;
#pragma unroll
            for (int t = 0; t < TR::TERMS; ++t) {
                const float sh = fp8_term_shift(t);
                terms[t][i] = to_e4m3(rem * sh);
                rem -= from_e4m3(terms[t][i]) / sh;
            }
        }
        // slot k = (t * PTERMS + s) * 6 + i holds term t of v_i (for every monomial term s)
#pragma unroll
        for (int kc = 0; kc < TR::ROW_BYTES / 16; ++kc) {
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t word = 0;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int k = kc * 16 + q * 4 + b;
                    const uint32_t e = (k < 6 * TR::TERMS * TR::PTERMS)
                                           ? terms[k / (6 * TR::PTERMS)][k % 6] : 0u;
                    word |= e << (8 * b);
                }
                w[q] = word;
            }
            *reinterpret_cast<uint4*>(mB + (r >> 3) * TR::SBO + kc * 128 + (r & 7) * 16) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
        return inv;
    } else {
        uint16_t terms[3][6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            float rem = v[i];
#pragma unroll
            for (int t = 0; t < TR::TERMS; ++t) {
                terms[t][i] = to_op<TR::HALF>(rem);
                rem -= from_op<TR::HALF>(terms[t][i]);
            }
        }
#pragma unroll
        for (int kc = 0; kc < TR::K / 8; ++kc) {
            uint16_t e[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int kk = kc * 8 + i;
                e[i] = (kk < 6 * TR::TERMS) ? terms[kk / 6][kk % 6] : (uint16_t)0;
            }
            store_row_chunk<V>(mB, r, kc, e);
        }
        return 1.0f;
    }
}

// Both rows of a splat (ju: upper reference, jl: lower) of a 16-bit variant.
// Their three quadratic coefficients are the same numbers and are split once
// (unless coeff_row replaced one of the rows).
template <int V>
__device__ __forceinline__ void store_coeff_pair(uint8_t* mB, int ju, int jl, const float (&vu)[6],
                                                 const float (&vl)[6]) {
    using TR = Traits<V>;
    uint16_t terms[3][6];
    auto split = [&](int i, float v) {
        float rem = v;
#pragma unroll
        for (int t = 0; t < TR::TERMS; ++t) {
            terms[t][i] = to_op<TR::HALF>(rem);
            rem -= from_op<TR::HALF>(terms[t][i]);
        }
    };
    auto store = [&](int row) {
#pragma unroll
        for (int kc = 0; kc < TR::K / 8; ++kc) {
            uint16_t e[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int kk = kc * 8 + i;
                e[i] = (kk < 6 * TR::TERMS) ? terms[kk / 6][kk % 6] : (uint16_t)0;
            }
            store_row_chunk<V>(mB, row, kc, e);
        }
    };
#pragma unroll
    for (int i = 0; i < 6; ++i) split(i, vu[i]);
    store(ju);
    if (vl[0] != vu[0] || vl[1] != vu[1] || vl[2] != vu[2]) {
#pragma unroll
        for (int i = 0; i < 3; ++i) split(i, vl[i]);
    }
#pragma unroll
    for (int i = 3; i < 6; ++i) split(i, vl[i]);
    store(jl);
}

// The CUDA-core variant's B stage: splat j's two FP32 rows, 12 floats at 48 j
// (upper row 0..5, lower row 6..11).
__device__ __forceinline__ void store_cc_rows(uint8_t* mB, int j, const float (&vu)[6], const float (&vl)[6]) {
    float4* d = reinterpret_cast<float4*>(mB + 48 * j);
    d[0] = make_float4(vu[0], vu[1], vu[2], vu[3]);
    d[1] = make_float4(vu[4], vu[5], vl[0], vl[1]);
    d[2] = make_float4(vl[2], vl[3], vl[4], vl[5]);
}

// Row `row` of M_p, the pixel-monomial operand: the 6 monomials of the pixel
// (offsets xb, yb from its half's reference), in the slot order of
// store_coeff_row (for FP8 each monomial as 2 exact e4m3 terms).
template <int V>
__device__ __forceinline__ void store_mp_row(uint8_t* sA, int row, float xb, float yb) {
    using TR = Traits<V>;
    const float vp[6] = {xb * xb, yb * yb, xb * yb, xb, yb, 1.0f};
    if constexpr (TR::FP8) {
        float pv[2][6];  // the 2 exact e4m3 terms of each monomial
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            pv[0][i] = from_e4m3(to_e4m3(vp[i]));
            pv[1][i] = vp[i] - pv[0][i];
        }
#pragma unroll
        for (int kc = 0; kc < TR::ROW_BYTES / 16; ++kc) {
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t word = 0;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int k = kc * 16 + q * 4 + b;
                    const uint32_t e = (k < 6 * TR::TERMS * TR::PTERMS)
                                           ? to_e4m3(pv[(k / 6) % TR::PTERMS][k % 6] / fp8_term_shift(k / (6 * TR::PTERMS)))
                                           : 0u;
                    word |= e << (8 * b);
                }
                w[q] = word;
            }
            *reinterpret_cast<uint4*>(sA + (row >> 3) * TR::SBO + kc * 128 + (row & 7) * 16) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else {
#pragma unroll
        for (int kc = 0; kc < TR::K / 8; ++kc) {
            uint16_t e[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int k = kc * 8 + i;
                e[i] = (k < 6 * TR::TERMS) ? to_op<TR::HALF>(vp[k % 6]) : (uint16_t)0;
            }
            store_row_chunk<V>(sA, row, kc, e);
        }
    }
}

__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld_32x32b_x8(uint32_t taddr, uint32_t (&v)[8]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_32x32b_x4(uint32_t taddr, uint32_t (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr));
}

// Copies the nine values of item g of view v (mean, conic, opacity, colour) to
// d[0], d[kGroup], ..., d[8 kGroup] asynchronously (cp.async; the caller commits).
__device__ __forceinline__ void copy_splat_async(const BlendArgs& a, float* d, uint32_t g, int v) {
    const float* m = reinterpret_cast<const float*>(a.mean2d + g);
    cp_async4(d, m);
    cp_async4(d + kGroup, m + 1);
    const float* cn = a.conic + 3 * (size_t)g;
    cp_async4(d + 2 * kGroup, cn);
    cp_async4(d + 3 * kGroup, cn + 1);
    cp_async4(d + 4 * kGroup, cn + 2);
    cp_async4(d + 5 * kGroup, a.opac + (g - (uint32_t)(v * a.n_per_view)));
    if (a.rgb) {
        const float* cl = a.rgb + 3 * (size_t)g;
        cp_async4(d + 6 * kGroup, cl);
        cp_async4(d + 7 * kGroup, cl + 1);
        cp_async4(d + 8 * kGroup, cl + 2);
    }
}

// Queue items a block claims at once after a short tile, `left` being unclaimed: up
// to 4 where the tiles come longest first (the next ones are no longer), else up
// to 2 (more would deal neighbouring dense tiles of an unsorted queue to one
// block), and no more than half a block's share of what is left, so that the last
// claims are single.  17190 tiles of 7 splats each, 3053 x 1439: 88 -> 78 us.  (In
// the backward the same gained 6% there and cost 3% at 3840 x 2160, where the tile
// headers are hidden anyway: not used.)
__device__ __forceinline__ int short_claim(int left, bool ordered) {
    return max(1, min(ordered ? 4 : 2, left / (2 * (int)gridDim.x)));
}

__device__ __forceinline__ float log2_opacity(float o) { return o > 0.f ? __log2f(o) : -INFINITY; }
__device__ __forceinline__ float sat(float x) { return __saturatef(x); }

// Work item of one pipeline stage.  n > 0: chunk [base, base + n) of the
// tile's list; n == 0: the tile is empty; n < 0: end of the queue.
struct StageHdr {
    int tile;  // global tile id
    int seq;   // this CTA's running tile number
    int base;  // list position of the chunk's first splat
    int n;
    int slot;  // queue position of the tile (gs_tile_power output row)
    float xc, yc;  // the upper half's reference pixel
    int upto;      // list entries up to the chunk's end; 0: up to its last splat
};

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// COUNT: adds to *a.issued (a kernel of its own: counting in the row builder cost the
// calls that do not ask for it 1 to 2%)
template <int V, int CH, int SS, bool DUMP, bool COUNT>
__global__ void __launch_bounds__(kThreads, 4) k_blend_tc(const __grid_constant__ BlendArgs a) {
    using TR = Traits<V>;
    using LY = Layout<SS, CH, V>;
    constexpr int SBO = TR::SBO, RAW = LY::RAW;
    constexpr uint32_t IDESC = idesc_f16(TR::FMT, 128, 2 * CH);
    // columns an epilogue thread takes at a time (CC: of shared memory, more loads in
    // flight; 3840 x 2160, 3M 621 -> 611 us, 1920 x 1080 465 -> 452)
    constexpr int EC = TR::CC ? 8 : 4;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sA = smem;
    uint8_t* sB = smem + LY::OFF_B;
    float4* sRec = reinterpret_cast<float4*>(smem + LY::OFF_REC);  // r, g, b, cap
    float* sIdx = reinterpret_cast<float*>(smem + LY::OFF_IDX);
    float2* sScl = reinterpret_cast<float2*>(smem + LY::OFF_SCL);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + LY::OFF_BAR);
    StageHdr* sHdr = reinterpret_cast<StageHdr*>(smem + LY::OFF_HDR);
    float* sRaw = reinterpret_cast<float*>(smem + LY::OFF_RAW);  // [slot][field][splat]
    StageHdr* sRawHdr = reinterpret_cast<StageHdr*>(smem + LY::OFF_RAWHDR);
    uint32_t* sTmem = reinterpret_cast<uint32_t*>(smem + LY::OFF_MISC);
    volatile int* sAbort = reinterpret_cast<volatile int*>(smem + LY::OFF_MISC + 4);
    volatile int* sDoneRing = reinterpret_cast<volatile int*>(smem + LY::OFF_MISC + 16);
    auto bar_full = [&](int s) { return smem_u32(bars + s); };
    auto bar_empty = [&](int s) { return smem_u32(bars + SS + s); };
    auto bar_tfull = [&](int t) { return smem_u32(bars + 2 * SS + t); };
    auto bar_tempty = [&](int t) { return smem_u32(bars + 2 * SS + kTStages + t); };
    const uint32_t bar_drain = smem_u32(bars + 2 * SS + 2 * kTStages);
    auto bar_rfull = [&](int r) { return smem_u32(bars + 2 * SS + 2 * kTStages + 1 + r); };
    auto bar_rempty = [&](int r) { return smem_u32(bars + 2 * SS + 2 * kTStages + 1 + RAW + r); };
    auto bar_rec = [&](int r) { return smem_u32(bars + 2 * SS + 2 * kTStages + 1 + 2 * RAW + r); };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_items = a.total_tiles;  // gs_tile_power: the number of listed tiles
    const bool origin = a.ref_origin != 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < SS; ++s) {
            mbar_init(bar_full(s), 1);
            mbar_init(bar_empty(s), 1 + kEpiWarps);
        }
        for (int t = 0; t < kTStages; ++t) {
            mbar_init(bar_tfull(t), 1);
            mbar_init(bar_tempty(t), kEpiWarps);
        }
        mbar_init(bar_drain, 1);
        for (int r = 0; r < RAW; ++r) {
            mbar_init(bar_rfull(r), 1);
            mbar_init(bar_rempty(r), 1);
        }
        for (int r = 0; r < kRecSlots; ++r) mbar_init(bar_rec(r), 1);
        *sAbort = 0;
        mbar_fence_init();
    }
    // pixel matrix M_p of a 16 x 8 half-tile (A operand)
    for (int row = threadIdx.x; row < 128; row += kThreads) {
        const float xb = (origin ? 0.f : 7.5f) - (float)lane_col(row);
        const float yb = (origin ? 0.f : 3.5f) - (float)lane_row(row);
        store_mp_row<V>(sA, row, xb, yb);
    }
    fence_proxy_async_smem();
    if (warp == 5) {
        tmem_alloc(smem_u32(sTmem), LY::TCOLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *sTmem;
    const uint64_t tmo = a.timeout_ns;

    if (warp < kEpiWarps) {
        // ------------------------------------------------------- epilogue --
        const int r = warp * 32 + lane;  // accumulator lane: pixel r of each half
        // this lane's pixel monomials (the same in both halves), as M_p holds them
        float mp[5];
        {
            const float xb = (origin ? 0.f : 7.5f) - (float)lane_col(r);
            const float yb = (origin ? 0.f : 3.5f) - (float)lane_row(r);
            mp[0] = xb * xb;
            mp[1] = yb * yb;
            mp[2] = xb * yb;
            mp[3] = xb;
            mp[4] = yb;
        }
        int cur_seq = -1, slot = 0;
        int px = 0, py_up = 0, W = 0, H = 0;
        bool in_up = false, in_lo = false, wdone = true;
        long long pix_off = 0;
        float2 T = make_float2(0.f, 0.f), Tstop = T, last = T, Cr = T, Cg = T, Cb = T;
        for (int k = 0;; ++k) {
            const int s = k % SS, t = k % kTStages;
            const uint32_t ps = (uint32_t)(k / SS) & 1u, pt = (uint32_t)(k / kTStages) & 1u;
            if (!mbar_wait_bounded(bar_tfull(t), pt, tmo, sAbort) || !mbar_wait_bounded(bar_full(s), ps, tmo, sAbort)) {
                *sAbort = 1;
                atomicOr(a.err, kErrTimeout);
                break;
            }
            const StageHdr hd = sHdr[s];
            if (hd.seq != cur_seq) {
                if (!DUMP && cur_seq >= 0) {  // write the finished tile's pixels
                    const size_t plane = (size_t)W * H;
                    float* img = a.image + 3 * pix_off;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h ? in_lo : in_up) {
                            const size_t p = (size_t)(py_up + 8 * h) * W + px;
                            const float Tf = h ? T.y + Tstop.y : T.x + Tstop.x;
                            img[p] = (h ? Cr.y : Cr.x) + Tf * a.bg[0];
                            img[plane + p] = (h ? Cg.y : Cg.x) + Tf * a.bg[1];
                            img[2 * plane + p] = (h ? Cb.y : Cb.x) + Tf * a.bg[2];
                            a.T_final[pix_off + p] = Tf;
                            a.n_contrib[pix_off + p] = (int)(h ? last.y : last.x);
                        }
                    }
                }
                if (hd.n < 0) break;
                cur_seq = hd.seq;
                const int v = view_of(a, hd.tile);
                const ViewDesc vd = a.views[v];
                const int lt = hd.tile - vd.tile_begin;
                W = vd.W;
                H = vd.H;
                pix_off = vd.pix_off;
                px = (lt % vd.tiles_x) * kTile + lane_col(r);
                py_up = (lt / vd.tiles_x) * kTile + lane_row(r);
                in_up = px < W && py_up < H;
                in_lo = px < W && py_up + 8 < H;
                slot = hd.slot;
                T = make_float2(in_up || DUMP ? 1.f : 0.f, in_lo || DUMP ? 1.f : 0.f);
                Tstop = last = Cr = Cg = Cb = make_float2(0.f, 0.f);
                wdone = DUMP ? false : __all_sync(0xffffffffu, T.x == 0.f && T.y == 0.f);
                if (!DUMP && wdone && lane == 0) atomicAdd((int*)&sDoneRing[cur_seq % kDoneRing], 1);
            }
            tc_fence_after();
            const int n = hd.n;
            const int base = hd.base;
            if (n > 0 && !wdone) {
                const uint32_t tb = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(t * 2 * CH);
                const float4* rec = sRec + s * CH;
                const float* idx1 = sIdx + s * CH;
#pragma unroll 1
                for (int c0 = 0; c0 < n; c0 += EC) {
                    // every pixel of this warp has stopped: the chunk's later splats change nothing
                    if (!DUMP && c0 > 0 && __all_sync(0xffffffffu, T.x == 0.f && T.y == 0.f)) break;
                    uint32_t vu[EC], vl[EC];
                    // CC: Eq. 6 on the CUDA cores, column by column below (both pixels of
                    // the lane share their monomials)
                    const float* rows = reinterpret_cast<const float*>(sB + s * LY::B_BYTES) + (size_t)c0 * 12;
                    auto cc_power = [&](int c) {
                        const float4 a0 = *reinterpret_cast<const float4*>(rows + 12 * c);
                        const float4 a1 = *reinterpret_cast<const float4*>(rows + 12 * c + 4);
                        const float4 a2 = *reinterpret_cast<const float4*>(rows + 12 * c + 8);
                        float2 p = __fmul2_rn(make_float2(a0.x, a1.z), make_float2(mp[0], mp[0]));
                        p = __ffma2_rn(make_float2(a0.y, a1.w), make_float2(mp[1], mp[1]), p);
                        p = __ffma2_rn(make_float2(a0.z, a2.x), make_float2(mp[2], mp[2]), p);
                        p = __ffma2_rn(make_float2(a0.w, a2.y), make_float2(mp[3], mp[3]), p);
                        p = __ffma2_rn(make_float2(a1.x, a2.z), make_float2(mp[4], mp[4]), p);
                        return __fadd2_rn(make_float2(a1.y, a2.w), p);
                    };
                    if constexpr (EC == 4 && !TR::CC) {
                        tmem_ld_32x32b_x4(tb + (uint32_t)c0, vu);
                        tmem_ld_32x32b_x4(tb + (uint32_t)(CH + c0), vl);
                        tmem_ld_wait();
                    }
                    if constexpr (TR::FP8) {  // undo the per-row scaling of the e4m3 operands
                        const float2* scl = sScl + s * CH;
#pragma unroll
                        for (int c = 0; c < EC; ++c) {
                            const float2 z = __fmul2_rn(make_float2(__uint_as_float(vu[c]), __uint_as_float(vl[c])),
                                                        scl[c0 + c]);
                            vu[c] = __float_as_uint(z.x);
                            vl[c] = __float_as_uint(z.y);
                        }
                    }
                    if constexpr (DUMP) {
#pragma unroll
                        for (int c = 0; c < EC; ++c) {
                            const int j = c0 + c;
                            if (j < n) {
                                float* o = a.dump + ((size_t)slot * a.max_len + (size_t)base + j) * 256;
                                const int p = 16 * lane_row(r) + lane_col(r);
                                o[p] = __uint_as_float(vu[c]);
                                o[p + 128] = __uint_as_float(vl[c]);
                            }
                        }
                    } else {
                        float ix[EC];
#pragma unroll
                        for (int q = 0; q < EC; q += 4)
                            *reinterpret_cast<float4*>(ix + q) = *reinterpret_cast<const float4*>(idx1 + c0 + q);
#pragma unroll
                        for (int c = 0; c < EC; ++c) {
                            float2 pw;
                            if constexpr (TR::CC) pw = cc_power(c);
                            else pw = make_float2(__uint_as_float(vu[c]), __uint_as_float(vl[c]));
                            const float4 rc = rec[c0 + c];
                            float2 al;
                            al.x = ex2_approx(fminf(pw.x, rc.w));
                            al.y = ex2_approx(fminf(pw.y, rc.w));
                            float2 cull;
                            cull.x = sat(fmaf(al.x, -kCullScale, kAlphaMin * kCullScale));
                            cull.y = sat(fmaf(al.y, -kCullScale, kAlphaMin * kCullScale));
                            al = __ffma2_rn(neg2(al), cull, al);
                            const float2 tT = __ffma2_rn(neg2(al), T, T);
                            float2 stop;
                            stop.x = sat(fmaf(tT.x, -kStopScale, kTMin * kStopScale));
                            stop.y = sat(fmaf(tT.y, -kStopScale, kTMin * kStopScale));
                            Tstop = __ffma2_rn(T, stop, Tstop);
                            const float2 a2 = __ffma2_rn(neg2(al), stop, al);
                            const float2 w = __fmul2_rn(a2, T);
                            T = __ffma2_rn(neg2(tT), stop, tT);
                            Cr.x = __fmaf_rn(rc.x, w.x, Cr.x);
                            Cr.y = __fmaf_rn(rc.x, w.y, Cr.y);
                            Cg.x = __fmaf_rn(rc.y, w.x, Cg.x);
                            Cg.y = __fmaf_rn(rc.y, w.y, Cg.y);
                            Cb.x = __fmaf_rn(rc.z, w.x, Cb.x);
                            Cb.y = __fmaf_rn(rc.z, w.y, Cb.y);
                            float2 used;
                            used.x = sat(a2.x * kCullScale);
                            used.y = sat(a2.y * kCullScale);
                            last = __ffma2_rn(used, __fadd2_rn(make_float2(ix[c], ix[c]), neg2(last)), last);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tempty(t));
            if (!DUMP && !wdone) {
                wdone = __all_sync(0xffffffffu, T.x == 0.f && T.y == 0.f);
                if (wdone && lane == 0) atomicAdd((int*)&sDoneRing[cur_seq % kDoneRing], 1);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_empty(s));
        }
    } else if (warp == kEpiWarps) {
        // -------------------------------------------------------- scanner --
        // Walks the tiles' lists in groups of 32 entries, one per lane, and packs
        // the entries that reach a pixel of the tile (splat_reaches), in list order,
        // into chunks of CH raw splats for the row builders.
        const float bx0 = origin ? -15.0f : -7.5f, bx1 = origin ? 0.0f : 7.5f;
        const float by0 = origin ? -7.0f : -3.5f, by1 = origin ? 0.0f : 3.5f;
        const bool use_rec = !DUMP && a.use_rec;
        const float* sRecT = reinterpret_cast<const float*>(smem + LY::OFF_RECT);
        // A group's splats are copied into a slot of shared memory a group ahead of
        // their use, without passing through registers: each lane its own entry's nine
        // values by cp.async, or (with splat records) by TMA gathers of four records.
        float* sGeo = reinterpret_cast<float*>(smem + LY::OFF_GEO) + lane;
        uint32_t rec_phase = 0, rec_flight = 0;  // per TMA slot: the phase to wait for, a copy in flight
        auto rec_wait = [&](int slot) -> bool {
            if (!((rec_flight >> slot) & 1u)) return true;
            if (!mbar_wait_bounded(bar_rec(slot), (rec_phase >> slot) & 1u, tmo, sAbort)) {
                *sAbort = 1;
                atomicOr(a.err, kErrTimeout);
                return false;
            }
            rec_phase ^= 1u << slot;
            rec_flight &= ~(1u << slot);
            return true;
        };
        auto fetch = [&](uint32_t g, int n, int v, int slot) {  // n: entries from the group's first on (may exceed 32)
            if (use_rec) {
                if (n <= 0 || !rec_wait(slot)) return;
                const uint32_t id = lane < n ? g : 0u;  // rows past n repeat id 0, a row of the table
                const int src = 4 * (lane & 7), ng = (min(n, kGroup) + 3) >> 2;
                const uint32_t g0 = __shfl_sync(0xffffffffu, id, src), g1 = __shfl_sync(0xffffffffu, id, src + 1);
                const uint32_t g2 = __shfl_sync(0xffffffffu, id, src + 2), g3 = __shfl_sync(0xffffffffu, id, src + 3);
                fence_proxy_async_smem();  // the slot's earlier reads before the copies' writes
                __syncwarp();
                if (lane == 0) mbar_arrive_expect_tx(bar_rec(slot), (uint32_t)(ng * 4 * kRecBytes));
                __syncwarp();
                if (lane < ng)
                    tma_gather4(smem_u32(sRecT + (size_t)(slot * kGroup + 4 * lane) * kRecFloats), &a.rec_map, 0, g0,
                                g1, g2, g3, bar_rec(slot));
                rec_flight |= 1u << slot;
            } else {
                if (lane < n) copy_splat_async(a, sGeo + slot * (kGeoFields * kGroup), g, v);
                cp_async_commit();
            }
        };
        // The next tile: its queue item is claimed when a tile starts, then its id, range,
        // first two groups of entries and first group of splats are looked up, one
        // dependent load per group of the current tile, so that a tile that ends early
        // (as dense ones do) finds them ready.  After a short tile, whose next one is not
        // ready, several items are claimed and looked up together, one per lane (short_claim).
        int claim = 0, n_claim = 1, b_q = 0, b_n = 0, b_i = 0;  // items b_q + [b_i, b_n) are claimed
        uint32_t b_tile = 0, b_start = 0, b_stop = 0;           // lane i: item b_q + i
        int q_next = 0, nt_step = 0, nt_tile = 0, nt_len = 0, nt_slot = 2;
        uint32_t nt_start = 0, nt_id = 0, nt_id2 = 0;
        auto step_next = [&]() {
            if (nt_step == 0 && b_i == b_n) {
                b_q = __shfl_sync(0xffffffffu, claim, 0);
                b_n = n_claim;
                b_i = 0;
                const int qi = b_q + lane;
                if (lane < b_n && qi < n_items)
                    b_tile = DUMP ? a.tiles[qi] : tile_at(a, qi * a.shard_count + a.shard_index);
            } else if (nt_step == 1 && b_i == 0) {
                if (lane < b_n && b_q + lane < n_items) {
                    b_start = a.ranges[2 * b_tile];
                    b_stop = a.ranges[2 * b_tile + 1];
                }
            } else if (nt_step <= 2) {
                q_next = b_q + b_i;
                if (q_next >= n_items) {
                    nt_step = 4;
                    return;
                }
                nt_tile = (int)__shfl_sync(0xffffffffu, b_tile, b_i);
                nt_start = __shfl_sync(0xffffffffu, b_start, b_i);
                const uint32_t stop = __shfl_sync(0xffffffffu, b_stop, b_i);
                ++b_i;
                nt_len = stop > nt_start ? (int)(stop - nt_start) : 0;
                if (DUMP && nt_len > a.max_len) nt_len = a.max_len;
                if (lane < nt_len) nt_id = a.ids[nt_start + lane];
                if (lane + kGroup < nt_len) nt_id2 = a.ids[nt_start + kGroup + lane];
                nt_step = 2;
            } else if (nt_step == 3) {
                fetch(nt_id, nt_len, view_of(a, nt_tile), nt_slot);
            } else {
                return;
            }
            ++nt_step;
        };
        // The open raw slot: free, and not yet published
        int k = 0;
        bool open = false, quit = false;
        auto acquire = [&]() -> bool {
            if (!mbar_wait_bounded(bar_rempty(k % RAW), ((uint32_t)(k / RAW) & 1u) ^ 1u, tmo, sAbort)) {
                *sAbort = 1;
                atomicOr(a.err, kErrTimeout);
                return false;
            }
            open = true;
            return !*sAbort;
        };
        auto publish = [&](const StageHdr& h) {
            if (lane == 0) sRawHdr[k % RAW] = h;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_rfull(k % RAW));
            ++k;
            open = false;
        };
        if (lane == 0) claim = (int)atomicAdd(a.queue, 1u);
        for (int seq = 0; !quit; ++seq) {
            while (nt_step < 4) step_next();
            const int q = q_next;
            if (q >= n_items) {
                if (acquire()) publish(StageHdr{0, -2, 0, -1, q, 0.f, 0.f, 0});
                break;
            }
            const int tile = nt_tile, len = nt_len, vview = view_of(a, tile);
            const uint32_t start = nt_start;
            uint32_t gn = nt_id2;  // the next group's entries
            int slot = nt_slot, ahead = 0;  // this group's slot, the next group's
            nt_slot ^= 1;
            nt_step = 0;
            if (b_i == b_n) {
                n_claim = len > 2 * kGroup ? 1 : short_claim(n_items - b_q, a.order != nullptr);
                if (lane == 0) claim = (int)atomicAdd(a.queue, (unsigned)n_claim);
            }
            const ViewDesc vd = a.views[vview];
            const int lt = tile - vd.tile_begin;
            const float xc = (float)((lt % vd.tiles_x) * kTile) + (origin ? 0.5f : 8.0f);
            const float yc = (float)((lt / vd.tiles_x) * kTile) + (origin ? 0.5f : 4.0f);
            if (lane == 0) sDoneRing[seq % kDoneRing] = 0;
            int fill = 0, sent = 0;  // splats in the open slot; splats published
            const int ng = (len + kGroup - 1) / kGroup;
            int gi = 0;
            for (; gi < ng; ++gi) {
                // every pixel of this tile has stopped: skip the rest of its list
                if (!DUMP && sent > 0 && __all_sync(0xffffffffu, sDoneRing[seq % kDoneRing] >= kEpiWarps)) {
                    fill = 0;  // the open slot, if any, goes to the next tile
                    if (!use_rec) cp_async_wait<0>();  // the copies of the group not taken, before their slot is reused
                    break;
                }
                const int e = gi * kGroup + lane;
                if (gi + 1 < ng) fetch(gn, len - (gi + 1) * kGroup, vview, ahead);
                float2 m;
                float A, B, C, l2o, cr = 0.f, cg = 0.f, cb = 0.f;
                if (use_rec) {
                    if (!rec_wait(slot)) {
                        quit = true;
                        break;
                    }
                    const float4* rp = reinterpret_cast<const float4*>(sRecT + (size_t)(slot * kGroup + lane) * kRecFloats);
                    const float4 r0 = rp[0], r1 = rp[1], r2 = rp[2];
                    m = make_float2(r0.x, r0.y);
                    A = r0.z;
                    B = r0.w;
                    C = r1.x;
                    l2o = r1.y;
                    cr = r2.x;
                    cg = r2.y;
                    cb = r2.z;
                } else {
                    // all groups but the one just requested have arrived (the lane's own copies)
                    if (gi + 1 < ng) cp_async_wait<1>();
                    else cp_async_wait<0>();
                    const float* d = sGeo + slot * (kGeoFields * kGroup);
                    m = make_float2(d[0], d[kGroup]);
                    A = d[2 * kGroup];
                    B = d[3 * kGroup];
                    C = d[4 * kGroup];
                    l2o = log2_opacity(d[5 * kGroup]);
                    if (a.rgb) {
                        cr = d[6 * kGroup];
                        cg = d[7 * kGroup];
                        cb = d[8 * kGroup];
                    }
                }
                slot = ahead;
                ahead ^= 1;
                if (e + 2 * kGroup < len) gn = a.ids[start + e + 2 * kGroup];
                const bool keep =
                    e < len && (DUMP || splat_reaches<V>(A, B, C, l2o, m.x - xc, m.y - yc, bx0, bx1, by0, by1));
                const unsigned kb = __ballot_sync(0xffffffffu, keep);
                if (kb != 0u) {
                    // slot position of this lane's splat, counted from the open slot's start
                    int pos = keep ? fill + __popc(kb & ((1u << lane) - 1u)) : -1;
                    fill += __popc(kb);
                    for (;;) {
                        if (!open && !acquire()) {
                            quit = true;
                            break;
                        }
                        if (pos >= 0 && pos < CH) {
                            float* w = sRaw + (k % RAW) * (kRawFields * CH) + pos;
                            w[0] = m.x;
                            w[CH] = m.y;
                            w[2 * CH] = A;
                            w[3 * CH] = B;
                            w[4 * CH] = C;
                            w[5 * CH] = l2o;
                            w[6 * CH] = cr;
                            w[7 * CH] = cg;
                            w[8 * CH] = cb;
                            w[9 * CH] = (float)(e + 1);
                        }
                        if (fill < CH) break;
                        publish(StageHdr{tile, seq, sent, CH, q, xc, yc, 0});
                        sent += CH;
                        fill -= CH;
                        pos -= CH;
                        if (fill == 0) break;
                    }
                    if (quit) break;
                }
                step_next();
            }
            if (quit) break;
            // the tile's last chunk; a tile of which nothing is left travels as one empty
            // chunk, so that its pixels are written
            if (fill > 0 || sent == 0) {
                if (!open && !acquire()) break;
                publish(StageHdr{tile, seq, sent, fill, q, xc, yc, len});
            } else if constexpr (COUNT) {
                // issued pairs: the entries after the last chunk, none of them kept (the
                // row builder counts the others)
                const int upto = (int)sRaw[(k - 1) % RAW * (kRawFields * CH) + 9 * CH + CH - 1];
                if (gi == ng && lane == 0 && sDoneRing[seq % kDoneRing] < kEpiWarps)
                    atomicAdd(a.issued, 256ull * (unsigned long long)(len - upto));
            }
        }
        // copies still in flight land before the block leaves
        for (int r = 0; r < kRecSlots; ++r)
            if ((rec_flight >> r) & 1u) mbar_wait_bounded(bar_rec(r), (rec_phase >> r) & 1u, 1000000000ull, nullptr);
    } else {
        // ---------------------------------------------------- row builder --
        // Turns each raw chunk into a stage: the coefficient rows of both halves and
        // the epilogue's records.  A chunk of a tile whose pixels have all stopped
        // meanwhile is dropped.
        const float bx0 = origin ? -15.0f : -7.5f, bx1 = origin ? 0.0f : 7.5f;
        const float by0 = origin ? -7.0f : -3.5f, by1 = origin ? 0.0f : 3.5f;
        int k = 0;
        // issued pairs: every list entry up to the end of each chunk that is evaluated
        [[maybe_unused]] uint32_t issued = 0;
        [[maybe_unused]] int upto = 0;
        for (int kr = 0;; ++kr) {
            const int s = k % SS, rs = kr % RAW;
            if (!mbar_wait_bounded(bar_rfull(rs), (uint32_t)(kr / RAW) & 1u, tmo, sAbort) ||
                !mbar_wait_bounded(bar_empty(s), ((uint32_t)(k / SS) & 1u) ^ 1u, tmo, sAbort)) {
                *sAbort = 1;
                atomicOr(a.err, kErrTimeout);
                break;
            }
            const StageHdr hd = sRawHdr[rs];
            if (!DUMP && hd.n > 0 && hd.base > 0 && __all_sync(0xffffffffu, sDoneRing[hd.seq % kDoneRing] >= kEpiWarps)) {
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_rempty(rs));
                continue;
            }
            if (hd.n > 0) {
                uint8_t* mB = sB + s * LY::B_BYTES;
                if constexpr (CH == 16 && !TR::CC) {
                    // one row per lane: lanes 0..15 the upper half's, 16..31 the lower half's
                    const int j = lane & 15;
                    const bool lower = lane >= 16;
                    const float* w = sRaw + rs * (kRawFields * CH) + j;
                    float v[6] = {0.f, 0.f, 0.f, 0.f, 0.f, kDeadPower};  // padding column: dead rows, no colour
                    float4 rc = make_float4(0.f, 0.f, 0.f, 0.f);
                    float ix = 0.f;
                    if (j < hd.n) {
                        const float l2o = w[5 * CH];
                        coeff_row<TR::HALF>(w[2 * CH], w[3 * CH], w[4 * CH], l2o, w[0] - hd.xc,
                                            w[CH] - (lower ? hd.yc + 8.0f : hd.yc), bx0, bx1, by0, by1, v);
                        rc = make_float4(w[6 * CH], w[7 * CH], w[8 * CH], fminf(l2o, kLog2AlphaMax));
                        ix = w[9 * CH];
                    }
                    if (!lower) {
                        sRec[s * CH + j] = rc;
                        sIdx[s * CH + j] = ix;
                    }
                    const float sc = store_coeff_row<V>(mB, lower ? CH + j : j, v);
                    if constexpr (TR::FP8) reinterpret_cast<float*>(sScl + s * CH + j)[lower ? 1 : 0] = sc;
                } else {
                for (int j = lane; j < CH; j += 32) {
                    const float* w = sRaw + rs * (kRawFields * CH) + j;
                    float vu[6] = {0.f, 0.f, 0.f, 0.f, 0.f, kDeadPower};  // padding column: dead rows, no colour
                    float vl[6] = {0.f, 0.f, 0.f, 0.f, 0.f, kDeadPower};
                    float4 rc = make_float4(0.f, 0.f, 0.f, 0.f);
                    float ix = 0.f;
                    if (j < hd.n) {
                        const float A = w[2 * CH], B = w[3 * CH], C = w[4 * CH], l2o = w[5 * CH];
                        const float xh = w[0] - hd.xc;
                        coeff_row<TR::HALF && !TR::CC>(A, B, C, l2o, xh, w[CH] - hd.yc, bx0, bx1, by0, by1, vu);
                        coeff_row<TR::HALF && !TR::CC>(A, B, C, l2o, xh, w[CH] - (hd.yc + 8.0f), bx0, bx1, by0, by1,
                                                       vl);
                        rc = make_float4(w[6 * CH], w[7 * CH], w[8 * CH], fminf(l2o, kLog2AlphaMax));
                        ix = w[9 * CH];
                    }
                    sRec[s * CH + j] = rc;
                    sIdx[s * CH + j] = ix;
                    if constexpr (TR::CC) {
                        store_cc_rows(mB, j, vu, vl);
                    } else if constexpr (TR::FP8) {
                        const float su = store_coeff_row<V>(mB, j, vu);
                        const float sl = store_coeff_row<V>(mB, CH + j, vl);
                        sScl[s * CH + j] = make_float2(su, sl);
                    } else {
                        store_coeff_pair<V>(mB, j, CH + j, vu, vl);
                    }
                }
                }
            }
            if (lane == 0) sHdr[s] = hd;
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_rempty(rs));
            // the TMEM stage must be free even for a stage without an MMA, so
            // that tfull[t] never runs two phases ahead of a waiting epilogue warp
            const int t = k % kTStages;
            if (!mbar_wait_bounded(bar_tempty(t), ((uint32_t)(k / kTStages) & 1u) ^ 1u, tmo, sAbort)) {
                *sAbort = 1;
                atomicOr(a.err, kErrTimeout);
                break;
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar_full(s));
                if (hd.n > 0 && !TR::CC) {  // CC: the epilogue contracts the rows itself
                    tc_fence_after();
                    const uint32_t aA = smem_u32(sA), aB = smem_u32(sB + s * LY::B_BYTES);
#pragma unroll
                    for (int ks = 0; ks < TR::KSTEPS; ++ks) {
                        const uint64_t ad = smem_desc(aA + (uint32_t)(ks * 256), 128, SBO);
                        const uint64_t bd = smem_desc(aB + (uint32_t)(ks * 256), 128, SBO);
                        tc_mma<V>(tmem + (uint32_t)(t * 2 * CH), ad, bd, IDESC, ks > 0 ? 1u : 0u);
                    }
                    tc_commit(bar_tfull(t));
                    tc_commit(bar_empty(s));
                } else {
                    mbar_arrive(bar_tfull(t));
                    if (hd.n >= 0) mbar_arrive(bar_empty(s));
                }
            }
            __syncwarp();
            if constexpr (COUNT)
                if (hd.n >= 0) {  // (only this warp writes the stage)
                    const int to = hd.upto > 0 || hd.n == 0 ? hd.upto : (int)sIdx[s * CH + hd.n - 1];
                    issued += (uint32_t)(to - (hd.base > 0 ? upto : 0));
                    upto = to;
                }
            ++k;
            if (hd.n < 0) break;
        }
        if (lane == 0) {
            if constexpr (COUNT)
                if (issued > 0) atomicAdd(a.issued, 256ull * issued);
            // every MMA this thread issued has finished before TMEM is freed (a
            // fresh barrier: no phase of another stage can be mistaken for it)
            tc_commit(bar_drain);
            mbar_wait_bounded(bar_drain, 0, 1000000000ull, nullptr);
        }
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 5) tmem_dealloc(tmem, LY::TCOLS);
}

// Persistent grid: as many CTAs as fit on the GPU at once, from the kernel's
// registers, shared memory and threads and the SM's 512 TMEM columns.
template <int V, int CH, int SS, bool DUMP, bool COUNT = false>
cudaError_t launch_inst(const BlendArgs& a, int items, cudaStream_t s) {
    if constexpr (!DUMP && !COUNT)
        if (a.issued != nullptr) return launch_inst<V, CH, SS, DUMP, true>(a, items, s);
    using LY = Layout<SS, CH, V>;
    constexpr int bytes = LY::BYTES;
    auto kern = k_blend_tc<V, CH, SS, DUMP, COUNT>;
    static std::mutex mu;
    static LaunchShape cache;
    LaunchShape sh;
    const cudaError_t es = cached_shape(mu, cache, sh, [&](LaunchShape& r) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        int dev = 0, smem_sm = 0;
        cudaFuncAttributes fa{};
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess)
            return e;
        if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
        // registers are granted per warp in units of 256
        const int regs_warp = ((fa.numRegs * 32 + 255) / 256) * 256;
        const int by_regs = 65536 / (regs_warp * (kThreads / 32));
        const int by_smem = smem_sm / (bytes + (int)fa.sharedSizeBytes + 1024);
        const int by_threads = 2048 / kThreads;
        const int by_tmem = (int)(512 / LY::TCOLS);
        r.per_sm = by_regs;
        if (by_smem < r.per_sm) r.per_sm = by_smem;
        if (by_threads < r.per_sm) r.per_sm = by_threads;
        if (by_tmem < r.per_sm) r.per_sm = by_tmem;
        if (r.per_sm < 1) r.per_sm = 1;
        return cudaSuccess;
    });
    if (es != cudaSuccess) return es;
    const int grid = items < sh.per_sm * sh.sms ? (items > 0 ? items : 1) : sh.per_sm * sh.sms;
    kern<<<grid, kThreads, bytes, s>>>(a);
    count_launches();
    return cudaGetLastError();
}

// Instantiated per variant in blend_tc_v<V>.cu
template <int V>
cudaError_t launch_variant(const BlendArgs& a, int chunk, int stages, bool dump, int grid, cudaStream_t s);
template <>
cudaError_t launch_variant<1>(const BlendArgs&, int, int, bool, int, cudaStream_t);
template <>
cudaError_t launch_variant<2>(const BlendArgs&, int, int, bool, int, cudaStream_t);
template <>
cudaError_t launch_variant<3>(const BlendArgs&, int, int, bool, int, cudaStream_t);
template <>
cudaError_t launch_variant<4>(const BlendArgs&, int, int, bool, int, cudaStream_t);
template <>
cudaError_t launch_variant<5>(const BlendArgs&, int, int, bool, int, cudaStream_t);
template <>
cudaError_t launch_variant<6>(const BlendArgs&, int, int, bool, int, cudaStream_t);

}  // namespace tc
}  // namespace gs
