// Gradient of the tensor-core blend (the backward pass of Alg. 2).
//
// Same persistent structure as the forward kernel: warps 0-3 work on pixels
// (warp w owns TMEM lanes 32 w .. 32 w + 31, an 8 x 4 pixel block of each
// half; thread r holds pixel r of the tile's upper 16 x 8 half and pixel r of
// the lower half), warp 4 scans the lists of the global tile queue from each
// tile's largest n_contrib to the front, drops the entries that reach no pixel
// of the tile (splat_reaches, as in the forward) and packs the others into
// chunks of CH = 16 splats, back to front, and warp 5 builds the coefficient
// rows and issues the MMAs.
// Two MMAs per chunk:
//  1. exponents, exactly as in the forward pass (Eq. 6): D1 (128 pixels x 32)
//     = M_p (128 x K) . [v_g of the 16 splats for the upper and the lower
//     reference pixel], so the backward pass recomputes the forward's alpha;
//  2. the sums over pixels that make up each splat's gradient: every pixel
//     thread writes two per-(splat, pixel) values, the exponent gradient
//     dL/dpower (fp16 hi + lo) and the blending weight w = alpha T (fp16),
//     into A2 (96 rows = dpow {upper, lower half} x {hi, lo} x 16 splats and
//     w {upper, lower} x 16 splats, K = the 128 pixels of a half, stored
//     MN-major so that a thread writes 8 splats of its pixel with one 16-byte
//     store), and D2 (128 x 32) = A2 . B2 where B2 holds per pixel the
//     monomials [xb^2, yb^2, xb yb, xb, yb, 1] of Eq. 6 (exact in fp16) and
//     the pixel's dL/dimage (hi + lo, separately for each half).  Row
//     (dpow, h, s, j) of D2 then holds sum_p dpow m_p for splat j over half
//     h, from which the conic, mean and opacity gradients follow by the chain
//     rule; row (w, h, j) holds sum_p w dL/dC_p, the colour gradient.  The MMA
//     runs with M = 128: rows 96..127 of D2 read past the 96 rows (the next
//     8-pixel group, or the buffer's padding) and are ignored.
//
// Per pixel the splats are visited back to front (chunks in reverse order,
// splats inside a chunk from last to first), starting from T_final and the
// background: for each splat j < n_contrib that passes the 1/255 test,
//   T_j = T_{j+1} / (1 - a_j),  w_j = a_j T_j,
//   dL/da_j = T_j (c_j . g - S_j . g),  S_{j-1} . g = S_j . g + a_j (c_j . g - S_j . g)
// (S = the colour behind splat j, starting at the background), and
// dL/dpower = a dL/da (0 where alpha is clamped at 0.99), dL/do = sum dpow / o.
// Scaling keeps the fp16 operands in range: dL/dimage is multiplied by
// 2^(-E) with 2^E the largest |dL/dimage| of the tile, T by 2^12; the sums
// are scaled back in the finishing step.
//
// A2 and D2 are double buffered: chunk c writes A2[c % 2] while the MMA of
// chunk c - 1 runs, and the finishing step of chunk c - 1 (reading D2, chain
// rule, atomics) follows chunk c's stores, so the MMA's latency is hidden
// behind a whole chunk.  At a new tile B2 changes: its new columns wait for
// the pending chunk's MMA.  Each epilogue warp finishes its own rows, so the
// four warps never wait for one another.  D2's rows are ordered so that both
// halves of a splat lie in one warp: their gradients are added there and go
// out in 9 atomics per splat and tile (15 with one set per half).
// All waits are bounded by opts.timeout_ns as in the forward kernel.
//
// What bounds it: issue slots (56 to 62% of them, about 70 instructions per
// splat and warp) and the instruction cache: with all 16 splats of a chunk
// unrolled and the finishing step written out twice, a third of the stalls at
// 3840 x 2160 were warps without an instruction.  So the splats go through a
// rolled loop of two groups of 8, and every larger piece of code (finishing
// step, tile header, group copy) stands in one place.
// 1920 x 1080, 1M clustered splats, full rectangles (bf16 split): 1.671 ->
// 0.629 ms; opacity-aware (fp16 split): 0.538 -> 0.526; 1280 x 720, 200k, full
// (fp16 split): 0.202 -> 0.133; 3840 x 2160, 3M, opacity-aware (bf16 split):
// 0.991 -> 0.787; 256 x 256, 10k: 0.055 -> 0.046 ms.
#pragma once

#include "blend_tc.cuh"

namespace gs {
namespace tc {

constexpr int kBwdChunk = 16;
// Default depth of the ring of chunk splats: the deepest that keeps 3 blocks per SM
// for the bf16 and FP8 rows (76.6 KB each).
constexpr int kBwdStages = 4;
constexpr float kTScale = 4096.0f;  // 2^12

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One splat of a chunk, as the scanner packs it: what the row builder, the pixel
// arithmetic (col, idx) and the finishing step read.
struct alignas(16) BwdSplat {
    float r, g, b, cap;    // colour, exponent ceiling min(log2 0.99, log2 o)
    float mx, my, A, B;    // mean, conic
    float C, o, idx;       // conic, opacity, list position
    uint32_t item;         // item index (0xffffffff: padding)
};

// Stage header of the backward pipeline.
struct BwdHdr {
    int tile, seq, n;        // n > 0 chunk, < 0 end
    float gscale;            // 2^(-E-12): dL/dimage scale for the pixel arithmetic
    float bscale;            // 2^(-E): dL/dimage scale in B2
    float undp, uncol;       // 2^E, 2^(E-12): scale of the D2 sums back
    float xc, yc;            // the upper half's reference pixel
    uint32_t goff;           // item index of the view's first Gaussian
    int pad;
};

template <int SS, int V>
struct BwdLayout {
    static constexpr int CH = kBwdChunk;
    static constexpr int A2_ROWS = 96;
    static constexpr int A2_LBO = A2_ROWS / 8 * 128;            // bytes per 8-pixel group: 1536
    static constexpr int A2_BYTES = 16 * A2_LBO + 512;           // + what the M = 128 MMA reads past row 96
    static constexpr int B2_BYTES = 32 * 128 * 2;   // 32 columns x 128 pixels, fp16
    static constexpr int A1_BYTES = 128 * Traits<V>::ROW_BYTES;
    static constexpr int B1_BYTES = 2 * CH * Traits<V>::ROW_BYTES;
    static constexpr int OFF_A2 = 0;
    static constexpr int OFF_B2 = OFF_A2 + 2 * A2_BYTES;
    static constexpr int OFF_A1 = OFF_B2 + B2_BYTES;
    static constexpr int OFF_B1 = OFF_A1 + A1_BYTES;  // 2 stages of coefficient rows
    static constexpr int OFF_SPL = OFF_B1 + 2 * B1_BYTES;  // SS slots of chunk splats
    static constexpr int OFF_GEO = OFF_SPL + SS * CH * (int)sizeof(BwdSplat);  // 2 groups of 32 entries copied ahead
    static constexpr int OFF_SCL = OFF_GEO + 2 * kGeoFields * kGroup * 4;  // FP8 only: row scales
    static constexpr int OFF_BAR = OFF_SCL + (Traits<V>::FP8 ? 2 * CH * 8 : 0);
    // full[SS], empty[SS], bempty[2], tfull[2], tempty[2], a2full[2], m2done[2], drain
    static constexpr int NBAR = 2 * SS + 2 + 2 * kTStages + 5;
    static constexpr int OFF_HDR = OFF_BAR + NBAR * 8;
    static constexpr int OFF_MISC = OFF_HDR + SS * (int)sizeof(BwdHdr);
    static constexpr int BYTES = OFF_MISC + 16;
    static constexpr uint32_t D2_COL = 2 * kTStages * CH;  // 64: after the two exponent stages; 2 x 32
    static constexpr uint32_t TCOLS = 128;
    static_assert(D2_COL + 64 <= TCOLS, "TMEM columns");
};

// 16-byte store into A2 (MN-major: core matrix = 8 pixels x 8 rows; rows
// contiguous, SBO = 128 B between 8-row groups, LBO = 1536 B between 8-pixel groups).
__device__ __forceinline__ void a2_store(uint8_t* A2, int pix, int mblk, const uint4& v) {
    *reinterpret_cast<uint4*>(A2 + (pix >> 3) * 1536 + mblk * 128 + (pix & 7) * 16) = v;
}
// One fp16 element of B2 (K-major: core matrix = 8 columns x 8 pixels).
__device__ __forceinline__ void b2_store(uint8_t* B2, int col, int pix, __half v) {
    *reinterpret_cast<__half*>(B2 + (col >> 3) * 2048 + (pix >> 3) * 128 + (col & 7) * 16 + (pix & 7) * 2) = v;
}

// x0, x1 -> fp16 hi (x0 in the low half) and the fp16 of the remainder.
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(x0, x1);
    const float2 hf = __half22float2(h);
    const float2 r = __fadd2_rn(make_float2(x0, x1), neg2(hf));
    const __half2 l = __floats2half2_rn(r.x, r.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Gradients of one chunk's splats from the sums in D2 (d2: this warp's lanes, the
// chunk's columns), added to the outputs: warps 0 and 1 the geometry and opacity of
// 8 splats each, warp 2 the colours.
__device__ __forceinline__ void finish_chunk(float* dmean2d, float* dconic, float* dopac, float* drgb, const BwdSplat* spl, uint32_t d2, int warp,
                                                 int lane, int p_n, uint32_t p_goff, float p_undp, float p_uncol,
                                                 float p_xc, float p_yc) {
    if (warp < 2) {
        // rows 16 h + 8 s + (j & 7) of splats j = 8 warp + 0..7: monomial moments, hi + lo
        uint32_t v[8];
        tmem_ld_32x32b_x8(d2, v);
        tmem_ld_wait();
        float S[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            S[k] = __uint_as_float(v[k]);
            S[k] += __shfl_xor_sync(0xffffffffu, S[k], 8);
        }
        const int j = 8 * warp + (lane & 7);
        const BwdSplat& f = spl[j];
        const float A = f.A, B = f.B, C = f.C, o = f.o;
        const float xh = f.mx - p_xc;
        float yh = f.my - p_yc;
        if (lane & 16) yh -= 8.0f;  // the lower half's reference
        const float Sx = fmaf(xh, S[5], S[3]), Sy = fmaf(yh, S[5], S[4]);
        float G[6];
        G[0] = -fmaf(A, Sx, B * Sy);
        G[1] = -fmaf(B, Sx, C * Sy);
        G[2] = -0.5f * fmaf(xh, fmaf(xh, S[5], 2.0f * S[3]), S[0]);
        G[3] = -fmaf(xh, fmaf(yh, S[5], S[4]), fmaf(yh, S[3], S[2]));
        G[4] = -0.5f * fmaf(yh, fmaf(yh, S[5], 2.0f * S[4]), S[1]);
        G[5] = S[5] * (o > 0.f ? 1.0f / o : 0.f);
        // both halves of the tile, then one atomic per value and tile
#pragma unroll
        for (int k = 0; k < 6; ++k) G[k] = p_undp * (G[k] + __shfl_xor_sync(0xffffffffu, G[k], 16));
        if (lane < 8 && j < p_n) {
            const size_t g = f.item;
            float* dm = dmean2d + 2 * g;
            red_add(dm, G[0]);
            red_add(dm + 1, G[1]);
            float* dc = dconic + 3 * g;
            red_add(dc, G[2]);
            red_add(dc + 1, G[3]);
            red_add(dc + 2, G[4]);
            red_add(dopac + (f.item - p_goff), G[5]);
        }
    } else {
        // rows (h = lane >> 4, j = lane & 15): w . dL/dimage (hi + lo columns 8..23)
        uint32_t v[16];
        tmem_ld_32x32b_x16(d2 + 8u, v);
        tmem_ld_wait();
        const bool lower = (lane >> 4) != 0;
        float S[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            S[ch] = lower ? __uint_as_float(v[8 + ch]) + __uint_as_float(v[11 + ch])
                          : __uint_as_float(v[ch]) + __uint_as_float(v[3 + ch]);
            S[ch] += __shfl_xor_sync(0xffffffffu, S[ch], 16);
        }
        if (lane < 16 && lane < p_n) {
            float* dr = drgb + 3 * (size_t)spl[lane].item;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) red_add(dr + ch, S[ch] * p_uncol);
        }
    }
}

template <int V, int SS>
__global__ void __launch_bounds__(kThreads, 3) k_blend_tc_bwd(const __grid_constant__ BlendArgs a,
                                                              const __grid_constant__ GradArgs gr) {
    using TR = Traits<V>;
    using LY = BwdLayout<SS, V>;
    constexpr int CH = LY::CH;
    constexpr uint32_t IDESC1 = idesc_f16(TR::FMT, 128, 2 * CH);
    constexpr uint32_t IDESC2 = idesc_f16(0u, 128, 32) | (1u << 15);  // fp16, A MN-major
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sA2 = smem + LY::OFF_A2;
    uint8_t* sB2 = smem + LY::OFF_B2;
    uint8_t* sA1 = smem + LY::OFF_A1;
    uint8_t* sB1 = smem + LY::OFF_B1;
    BwdSplat* sSpl = reinterpret_cast<BwdSplat*>(smem + LY::OFF_SPL);
    float2* sScl = reinterpret_cast<float2*>(smem + LY::OFF_SCL);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + LY::OFF_BAR);
    BwdHdr* sHdr = reinterpret_cast<BwdHdr*>(smem + LY::OFF_HDR);
    uint32_t* sTmem = reinterpret_cast<uint32_t*>(smem + LY::OFF_MISC);
    volatile int* sAbort = reinterpret_cast<volatile int*>(smem + LY::OFF_MISC + 4);
    auto bar_full = [&](int s) { return smem_u32(bars + s); };
    auto bar_empty = [&](int s) { return smem_u32(bars + SS + s); };
    auto bar_bempty = [&](int b) { return smem_u32(bars + 2 * SS + b); };
    auto bar_tfull = [&](int t) { return smem_u32(bars + 2 * SS + 2 + t); };
    auto bar_tempty = [&](int t) { return smem_u32(bars + 2 * SS + 2 + kTStages + t); };
    auto bar_a2full = [&](int b) { return smem_u32(bars + 2 * SS + 2 + 2 * kTStages + b); };
    auto bar_m2done = [&](int b) { return smem_u32(bars + 2 * SS + 2 + 2 * kTStages + 2 + b); };
    const uint32_t bar_drain = smem_u32(bars + 2 * SS + 2 + 2 * kTStages + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool origin = a.ref_origin != 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < SS; ++s) {
            mbar_init(bar_full(s), 1);
            mbar_init(bar_empty(s), kEpiWarps);
        }
        for (int b = 0; b < 2; ++b) mbar_init(bar_bempty(b), 1);
        for (int t = 0; t < kTStages; ++t) {
            mbar_init(bar_tfull(t), 1);
            mbar_init(bar_tempty(t), kEpiWarps);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_a2full(b), kEpiWarps);
            mbar_init(bar_m2done(b), 1);
        }
        mbar_init(bar_drain, 1);
        *sAbort = 0;
        mbar_fence_init();
    }
    // M_p of a 16 x 8 half (A operand of the exponent MMA), as in the forward kernel
    for (int row = threadIdx.x; row < 128; row += kThreads) {
        const float xb = (origin ? 0.f : 7.5f) - (float)lane_col(row);
        const float yb = (origin ? 0.f : 3.5f) - (float)lane_row(row);
        store_mp_row<V>(sA1, row, xb, yb);
    }
    // B2: zero, then the monomial columns 0..5 (the dL/dimage columns are per tile)
    for (int i = threadIdx.x; i < LY::B2_BYTES / 16; i += kThreads)
        reinterpret_cast<uint4*>(sB2)[i] = make_uint4(0, 0, 0, 0);
    for (int i = threadIdx.x; i < 2 * LY::A2_BYTES / 16; i += kThreads)
        reinterpret_cast<uint4*>(sA2)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    if (threadIdx.x < 128) {
        const int pix = threadIdx.x;
        const float xb = (origin ? 0.f : 7.5f) - (float)lane_col(pix);
        const float yb = (origin ? 0.f : 3.5f) - (float)lane_row(pix);
        const float vp[6] = {xb * xb, yb * yb, xb * yb, xb, yb, 1.0f};
#pragma unroll
        for (int i = 0; i < 6; ++i) b2_store(sB2, i, pix, __float2half_rn(vp[i]));
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
    auto fail = [&]() {
        *sAbort = 1;
        atomicOr(a.err, kErrTimeout);
    };

    if (warp < kEpiWarps) {
        // ------------------------------------------------------- epilogue --
        const int r = warp * 32 + lane;
        int cur_seq = -1;
        float2 T = make_float2(0.f, 0.f), Sg = T, ncf = T, g0 = T, g1 = T, g2 = T;
        // pending chunk (finishing step not done yet)
        int p_stage = -1, p_n = 0;
        uint32_t p_c2 = 0;
        float p_undp = 0.f, p_uncol = 0.f, p_xc = 0.f, p_yc = 0.f;
        uint32_t p_goff = 0;
        uint32_t c2 = 0;  // chunks with an A2/MMA2 so far

        auto finish = [&]() -> bool {
            const int pb = (int)(p_c2 & 1u);
            if (!mbar_wait_bounded(bar_m2done(pb), (p_c2 >> 1) & 1u, tmo, sAbort)) {
                fail();
                return false;
            }
            tc_fence_after();
            if (warp < 3)
                finish_chunk(reinterpret_cast<float*>(gr.dmean2d), gr.dconic, gr.dopac, gr.drgb, sSpl + p_stage * CH,
                             tmem + ((uint32_t)(warp * 32) << 16) + LY::D2_COL + (uint32_t)(32 * pb), warp, lane, p_n,
                             p_goff, p_undp, p_uncol, p_xc, p_yc);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_empty(p_stage));
            p_stage = -1;
            return true;
        };

        for (int k = 0;; ++k) {
            const int s = k % SS, t = k % kTStages;
            const uint32_t ps = (uint32_t)(k / SS) & 1u, pt = (uint32_t)(k / kTStages) & 1u;
            if (!mbar_wait_bounded(bar_tfull(t), pt, tmo, sAbort) || !mbar_wait_bounded(bar_full(s), ps, tmo, sAbort)) {
                fail();
                break;
            }
            const BwdHdr hd = sHdr[s];
            const int n = hd.n;
            if (p_stage >= 0 && hd.seq != cur_seq) {
                // B2 changes: the MMA of the pending chunk, of an earlier tile, has read it
                if (!mbar_wait_bounded(bar_m2done((int)(p_c2 & 1u)), (p_c2 >> 1) & 1u, tmo, sAbort)) {
                    fail();
                    break;
                }
            }
            if (n > 0) {
                if (hd.seq != cur_seq) {
                    cur_seq = hd.seq;
                    const int v = view_of(a, hd.tile);
                    const ViewDesc vd = a.views[v];
                    const int lt = hd.tile - vd.tile_begin;
                    const int px = (lt % vd.tiles_x) * kTile + lane_col(r);
                    const int py = (lt / vd.tiles_x) * kTile + lane_row(r);
                    const size_t plane = (size_t)vd.W * vd.H;
                    float gv[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
                    float Tf[2] = {0.f, 0.f}, nc[2] = {0.f, 0.f};
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int y = py + 8 * h;
                        if (px < vd.W && y < vd.H) {
                            const size_t p = (size_t)y * vd.W + px;
                            nc[h] = (float)gr.n_contrib[vd.pix_off + p];
                            Tf[h] = gr.T_final[vd.pix_off + p];
                            const float* dl = gr.dL_dimage + 3 * vd.pix_off + p;
#pragma unroll
                            for (int ch = 0; ch < 3; ++ch) gv[h][ch] = dl[ch * plane];
                        }
#pragma unroll
                        for (int ch = 0; ch < 3; ++ch) {
                            const float bg = gv[h][ch] * hd.bscale;
                            const __half hi = __float2half_rn(bg);
                            const __half lo = __float2half_rn(bg - __half2float(hi));
                            b2_store(sB2, 8 + 8 * h + ch, r, hi);
                            b2_store(sB2, 8 + 8 * h + 3 + ch, r, lo);
                        }
                    }
                    T = make_float2(Tf[0] * kTScale, Tf[1] * kTScale);
                    ncf = make_float2(nc[0], nc[1]);
                    g0 = make_float2(gv[0][0] * hd.gscale, gv[1][0] * hd.gscale);
                    g1 = make_float2(gv[0][1] * hd.gscale, gv[1][1] * hd.gscale);
                    g2 = make_float2(gv[0][2] * hd.gscale, gv[1][2] * hd.gscale);
                    Sg = __ffma2_rn(make_float2(a.bg[0], a.bg[0]), g0,
                                    __ffma2_rn(make_float2(a.bg[1], a.bg[1]), g1, __fmul2_rn(make_float2(a.bg[2], a.bg[2]), g2)));
                }
                tc_fence_after();
                const BwdSplat* spl = sSpl + s * CH;

                // the chunk's splats come back to front: two groups of 8, each group stored
                // to A2[b] as it is done (the MMA that last read A2[b] finished with chunk c2 - 2)
                const int b = (int)(c2 & 1u);
                uint8_t* A2 = sA2 + b * LY::A2_BYTES;
                uint32_t pu[8] = {}, pl[8] = {};  // the group's exponents at both pixels
                auto splat = [&](int j, float2& dp, float2& wt) {
                    const float4 rc = *reinterpret_cast<const float4*>(&spl[j].r);
                    const float idx = spl[j].idx;
                    const float zx = __uint_as_float(pu[j]), zy = __uint_as_float(pl[j]);
                    float2 al;
                    al.x = ex2_approx(fminf(zx, rc.w));
                    al.y = ex2_approx(fminf(zy, rc.w));
                    float2 cull;
                    cull.x = sat(fmaf(al.x, -kCullScale, kAlphaMin * kCullScale));
                    cull.y = sat(fmaf(al.y, -kCullScale, kAlphaMin * kCullScale));
                    al = __ffma2_rn(neg2(al), cull, al);
                    float2 in;
                    in.x = sat(ncf.x - idx);
                    in.y = sat(ncf.y - idx);
                    const float2 aa = __fmul2_rn(al, in);
                    const float2 om = __fadd2_rn(make_float2(1.f, 1.f), neg2(aa));
                    const float2 inv = make_float2(rcp_approx(om.x), rcp_approx(om.y));
                    const float2 Tj = __fmul2_rn(T, inv);
                    wt = __fmul2_rn(aa, Tj);
                    float2 cg;
                    cg.x = __fmaf_rn(rc.z, g2.x, __fmaf_rn(rc.y, g1.x, __fmul_rn(rc.x, g0.x)));
                    cg.y = __fmaf_rn(rc.z, g2.y, __fmaf_rn(rc.y, g1.y, __fmul_rn(rc.x, g0.y)));
                    const float2 diff = __fadd2_rn(cg, neg2(Sg));
                    const float2 dLda = __fmul2_rn(Tj, diff);
                    Sg = __ffma2_rn(aa, diff, Sg);
                    T = Tj;
                    float2 un;  // 0 where alpha is clamped at 0.99
                    un.x = sat(fmaf(zx, -kStopScale, kLog2AlphaMax * kStopScale));
                    un.y = sat(fmaf(zy, -kStopScale, kLog2AlphaMax * kStopScale));
                    dp = __fmul2_rn(dLda, __fmul2_rn(aa, un));
                };
                const uint32_t tb = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(t * 2 * CH);
#pragma unroll 1
                for (int grp = 0; grp < 2; ++grp, spl += 8) {
                    tmem_ld_32x32b_x8(tb + (uint32_t)(8 * grp), pu);
                    tmem_ld_32x32b_x8(tb + (uint32_t)(CH + 8 * grp), pl);
                    tmem_ld_wait();
                    if constexpr (TR::FP8) {  // undo the per-row scaling of the e4m3 operands
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float2 z = __fmul2_rn(make_float2(__uint_as_float(pu[j]), __uint_as_float(pl[j])),
                                                        sScl[t * CH + 8 * grp + j]);
                            pu[j] = __float_as_uint(z.x);
                            pl[j] = __float_as_uint(z.y);
                        }
                    }
                    if (grp == 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_tempty(t));
                    }
                    uint32_t wv[3][2][4];  // [dpow hi, dpow lo, w][h][word]
#pragma unroll
                    for (int pr = 0; pr < 4; ++pr) {
                        float2 dpA, wA, dpB, wB;
                        splat(2 * pr, dpA, wA);
                        splat(2 * pr + 1, dpB, wB);
                        split2(dpA.x, dpB.x, wv[0][0][pr], wv[1][0][pr]);
                        split2(dpA.y, dpB.y, wv[0][1][pr], wv[1][1][pr]);
                        const __half2 hu = __floats2half2_rn(wA.x, wB.x), hl = __floats2half2_rn(wA.y, wB.y);
                        wv[2][0][pr] = *reinterpret_cast<const uint32_t*>(&hu);
                        wv[2][1][pr] = *reinterpret_cast<const uint32_t*>(&hl);
                    }
                    // rows: dpow (h, s, j) = 32 (j >> 3) + 16 h + 8 s + (j & 7); w (h, j) = 64 + 16 h + j
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        a2_store(A2, r, 4 * grp + 2 * h, make_uint4(wv[0][h][0], wv[0][h][1], wv[0][h][2], wv[0][h][3]));
                        a2_store(A2, r, 4 * grp + 2 * h + 1,
                                 make_uint4(wv[1][h][0], wv[1][h][1], wv[1][h][2], wv[1][h][3]));
                        a2_store(A2, r, 8 + 2 * h + grp, make_uint4(wv[2][h][0], wv[2][h][1], wv[2][h][2], wv[2][h][3]));
                    }
                }
                fence_proxy_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_a2full(b));
            }
            // the previous chunk's sums (its MMA has had this whole chunk to finish)
            if (p_stage >= 0 && !finish()) break;
            if (n < 0) break;
            p_stage = s;
            p_n = n;
            p_c2 = c2++;
            p_undp = hd.undp;
            p_uncol = hd.uncol;
            p_xc = hd.xc;
            p_yc = hd.yc;
            p_goff = hd.goff;
        }
    } else if (warp == kEpiWarps) {
        // -------------------------------------------------------- scanner --
        // Walks each tile's list from its largest n_contrib back to the front in groups
        // of 32 entries, one per lane, copied a group ahead by cp.async, and packs the
        // entries that reach a pixel of the tile (splat_reaches) into chunks of CH, back
        // to front.  A tile's header (queue item, range, the largest n_contrib and
        // |dL/dimage| of its pixels, the scales) is worked out for the next tile once the
        // current tile's first group is done, so those loads overlap the current tile's
        // chunks and leave the tile's pixel data in the cache for the epilogue.
        struct TileHead {
            int q, vview, maxnc;
            uint32_t start;
            BwdHdr hd;
        };
        auto head = [&](int qi) {
            TileHead th{};
            th.q = qi;
            if (qi >= a.total_tiles) return th;
            th.hd.tile = tile_at(a, qi * a.shard_count + a.shard_index);
            th.start = a.ranges[2 * th.hd.tile];
            const uint32_t stop = a.ranges[2 * th.hd.tile + 1];
            const int len = stop > th.start ? (int)(stop - th.start) : 0;
            th.vview = view_of(a, th.hd.tile);
            const ViewDesc vd = a.views[th.vview];
            const int lt = th.hd.tile - vd.tile_begin;
            const int x0 = (lt % vd.tiles_x) * kTile, y0 = (lt / vd.tiles_x) * kTile;
            th.hd.xc = (float)x0 + (origin ? 0.5f : 8.0f);
            th.hd.yc = (float)y0 + (origin ? 0.5f : 4.0f);
            th.hd.goff = (uint32_t)(th.vview * a.n_per_view);
            // largest n_contrib and |dL/dimage| over the tile's pixels
            int maxnc = 0;
            float gmax = 0.f;
            const size_t plane = (size_t)vd.W * vd.H;
            for (int p = lane; p < kTilePixels; p += 32) {
                const int px = x0 + (p & 15), py = y0 + (p >> 4);
                if (px < vd.W && py < vd.H) {
                    const size_t pp = (size_t)py * vd.W + px;
                    // T_final is read by the epilogue when the tile starts (n_contrib and
                    // dL/dimage pass through the cache here already)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(gr.T_final + vd.pix_off + pp));
                    maxnc = max(maxnc, gr.n_contrib[vd.pix_off + pp]);
                    const float* dl = gr.dL_dimage + 3 * vd.pix_off + pp;
                    gmax = fmaxf(gmax, fmaxf(fabsf(dl[0]), fmaxf(fabsf(dl[plane]), fabsf(dl[2 * plane]))));
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                maxnc = max(maxnc, __shfl_xor_sync(0xffffffffu, maxnc, o));
                gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
            }
            th.maxnc = min(maxnc, len);
            // 2^E <= gmax < 2^(E + 1), E clamped so that every scale is a normal float
            int E = 0;
            if (gmax > 0.f) E = ((__float_as_int(gmax) >> 23) & 0xff) - 127;
            E = max(-100, min(100, E));
            th.hd.gscale = __int_as_float((127 - E - 12) << 23);
            th.hd.bscale = __int_as_float((127 - E) << 23);
            th.hd.undp = __int_as_float((127 + E) << 23);
            th.hd.uncol = __int_as_float((127 + E - 12) << 23);
            return th;
        };
        const float bx0 = origin ? -15.0f : -7.5f, bx1 = origin ? 0.0f : 7.5f;
        const float by0 = origin ? -7.0f : -3.5f, by1 = origin ? 0.0f : 3.5f;
        float* sGeo = reinterpret_cast<float*>(smem + LY::OFF_GEO) + lane;
        auto fetch = [&](uint32_t g, int n, int v, int slot) {  // n: entries from the group's first on
            if (lane < n) copy_splat_async(a, sGeo + slot * (kGeoFields * kGroup), g, v);
            cp_async_commit();
        };
        int k = 0, slot = 0;
        bool open = false, quit = false, ready = false;  // ready: the tile's first group is in its slot already
        auto acquire = [&]() -> bool {
            if (!mbar_wait_bounded(bar_empty(k % SS), ((uint32_t)(k / SS) & 1u) ^ 1u, tmo, sAbort)) {
                fail();
                return false;
            }
            open = true;
            return !*sAbort;
        };
        auto publish = [&](BwdHdr hd, int seq, int n) {
            hd.seq = seq;
            hd.n = n;
            if (lane == 0) sHdr[k % SS] = hd;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_full(k % SS));
            ++k;
            open = false;
        };
        int q_next = 0;
        // entries of the group at hand, of the one being copied and of the next to copy
        uint32_t gcur = 0, gahead = 0, gn = 0;
        TileHead nxt{};  // no tile yet: the first round only looks one up
        nxt.q = -1;
        for (int seq = -1; !quit; ++seq) {
            const TileHead cur = nxt;
            if (cur.q >= a.total_tiles) {
                if (acquire()) publish(cur.hd, -2, -1);
                break;
            }
            if (lane == 0) q_next = (int)atomicAdd(a.queue, 1u);  // read after this tile's first group
            const int maxnc = cur.maxnc, ng = (maxnc + kGroup - 1) / kGroup;
            int fill = 0;
            // Group gi is taken while group gi + 1, or the next tile's first, is copied;
            // round -1 copies group 0 where the previous tile's last round did not.
            for (int gi = ready || ng == 0 ? 0 : -1; gi < max(ng, 1); ++gi) {
                const bool more = gi + 1 < ng;
                // the next tile is known from the first group on, its entries from the last but one
                const bool over = !more && gi > 1 && nxt.q < a.total_tiles && nxt.maxnc > 0;
                gcur = gahead;
                if (more || over) {
                    fetch(gn, more ? maxnc - (gi + 1) * kGroup : nxt.maxnc, more ? cur.vview : nxt.vview, slot ^ 1);
                    gahead = gn;
                }
                ready = over;
                // entries to copy next: entry e of a list counts back from its last contributing position
                {
                    const bool mine = gi + 2 < ng;
                    const int left = mine ? maxnc - (gi + 2) * kGroup : gi > 0 && more && nxt.q < a.total_tiles ? nxt.maxnc : 0;
                    if (lane < left) gn = a.ids[(mine ? cur.start : nxt.start) + (uint32_t)(left - 1 - lane)];
                }
                if (gi >= 0 && ng > 0) {
                    if (more || over) cp_async_wait<1>();
                    else cp_async_wait<0>();
                    const int e = gi * kGroup + lane;
                    const float* d = sGeo + slot * (kGeoFields * kGroup);
                    const float mx = d[0], my = d[kGroup], A = d[2 * kGroup], B = d[3 * kGroup], C = d[4 * kGroup];
                    const float o = d[5 * kGroup];
                    const float l2o = log2_opacity(o);
                    const bool keep = e < maxnc && splat_reaches<V>(A, B, C, l2o, mx - cur.hd.xc, my - cur.hd.yc, bx0,
                                                                    bx1, by0, by1);
                    const unsigned kb = __ballot_sync(0xffffffffu, keep);
                    int pos = keep ? fill + __popc(kb & ((1u << lane) - 1u)) : -1;
                    fill += __popc(kb);
                    const bool last = gi + 1 == ng;
                    while (fill > 0) {
                        if (!open && !acquire()) {
                            quit = true;
                            break;
                        }
                        float4* w = reinterpret_cast<float4*>(sSpl + (k % SS) * CH);
                        if (pos >= 0 && pos < CH) {
                            w[3 * pos] = make_float4(d[6 * kGroup], d[7 * kGroup], d[8 * kGroup],
                                                     fminf(l2o, kLog2AlphaMax));
                            w[3 * pos + 1] = make_float4(mx, my, A, B);
                            w[3 * pos + 2] = make_float4(C, o, (float)(maxnc - 1 - e), __uint_as_float(gcur));
                        }
                        if (fill < CH && !last) break;
                        if (lane >= fill && lane < CH) {  // the tile's last chunk is padded with dead splats
                            w[3 * lane] = make_float4(0.f, 0.f, 0.f, kDeadPower);
                            w[3 * lane + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
                            w[3 * lane + 2] = make_float4(0.f, 0.f, 0.f, __uint_as_float(0xffffffffu));
                        }
                        publish(cur.hd, seq, min(fill, CH));
                        fill = max(fill - CH, 0);
                        pos -= CH;
                    }
                    if (quit) break;
                }
                if (gi == 0) nxt = head(__shfl_sync(0xffffffffu, q_next, 0));
                if (more || over) slot ^= 1;
            }
            if (quit) break;
            const int skip = ready ? kGroup : 0;  // its first group is under way
            if (nxt.q < a.total_tiles && lane + skip < nxt.maxnc)
                gn = a.ids[nxt.start + (uint32_t)(nxt.maxnc - 1 - skip - lane)];
        }
        cp_async_wait<0>();
    } else {
        // ---------------------------------------------- row builder, MMAs --
        const float bx0 = origin ? -15.0f : -7.5f, bx1 = origin ? 0.0f : 7.5f;
        const float by0 = origin ? -7.0f : -3.5f, by1 = origin ? 0.0f : 3.5f;
        const uint32_t aA1 = smem_u32(sA1), aB2 = smem_u32(sB2);
        for (int k = 0;; ++k) {
            const int s = k % SS, t = k % 2;  // t: coefficient rows and exponents (kTStages = 2)
            if (!mbar_wait_bounded(bar_full(s), (uint32_t)(k / SS) & 1u, tmo, sAbort) ||
                !mbar_wait_bounded(bar_bempty(t), ((uint32_t)(k / 2) & 1u) ^ 1u, tmo, sAbort)) {
                fail();
                break;
            }
            const BwdHdr& hd = sHdr[s];
            const int n = hd.n;
            if (n > 0) {
                // lanes 0..15: upper reference rows, 16..31: lower, for splat j = lane & 15
                const int j = lane & 15;
                const bool upper = lane < 16;
                uint8_t* mB = sB1 + t * LY::B1_BYTES;
                float v[6] = {0.f, 0.f, 0.f, 0.f, 0.f, kDeadPower};
                if (j < n) {
                    const BwdSplat& f = sSpl[s * CH + j];
                    const float yh = f.my - hd.yc;
                    coeff_row<TR::HALF>(f.A, f.B, f.C, log2_opacity(f.o), f.mx - hd.xc, upper ? yh : yh - 8.0f, bx0, bx1,
                                        by0, by1, v);
                }
                const float rs = store_coeff_row<V>(mB, upper ? j : CH + j, v);
                if constexpr (TR::FP8) reinterpret_cast<float*>(sScl + t * CH + j)[upper ? 0 : 1] = rs;
            }
            fence_proxy_async_smem();
            if (!mbar_wait_bounded(bar_tempty(t), ((uint32_t)(k / 2) & 1u) ^ 1u, tmo, sAbort)) {
                fail();
                break;
            }
            __syncwarp();
            if (lane == 0) {
                if (n > 0) {
                    tc_fence_after();
                    const uint32_t aB1 = smem_u32(sB1 + t * LY::B1_BYTES);
#pragma unroll
                    for (int ks = 0; ks < TR::KSTEPS; ++ks) {
                        const uint64_t ad = smem_desc(aA1 + (uint32_t)(ks * 256), 128, TR::SBO);
                        const uint64_t bd = smem_desc(aB1 + (uint32_t)(ks * 256), 128, TR::SBO);
                        tc_mma<V>(tmem + (uint32_t)(t * 2 * CH), ad, bd, IDESC1, ks > 0 ? 1u : 0u);
                    }
                    tc_commit(bar_tfull(t));
                    tc_commit(bar_bempty(t));
                } else {
                    mbar_arrive(bar_tfull(t));
                }
            }
            __syncwarp();
            // the previous chunk's sums, once its A2 is written
            if (k > 0) {
                const int pb = (k - 1) & 1;
                if (!mbar_wait_bounded(bar_a2full(pb), (uint32_t)((k - 1) >> 1) & 1u, tmo, sAbort)) {
                    fail();
                    break;
                }
                if (lane == 0) {
                    tc_fence_after();
                    const uint32_t aA2 = smem_u32(sA2 + pb * LY::A2_BYTES);
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint64_t ad = smem_desc(aA2 + (uint32_t)(ks * 2 * LY::A2_LBO), LY::A2_LBO, 128);
                        const uint64_t bd = smem_desc(aB2 + (uint32_t)(ks * 256), 128, 2048);
                        tc_mma_f16(tmem + LY::D2_COL + (uint32_t)(32 * pb), ad, bd, IDESC2, ks > 0 ? 1u : 0u);
                    }
                    tc_commit(bar_m2done(pb));
                }
                __syncwarp();
            }
            if (n < 0) break;
        }
        if (lane == 0) {
            // every MMA this thread issued has finished before TMEM is freed
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

template <int V, int SS>
cudaError_t launch_bwd_inst(const BlendArgs& a, const GradArgs& g, cudaStream_t s) {
    using LY = BwdLayout<SS, V>;
    constexpr int bytes = LY::BYTES;
    auto kern = k_blend_tc_bwd<V, SS>;
    static std::mutex mu;
    static LaunchShape cache;
    LaunchShape sh;
    const cudaError_t es = cached_shape(mu, cache, sh, [&](LaunchShape& r) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        // all of the SM's unified L1/shared storage as shared memory, so that
        // the residency computed below is what the hardware grants
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100)) != cudaSuccess)
            return e;
        int dev = 0, smem_sm = 0;
        cudaFuncAttributes fa{};
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess)
            return e;
        if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
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
    const int items = a.total_tiles;
    const int grid = items < sh.per_sm * sh.sms ? (items > 0 ? items : 1) : sh.per_sm * sh.sms;
    kern<<<grid, kThreads, bytes, s>>>(a, g);
    count_launches();
    return cudaGetLastError();
}

// stages 0: the default; otherwise one of kBwdStagesBuilt
template <int V, int I = 0>
cudaError_t launch_bwd_stages(const BlendArgs& a, const GradArgs& g, int stages, cudaStream_t s) {
    if constexpr (I < (int)(sizeof(kBwdStagesBuilt) / sizeof(int))) {
        if ((stages == 0 ? kBwdStages : stages) == kBwdStagesBuilt[I])
            return launch_bwd_inst<V, kBwdStagesBuilt[I]>(a, g, s);
        return launch_bwd_stages<V, I + 1>(a, g, stages, s);
    }
    return cudaErrorInvalidValue;
}

// Instantiated per variant in blend_tc_bwd_v<V>.cu
template <int V>
cudaError_t launch_bwd_variant(const BlendArgs& a, const GradArgs& g, int stages, cudaStream_t s);
template <>
cudaError_t launch_bwd_variant<1>(const BlendArgs&, const GradArgs&, int, cudaStream_t);
template <>
cudaError_t launch_bwd_variant<2>(const BlendArgs&, const GradArgs&, int, cudaStream_t);
template <>
cudaError_t launch_bwd_variant<3>(const BlendArgs&, const GradArgs&, int, cudaStream_t);
template <>
cudaError_t launch_bwd_variant<4>(const BlendArgs&, const GradArgs&, int, cudaStream_t);
template <>
cudaError_t launch_bwd_variant<5>(const BlendArgs&, const GradArgs&, int, cudaStream_t);

}  // namespace tc
}  // namespace gs
