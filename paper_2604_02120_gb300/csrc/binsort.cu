// Duplication and sorting stages (Sec. 2.1 (b), (c)).
//
// The result equals a stable sort of (tile << 32 | depth_bits) keys emitted in
// Gaussian order, i.e. every tile's list ordered by (depth bits, Gaussian
// index).  It is produced without sorting the instances themselves:
//   1. stable LSD radix sort of the N items by depth bits (32-bit keys);
//   2. coarse duplication in that depth order: one (supertile, item) pair
//      per supertile (4 x 4 tiles) holding at least one of the item's
//      instances (about an eighth of the instances), with the pair's 16-bit
//      mask of those instances, and the count of all instances;
//   3. stable LSD radix sort of those pairs by supertile id, so each
//      supertile's items are contiguous and in depth order;
//   4. the instances of each tile counted from the pairs' masks, a scan over
//      the tiles gives every tile's range, and one block per supertile walks
//      its pairs writing each instance's id once, at its tile's next
//      position: a stable per-tile compaction, so every list keeps the depth
//      (then index) order of step 1.
// Each instance is written once (4 bytes of id, plus its key if asked for)
// instead of being duplicated and moved by a radix pass per 8 bits of tile id.
//
// Every radix pass is one launch.  The digit histograms of all passes are
// counted up front by the kernel that produces the keys (the counts of an LSD
// pass do not depend on the order the previous pass leaves), and each block
// finds where its digits go among the blocks before it by decoupled
// look-back: blocks take tile numbers from an atomic ticket in the order they
// start, publish their per-digit counts, then add up their predecessors'
// published counts until one carries an inclusive prefix.  A block only waits
// for blocks that started before it, so the waits always end; each is still
// bounded in time.  One that gives up sets the timeout bit of the error word and
// the call's own flag (GiveUp): its kernel goes on with a prefix too small, so
// everything after it holds holes and stale words, which every kernel up to the
// pair sort bounds before it writes, and the tile counts are left at zero: every
// list comes out empty, and nothing is read through ids that were never written.
// The scan of coarse counts in depth order is done the same way inside the
// duplication kernels (k_dup_rect for full rectangles, k_dup_coarse for
// opacity-aware lists), so the whole stage is
//   memset, keys, 4 depth passes, coarse duplicate, ceil(bits / 8) supertile
//   passes, tile counts, tile scan, fine write.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "tight.cuh"

namespace gs {
namespace {

constexpr int kThreads = 256;
constexpr int kDupTile = kThreads;          // items per tile of the opacity-aware duplication
constexpr int kMaxPasses = 8;               // 4 depth passes + up to 4 tile-id passes
#ifndef GS_LOOKBACK_LIMIT_NS
#define GS_LOOKBACK_LIMIT_NS 2000000000ull  // 2 s; a test builds the file with 0
#endif
constexpr uint64_t kLookbackLimitNs = GS_LOOKBACK_LIMIT_NS;

// Where a look-back that gives up says so: the device's error word and the flag
// of this call, in its workspace (k_pair_masks reads it).
struct GiveUp {
    unsigned *err, *call;
    __device__ __forceinline__ void set() const {
        atomicOr(err, kErrTimeout);
        atomicOr(call, 1u);
    }
};

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
// Items per thread of a radix pass: tiles of 1024 up to 2^18 items, so that a
// small pass reaches all SMs; of 2048 up to 9 x 2^17 items, 576 tiles, the most that
// 4 blocks on each of 152 SMs take in one wave (a pass of 1M: 13.5 us, in tiles of
// 1024 17.4); of 4096 beyond, which halves the look-back.  (A literal: the workspace
// size is asked for without a device.)
inline int pass_items(uint64_t n) { return n <= 1u << 18 ? 4 : n <= 9u << 17 ? 8 : 16; }
// An upper bound of the radix tiles of a pass over at most m items; it grows with m
// (a pass of fewer items can have more tiles than one just past a step of
// pass_items: the first 2^20 items are counted in the smallest tiles).
inline int64_t radix_tiles_max(int64_t m) {
    return std::max(cdiv(std::min<int64_t>(m, 1 << 20), kThreads * 4), cdiv(m, kThreads * pass_items(m)));
}

// ---------------------------------------------------------- block helpers --

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// exclusive scan of one value per thread across a block of NT threads;
// returns the thread's exclusive prefix, `total` receives the block's sum.
template <typename T, int NT>
__device__ __forceinline__ T block_excl_scan(T v, T& total, T* s_warp /*[NT/32 + 1]*/) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = warp_incl_scan(v);
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < NT / 32 ? s_warp[lane] : T(0);
        T wi = warp_incl_scan(w);
        if (lane < NT / 32) s_warp[lane] = wi - w;
        if (lane == NT / 32 - 1) s_warp[NT / 32] = wi;
    }
    __syncthreads();
    T res = inc - v + s_warp[warp];
    total = s_warp[NT / 32];
    __syncthreads();
    return res;
}

// ------------------------------------------------------ look-back status --
//
// A status word holds a tag in bits [56, 64) and a count in bits [0, 56).
// Pass p publishes tag 2p + 1 (this block's own count) and then 2p + 2 (the
// inclusive prefix up to and including this block); any other tag (zero after
// the clear, or a value an earlier pass left in the same word) means "not yet".

constexpr uint64_t kValMask = (uint64_t(1) << 56) - 1;

__device__ __forceinline__ void st_status(unsigned long long* p, uint32_t tag, uint64_t v) {
    const unsigned long long w = ((unsigned long long)tag << 56) | (v & kValMask);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ unsigned long long ld_status(const unsigned long long* p) {
    unsigned long long w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
}

// Sum of the counts of groups [0, g) for one digit, walking back from g - 1
// until an inclusive prefix is found.  W predecessors are read per round trip;
// the ready ones nearest to this group are consumed, up to the first inclusive
// prefix.
__device__ __forceinline__ uint64_t lookback_serial(const unsigned long long* status, int64_t tile, int stride,
                                                    int d, uint32_t tag_agg, const GiveUp& gu) {
    constexpr int W = 4;
    uint64_t prefix = 0, t0 = 0;
    int64_t j = tile - 1;
    while (j >= 0) {
        unsigned long long w[W];
#pragma unroll
        for (int q = 0; q < W; ++q)
            w[q] = j - q >= 0 ? ld_status(status + (size_t)(j - q) * stride + d)
                              : ((unsigned long long)(tag_agg + 1) << 56);  // before tile 0: 0
        int used = 0;
        bool done = false, blocked = false;
#pragma unroll
        for (int q = 0; q < W; ++q) {
            if (done || blocked) continue;
            const uint32_t tag = (uint32_t)(w[q] >> 56);
            if (tag == tag_agg || tag == tag_agg + 1) {
                prefix += w[q] & kValMask;
                ++used;
                done = tag == tag_agg + 1;
            } else {
                blocked = true;
            }
        }
        if (done) break;
        j -= used;
        if (blocked) {
            __nanosleep(100);
            const uint64_t now = globaltimer_ns();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > kLookbackLimitNs) {
                gu.set();
                break;
            }
        }
    }
    return prefix;
}

// The radix passes look back over two levels.  A tile publishes its digit
// counts once (rows: 256 words of 32 bits, tag in bits [27, 32)) and adds up
// the rows before it in its group of kGroup tiles; the group's last tile
// publishes the group's counts and, after its own look-back, their inclusive
// prefix (64-bit words as above), and everybody looks back over groups.  With
// one level a tile walked over 150 rows (600 tiles are in flight, and rows turn
// inclusive only as walks end) and the reading, not the waiting, took longer
// than the tile's own work: windows of 16 or 32 rows were slower than 8.  Per
// pass, 200k / 1M / 3M / 14M items: 10.9 / 23.4 / 32 / 120 us with one level,
// 8.9 / 17.7 / 31 / 115 with two (16 tiles in a group, windows of 4), 25.5 and
// 77 for the large ones with the ranking below and groups of 8.
constexpr int kGroup = 8;
constexpr int kRowTagBit = 27;
__device__ __forceinline__ uint32_t group_sum(const uint32_t* rows, int64_t tile, int d, uint32_t tag, const GiveUp& gu) {
    const int m = (int)(tile % kGroup);
    const uint32_t* p = rows + (size_t)(tile - m) * 256 + d;
    uint64_t t0 = 0;
    for (;;) {
        uint32_t w[kGroup - 1];
#pragma unroll
        for (int q = 0; q < kGroup - 1; ++q) {
            w[q] = tag << kRowTagBit;
            if (q < m) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w[q]) : "l"(p + q * 256) : "memory");
        }
        uint32_t sum = 0;
        bool ready = true;
#pragma unroll
        for (int q = 0; q < kGroup - 1; ++q) {
            ready = ready && (w[q] >> kRowTagBit) == tag;
            sum += w[q] & ((1u << kRowTagBit) - 1);
        }
        if (ready) return sum;
        __nanosleep(100);
        const uint64_t now = globaltimer_ns();
        if (t0 == 0) {
            t0 = now;
        } else if (now - t0 > kLookbackLimitNs) {
            gu.set();
            return 0;
        }
    }
}

// The same for a single count per tile, by one warp over windows of 32
// predecessors (lane l reads tile j - l).  Every lane returns the prefix.
__device__ __forceinline__ uint64_t lookback_warp(const unsigned long long* status, int64_t tile, uint32_t tag_agg,
                                                  const GiveUp& gu) {
    const int lane = threadIdx.x & 31;
    uint64_t prefix = 0, t0 = 0;
    int64_t j = tile - 1;
    while (j >= 0) {
        const int64_t jj = j - lane;
        const unsigned long long w =
            jj >= 0 ? ld_status(status + jj) : ((unsigned long long)(tag_agg + 1) << 56);  // before tile 0: 0
        const uint32_t tag = (uint32_t)(w >> 56);
        const unsigned inc = __ballot_sync(0xffffffffu, tag == tag_agg + 1);
        const unsigned notready = __ballot_sync(0xffffffffu, tag != tag_agg && tag != tag_agg + 1);
        const int first_inc = inc ? __ffs(inc) - 1 : 32;
        const unsigned needed = first_inc == 32 ? 0xffffffffu : (0xffffffffu >> (31 - first_inc));
        if (notready & needed) {
            const uint64_t now = globaltimer_ns();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > kLookbackLimitNs) {
                if (lane == 0) gu.set();
                break;
            }
            continue;
        }
        uint64_t v = lane <= first_inc ? (uint64_t)(w & kValMask) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        prefix += v;
        if (first_inc < 32) break;
        j -= 32;
    }
    return prefix;
}

// s_h[bin] += 1 for every active lane: one atomic when the lanes agree on the
// bin (the high digits of nearby keys usually do, and same-address shared
// atomics serialise), else one per lane.
__device__ __forceinline__ void hist_add(uint32_t* s_h, uint32_t bin) {
    const unsigned act = __activemask();
    const int first = __ffs(act) - 1;
    const uint32_t b0 = __shfl_sync(act, bin, first);
    if (__all_sync(act, bin == b0)) {
        if ((int)(threadIdx.x & 31) == first) atomicAdd(&s_h[bin], (uint32_t)__popc(act));
    } else {
        atomicAdd(&s_h[bin], 1u);
    }
}

// Item count of a pass: the host value, or min(*n_dev, host value) in graph mode.
__device__ __forceinline__ uint32_t pass_count(uint32_t n_host, const uint64_t* n_dev) {
    if (n_dev == nullptr) return n_host;
    const uint64_t v = *n_dev;
    return v < n_host ? (uint32_t)v : n_host;
}

// ------------------------------------------------------------ radix pass --

// One stable pass on bits [shift, shift + 8).  The block takes the next tile
// of TILE items from the ticket; warp w owns the contiguous items
// [w * 32 ITEMS, (w + 1) * 32 ITEMS) walked in rounds of 32, so lane order is
// input order, and each item's rank among equal digits comes from the lanes
// with the same digit: FULL, for digits of more than 4 significant bits, ors the
// lane's bit into a word per warp and digit in shared memory and reads it back
// (14M items 117 -> 77 us against eight ballots, whose bit tests filled 69% of
// the ALU); else __match_any_sync, cheaper while few digits occur (the last
// pass over a short key: 70 us, with the shared words 86, as lanes then collide
// on them).  The ranking runs once: it keeps each item's rank among
// its warp's items of the same digit, so placing an item needs only its warp's
// start of the digit.  Items are placed in shared memory in digit order, then
// written so that consecutive threads write consecutive addresses of each
// digit's run.  hist holds the pass's global digit counts.
template <int ITEMS, bool FULL>
__global__ void __launch_bounds__(kThreads, 4) k_onesweep(const uint32_t* __restrict__ kin,
                                                       const uint32_t* __restrict__ vin, uint32_t n_host,
                                                       const uint64_t* __restrict__ n_dev, int shift, int pass_id,
                                                       const uint32_t* __restrict__ hist, uint32_t* tickets,
                                                       unsigned long long* status, uint32_t* __restrict__ kout,
                                                       uint32_t* __restrict__ vout, GiveUp gu) {
    constexpr int TILE = kThreads * ITEMS;
    __shared__ uint32_t s_w[kThreads / 32][256];  // per-warp digit counts, then local bases
    __shared__ uint32_t s_dbase[256];              // block-local start of each digit's run
    __shared__ uint32_t s_goff[256];               // global start of each digit's run
    __shared__ uint32_t s_warp[kThreads / 32 + 1];
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_buf[2 * TILE];
    uint32_t *s_key = s_buf, *s_val = s_buf + TILE;
    uint32_t* s_peers = s_buf;  // while ranking: per warp and digit, the lanes of the round that have it
    static_assert(2 * TILE >= kThreads / 32 * 256);
    const uint32_t n = pass_count(n_host, n_dev);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // persistent: the block takes tiles until the pass is done (a tile's
    // look-back waits only on tiles ticketed before it, which blocks are
    // already processing)
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(&tickets[pass_id], 1u);
        for (int i = threadIdx.x; i < (kThreads / 32) * 256; i += kThreads) {
            (&s_w[0][0])[i] = 0;
            if constexpr (FULL) s_peers[i] = 0;
        }
        __syncthreads();
        const uint32_t tile = s_tile;
        const int64_t bbase = (int64_t)tile * TILE;
        if (bbase >= n) return;  // uniform over the block; no later tile is needed either
        const int cnt = (int)((int64_t)n - bbase < TILE ? (int64_t)n - bbase : TILE);
        const int wbase = warp * (ITEMS * 32);
        uint32_t k[ITEMS];
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            const int i = wbase + r * 32 + lane;
            k[r] = i < cnt ? kin[bbase + i] : 0u;
        }
        const unsigned lt = (1u << lane) - 1u;
        // each item's rank among the warp's items with its digit (input order),
        // 16 bits per item: the warp's running count before this round plus the
        // lower lanes of the round with the same digit
        uint32_t rank[(ITEMS + 1) / 2];
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            const bool valid = wbase + r * 32 + lane < cnt;
            const uint32_t d = (k[r] >> shift) & 0xFFu;
            uint32_t* slot = s_peers + warp * 256 + d;
            uint32_t peers;
            if constexpr (FULL) {
                if (valid) atomicOr(slot, 1u << lane);
                __syncwarp();
                peers = *slot;
            } else {
                peers = __match_any_sync(0xffffffffu, valid ? d : 0x100u + lane);
            }
            const uint32_t before = s_w[warp][d];
            __syncwarp();
            if (valid && (peers & lt) == 0) {
                s_w[warp][d] = before + __popc(peers);
                if constexpr (FULL) *slot = 0;
            }
            __syncwarp();
            const uint32_t rk = before + __popc(peers & lt);
            if (r & 1)
                rank[r >> 1] |= rk << 16;
            else
                rank[r >> 1] = rk;
        }
        __syncthreads();
        {
            const int d = threadIdx.x;
            uint32_t c = 0;
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) c += s_w[w][d];
            // rows of 32 bits, then the full groups' rows: within the 256 64-bit words per tile
            uint32_t* rows = reinterpret_cast<uint32_t*>(status);
            unsigned long long* groups = status + ((size_t)n + TILE - 1) / TILE * 128;
            const uint32_t tag_agg = 2u * pass_id + 1u;
            asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(rows + (size_t)tile * 256 + d),
                         "r"(tag_agg << kRowTagBit | c)
                         : "memory");  // publish first, successors may be waiting
            uint32_t total;
            const uint32_t db = block_excl_scan<uint32_t, kThreads>(c, total, s_warp);
            const uint32_t gstart = block_excl_scan<uint32_t, kThreads>(hist[d], total, s_warp);
            uint32_t prefix = 0;
            const int64_t g = tile / kGroup;
            const bool closes = tile % kGroup == kGroup - 1;
            if (tile % kGroup) prefix = group_sum(rows, tile, d, tag_agg, gu);
            if (closes) st_status(groups + (size_t)g * 256 + d, g == 0 ? tag_agg + 1 : tag_agg, prefix + c);
            if (g > 0) {
                prefix += (uint32_t)lookback_serial(groups, g, 256, d, tag_agg, gu);
                if (closes) st_status(groups + (size_t)g * 256 + d, tag_agg + 1, prefix + c);
            }
            s_dbase[d] = db;
            s_goff[d] = gstart + prefix;
            uint32_t run = db;
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) {
                const uint32_t cw = s_w[w][d];
                s_w[w][d] = run;
                run += cw;
            }
        }
        // the values are needed only from here on (fewer registers live across the look-back)
        uint32_t v[ITEMS];
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            const int i = wbase + r * 32 + lane;
            v[r] = i < cnt ? vin[bbase + i] : 0u;
        }
        __syncthreads();
        // s_w[w][d] now holds warp w's block-local start of digit d
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (wbase + r * 32 + lane < cnt) {
                const uint32_t d = (k[r] >> shift) & 0xFFu;
                const uint32_t pos = s_w[warp][d] + ((rank[r >> 1] >> (16 * (r & 1))) & 0xFFFFu);
                s_key[pos] = k[r];
                s_val[pos] = v[r];
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < cnt; i += kThreads) {
            const uint32_t key = s_key[i];
            const uint32_t d = (key >> shift) & 0xFFu;
            const uint32_t g = s_goff[d] + (uint32_t)i - s_dbase[d];
            if (g < n) {  // always, unless a look-back gave up (timeout bit set)
                kout[g] = key;
                vout[g] = s_val[i];
            }
        }
        __syncthreads();  // shared memory is reused by the next tile
    }
}

struct PassScratch {
    const uint32_t* hist;  // [kMaxPasses][256] digit counts
    uint32_t* tickets;     // [kMaxPasses]
    unsigned long long* status;
    GiveUp gu;
};

// Stable LSD sort of (k[0], v[0]) on bits [0, bits) with pass ids
// first_pass, first_pass + 1, ...; the result ends in buffer *which.  n_host
// sizes the grid; in graph mode the passes sort min(*n_dev, n_host) items.
cudaError_t radix_sort(uint32_t* k[2], uint32_t* v[2], uint32_t n_host, const uint64_t* n_dev, int bits,
                       int first_pass, const PassScratch& ps, int* which, cudaStream_t s) {
    int cur = 0;
    const int items = pass_items(n_host);
    int dev = 0, sms = 0;
    cudaError_t ea = cudaGetDevice(&dev);
    if (ea == cudaSuccess) ea = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (ea != cudaSuccess) return ea;
    // persistent blocks: at most 4 per SM (a graph-mode grid sized for the capacity would
    // otherwise start many blocks that only find the pass done)
    const int nblk = (int)std::min<int64_t>(cdiv(n_host, (int64_t)kThreads * items), 4 * (int64_t)sms);
    for (int p = 0, shift = 0; shift < bits; ++p, shift += 8) {
        const int id = first_pass + p;
        const bool full = bits - shift > 4;  // k_onesweep: how equal digits are found
        auto kern = items == 4   ? (full ? k_onesweep<4, true> : k_onesweep<4, false>)
                    : items == 8 ? (full ? k_onesweep<8, true> : k_onesweep<8, false>)
                                 : (full ? k_onesweep<16, true> : k_onesweep<16, false>);
        kern<<<nblk, kThreads, 0, s>>>(k[cur], v[cur], n_host, n_dev, shift, id, ps.hist + 256 * id, ps.tickets,
                                       ps.status, k[cur ^ 1], v[cur ^ 1], ps.gu);
        count_launches();
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        cur ^= 1;
    }
    *which = cur;
    return cudaSuccess;
}

// ------------------------------------------------------ duplicate/finalize --

// ----------------------------------------------- opacity-aware membership --
//
// With sv.conic and sv.power_min set, tiles are kept by the rule of tight.cuh.
__device__ __forceinline__ TightRows item_tight_rows(const SortViews& sv, const float2* mean2d, uint32_t item) {
    const float2 m = mean2d[item];
    const uint32_t g = item - (item / (uint32_t)sv.n_per_view) * (uint32_t)sv.n_per_view;
    return tight_rows(m.x, m.y, sv.conic[3 * (size_t)item], sv.conic[3 * (size_t)item + 1],
                      sv.conic[3 * (size_t)item + 2], sv.power_min[g]);
}

// ------------------------------------------------------------ supertiles --
//
// A supertile is 4 x 4 tiles of one view.  Within one supertile row an item's
// supertiles are the union of [f / 4, l / 4] over the runs [f, l] of its (at
// most 4) tile rows there: up to 4 intervals, merged after a sorting network
// on their starts (registers only).  Every supertile counted holds at least
// one of the item's instances.
constexpr int kSuper = 4;

struct Iv {
    int lo, hi;  // empty: lo > hi (lo = INT_MAX sorts last)
};
__device__ __forceinline__ void iv_swap(Iv& a, Iv& b) {
    if (b.lo < a.lo) {
        const Iv t = a;
        a = b;
        b = t;
    }
}
// emit(lo, hi) for each maximal interval of the union; returns its size
template <class F>
__device__ __forceinline__ int iv_union4(Iv a, Iv b, Iv c, Iv d, F emit) {
    iv_swap(a, b);
    iv_swap(c, d);
    iv_swap(a, c);
    iv_swap(b, d);
    iv_swap(b, c);
    if (a.lo > a.hi) return 0;
    int n = 0, clo = a.lo, chi = a.hi;
    auto step = [&](const Iv& x) {
        if (x.lo > x.hi) return;
        if (x.lo <= chi + 1) {
            chi = max(chi, x.hi);
        } else {
            emit(clo, chi);
            n += chi - clo + 1;
            clo = x.lo;
            chi = x.hi;
        }
    };
    step(b);
    step(c);
    step(d);
    emit(clo, chi);
    return n + chi - clo + 1;
}

// The four tile-row runs of one supertile row (f > l: none).
struct Runs4 {
    int f[kSuper], l[kSuper];
};

// The 16-bit mask of supertile column sx within a supertile row's runs: bit
// 4 k + c for tile (4 sx + c) of the row's k-th tile row.
__device__ __forceinline__ uint32_t runs_mask(const Runs4& rr, int sx) {
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < kSuper; ++k) {
        const int a = max(rr.f[k], sx * kSuper), b = min(rr.l[k], sx * kSuper + kSuper - 1);
        if (a <= b) m |= ((1u << (b - a + 1)) - 1u) << (k * kSuper + a - sx * kSuper);
    }
    return m;
}

// The four tile-row runs of supertile row sy within the rectangle [x0, x1] x
// [y0, y1], and in *fine their instance count.
__device__ __forceinline__ Runs4 row_runs(const TightRows& t, int sy, int x0, int x1, int y0, int y1,
                                          uint32_t* fine) {
    Runs4 rr;
#pragma unroll
    for (int k = 0; k < kSuper; ++k) {
        const int y = sy * kSuper + k;
        int f, l;
        tight_row(t, y, x0, x1, f, l);
        if (y < y0 || y > y1) l = f - 1;
        rr.f[k] = f;
        rr.l[k] = l;
        *fine += (uint32_t)max(l - f + 1, 0);
    }
    return rr;
}

// The supertile columns holding an instance of the runs rr (emit(lo, hi) per
// maximal interval, in increasing order); returns their count.
template <class F>
__device__ __forceinline__ int runs_union(const Runs4& rr, F emit) {
    Iv r[kSuper];
#pragma unroll
    for (int k = 0; k < kSuper; ++k)
        r[k] = rr.f[k] <= rr.l[k] ? Iv{rr.f[k] / kSuper, rr.l[k] / kSuper} : Iv{0x7fffffff, -1};
    return iv_union4(r[0], r[1], r[2], r[3], emit);
}

// Per item: its depth key and index (the depth sort's input) and the keys'
// four digit histograms (pass ids 0..3).  Also clears the tile ranges and the
// look-back status words of the depth sort (clear) and of the duplication
// (clear2).
constexpr int kKeyItems = 4;
__global__ void __launch_bounds__(kThreads) k_keys(int n_items, const float* __restrict__ depth,
                                                   uint32_t* __restrict__ dkey, uint32_t* __restrict__ dval,
                                                   uint32_t* __restrict__ hist, uint4* __restrict__ clear,
                                                   size_t clear_n, unsigned long long* __restrict__ clear2,
                                                   size_t clear2_n, uint32_t* __restrict__ ranges, size_t ranges_n) {
    __shared__ uint32_t s_h[4 * 256];
    for (int i = threadIdx.x; i < 4 * 256; i += kThreads) s_h[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (kThreads * kKeyItems) + threadIdx.x;
    uint32_t key[kKeyItems];
#pragma unroll
    for (int q = 0; q < kKeyItems; ++q) {
        const int64_t i = base + q * kThreads;
        key[q] = i < n_items ? __float_as_uint(depth[i]) : 0u;
    }
#pragma unroll
    for (int q = 0; q < kKeyItems; ++q) {
        const int64_t i = base + q * kThreads;
        if (i < n_items) {
            dkey[i] = key[q];
            dval[i] = (uint32_t)i;
#pragma unroll
            for (int p = 0; p < 4; ++p) hist_add(s_h, p * 256 + ((key[q] >> (8 * p)) & 0xFFu));
        }
    }
    const size_t stride = (size_t)gridDim.x * kThreads;
    const uint4 z = make_uint4(0, 0, 0, 0);
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < clear_n; i += stride) clear[i] = z;
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < clear2_n; i += stride) clear2[i] = 0ull;
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < ranges_n; i += stride) ranges[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < 4 * 256; i += kThreads)
        if (s_h[i]) atomicAdd(&hist[i], s_h[i]);
}

// A unit's runs in four words (16 bits per end; an empty run as (1, 0)).
__device__ __forceinline__ uint4 pack_runs(const Runs4& rr) {
    uint32_t w[kSuper];
#pragma unroll
    for (int k = 0; k < kSuper; ++k)
        w[k] = rr.f[k] <= rr.l[k] ? ((uint32_t)rr.f[k] | ((uint32_t)rr.l[k] << 16)) : 1u;
    return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ Runs4 unpack_runs(uint4 v) {
    const uint32_t w[kSuper] = {v.x, v.y, v.z, v.w};
    Runs4 rr;
#pragma unroll
    for (int k = 0; k < kSuper; ++k) {
        rr.f[k] = (int)(w[k] & 0xFFFFu);
        rr.l[k] = (int)(w[k] >> 16);
    }
    return rr;
}

// Coarse duplication in depth order of opacity-aware lists, with the supertile
// counts and their scan folded in.  Persistent blocks take tiles of kDupTile
// depth-ordered items from the ticket.  A unit is one supertile row of an item:
// the block deals the tile's units out to its threads (a run of consecutive
// ones each, found by a search over the items' first units), evaluates each
// one's four tile runs once into shared memory with its supertile count, scans
// the counts and publishes the sum.  It then makes one (global supertile id,
// item) pair per supertile touched, supertile rows in order, consecutive
// threads on consecutive pairs: a search over the units' first pairs names the
// unit, and with `pack` the key's high half holds the pair's 16-bit tile mask.
// Up to kStagePairs pairs are made into shared memory, then the look-back
// gives their place and they are copied out; a tile of more looks back first.
// A tile of more than kStash units goes in batches, evaluated once for the
// count and once more for the pairs.  Writes stop at `limit`; the pair total
// goes to *total and the instance count to *fine_total.  The digit histograms
// of the written pairs' supertile ids go to hist (passes of them), so a
// truncated list still sorts into a permutation of what was written; they stay
// in shared memory over all tiles of a block.  With coarse_tile > 0 the block
// also clears the look-back status words (256 per radix tile, at radix_status)
// of the pair sort's tiles that start within its pairs (below `limit`), and
// the blocks together zero st_zero[0, st_n).
//
// Bound by issue slots (61%) and by waits of every kind in a tile's chain of
// about 34000 cycles: 20% the gathers of the items, 20% evaluating, 17% making
// pairs, 17% the look-back.  Nothing may wait between a tile's ticket and its
// sum: drawing the next ticket before the look-back's end (to load its items
// early) made the look-backs wait for one another, 469 us.  3840 x 2160, 3M
// splats, 7.2M units, 14.1M pairs: one block per tile with a row's pairs
// written by its lane 674 us; this kernel 308 us, without the staged pairs 320,
// with 3 / 5 blocks per SM 333 / 370 us.
__device__ __forceinline__ uint32_t pack16(int lo, int hi) { return __byte_perm((uint32_t)lo, (uint32_t)hi, 0x5410); }
// Byte k: table[min(max(v[k] + add, 0), 4)] of the 16-bit values v[0..3] in a and b
// (entry 4 is 0).
__device__ __forceinline__ uint32_t nibbles(uint32_t table, uint32_t a, uint32_t b, uint32_t add) {
    const uint32_t x = __viaddmin_s16x2_relu(a, add, 0x00040004u) | __viaddmin_s16x2_relu(b, add, 0x00040004u) << 8;
    return __byte_perm(table, 0u, x | x >> 12);
}
constexpr uint32_t kStash = 832;
constexpr uint32_t kStagePairs = 1536;
constexpr int kDupBlocks = 4;  // per SM
constexpr uint32_t kMaxSpan = 8000;  // supertiles of a unit whose relative runs fit 16 bits
__global__ void __launch_bounds__(kThreads, kDupBlocks)
    k_dup_coarse(int n_items, const uint32_t* __restrict__ perm, const __grid_constant__ SortViews sv,
                 const float2* __restrict__ mean2d, const int* __restrict__ radius, uint64_t limit, int passes,
                 bool pack, uint32_t* tickets, unsigned long long* status, uint32_t* __restrict__ ckey,
                 uint32_t* __restrict__ cval, uint32_t* __restrict__ hist, uint64_t* __restrict__ total,
                 unsigned long long* __restrict__ fine_total, unsigned long long* __restrict__ radix_status,
                 uint32_t coarse_tile, uint32_t* __restrict__ st_zero, int st_n, GiveUp gu) {
    __shared__ uint32_t s_warp[kThreads / 32 + 1];
    __shared__ uint64_t s_prefix;
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_h[4 * 256];
    // per item of the tile
    __shared__ uint32_t s_u[kDupTile + 1];  // its first unit
    __shared__ uint2 s_rect[kDupTile];      // x0 | x1 << 16, y0 | y1 << 16 in tiles
    __shared__ float4 s_ta[kDupTile], s_tb[kDupTile];  // its TightRows
    __shared__ uint32_t s_item[kDupTile];
    __shared__ uint32_t s_row[kDupTile], s_stx[kDupTile];  // id of supertile 0 in its first row, ids per row
    __shared__ uint8_t s_mode[kDupTile];
    // per unit of the batch
    __shared__ uint4 s_runs[kStash];     // relative to the first supertile (general: pack_runs)
    __shared__ uint32_t s_p[1024];       // its first pair
    __shared__ uint32_t s_key[kStash];   // id of its first supertile (general: of its row's supertile 0)
    __shared__ uint16_t s_who[kStash];   // item | general << 15
    static_assert(kDupTile <= 256 && kStash <= 1024);
    // the tile's pairs, made before the look-back (up to kStagePairs)
    __shared__ uint32_t s_pk[kStagePairs];
    __shared__ uint8_t s_pv[kStagePairs];
    if (st_zero != nullptr)  // the supertile counters of k_pair_masks
        for (int i = blockIdx.x * kThreads + threadIdx.x; i < st_n; i += gridDim.x * kThreads) st_zero[i] = 0;
    for (int i = threadIdx.x; i < passes * 256; i += kThreads) s_h[i] = 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long fine = 0;
    auto count = [&](uint32_t key) {  // into the digit histograms (with `pack` the id is the low half)
        for (int d = 0; d < passes; ++d) atomicAdd(&s_h[d * 256 + ((key >> (8 * d)) & 0xFFu)], 1u);
    };
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(&tickets[kMaxPasses], 1u);
        __syncthreads();  // (also: the last tile's pairs have left shared memory)
        const uint32_t tile = s_tile;
        const int64_t base = (int64_t)tile * kDupTile;
        if (base >= n_items) break;
        {
            const int64_t k = base + threadIdx.x;
            const uint32_t item = k < n_items ? perm[k] : 0xffffffffu;
            uint32_t units = 0;
            if (item < (uint32_t)n_items) {  // always, unless a look-back gave up (timeout bit set)
                const int v = (int)(item / (uint32_t)sv.n_per_view);
                // all of the item's loads at once
                const float2 m = mean2d[item];
                const int r = radius[item];
                const float ca = sv.conic[3 * (size_t)item], cb = sv.conic[3 * (size_t)item + 1],
                            cc = sv.conic[3 * (size_t)item + 2];
                const float pmin = sv.power_min[item - (uint32_t)v * (uint32_t)sv.n_per_view];
                int x0, x1, y0, y1;
                if (tile_rect(m.x, m.y, r, sv.views[v].W, sv.views[v].H, x0, x1, y0, y1)) {
                    const TightRows t = tight_rows(m.x, m.y, ca, cb, cc, pmin);
                    // rows beyond the ellipse's height hold nothing: leave them out (one pixel of slack)
                    if (t.mode == 2 && fabsf(t.my) + t.ymax < 1048576.f) {
                        y0 = max(y0, (int)floorf((t.my - t.ymax - 17.f) * 0.0625f));
                        y1 = min(y1, (int)floorf((t.my + t.ymax + 1.f) * 0.0625f));
                    }
                    if (t.mode != 1 && y0 <= y1) units = (uint32_t)(y1 / kSuper - y0 / kSuper + 1);
                    s_rect[threadIdx.x] =
                        make_uint2((uint32_t)x0 | ((uint32_t)x1 << 16), (uint32_t)y0 | ((uint32_t)y1 << 16));
                    s_ta[threadIdx.x] = make_float4(t.mx, t.my, t.nB, t.det);
                    s_tb[threadIdx.x] = make_float4(t.Atau, t.rA, t.ymax, t.dyr);
                    s_item[threadIdx.x] = item;
                    s_mode[threadIdx.x] = (uint8_t)t.mode;
                    s_row[threadIdx.x] =
                        (uint32_t)sv.st_begin[v] + (uint32_t)(max(y0, 0) / kSuper) * (uint32_t)sv.st_x[v];
                    s_stx[threadIdx.x] = (uint32_t)sv.st_x[v];
                }
            }
            uint32_t all;
            s_u[threadIdx.x] = block_excl_scan<uint32_t, kThreads>(units, all, s_warp);
            if (threadIdx.x == 0) s_u[kDupTile] = all;
            __syncthreads();
        }
        const uint32_t n_units = s_u[kDupTile];
        const uint32_t batches = max(1u, (n_units + kStash - 1) / kStash);
        uint64_t tile_sum = 0, at = 0;  // `at`: where the batch's pairs go
        for (uint32_t it = 0; it < (batches == 1 ? 1u : 2 * batches); ++it) {
            const bool counting = it < batches, writing = batches == 1 || !counting;
            const uint32_t b0 = (counting ? it : it - batches) * kStash, nu = min(kStash, n_units - b0);
            const uint32_t per = (nu + kThreads - 1) / kThreads;
            const uint32_t f0 = min(threadIdx.x * per, nu), f1 = min(f0 + per, nu);
            uint32_t sum = 0;
            int i = 0;  // the last item whose first unit is at or before b0 + f0
#pragma unroll
            for (int d = kDupTile / 2; d > 0; d >>= 1)
                if (s_u[i + d] <= b0 + f0) i += d;
            for (uint32_t r = 0; r < per; ++r) {
                const uint32_t f = f0 + r;
                if (f < f1)
                    while (s_u[i + 1] <= b0 + f) ++i;  // (ends: s_u[kDupTile] is above every unit)
                __syncwarp();                          // the lanes step apart: together again for the row's work
                if (f < f1) {
                    const uint2 q = s_rect[i];
                    const float4 ta = s_ta[i], tb = s_tb[i];
                    const TightRows t{(int)s_mode[i], ta.x, ta.y, ta.z, ta.w, tb.x, tb.y, tb.z, tb.w};
                    const int y0 = (int)(q.y & 0xFFFFu), u = (int)(b0 + f - s_u[i]), sy = y0 / kSuper + u;
                    uint32_t inst = 0;
                    const Runs4 rr =
                        row_runs(t, sy, (int)(q.x & 0xFFFFu), (int)(q.x >> 16), y0, (int)(q.y >> 16), &inst);
                    // the runs of a convex shape join up; any gap between them takes the general union
                    // (selects, no branches: the lanes' patterns of empty rows differ)
                    int lo = 0x3fffffff, hi = -1;
                    bool gap = false;
#pragma unroll
                    for (int k = 0; k < kSuper; ++k) {
                        const bool some = rr.f[k] <= rr.l[k];
                        const int a = some ? rr.f[k] / kSuper : 0x3fffffff, b = some ? rr.l[k] / kSuper : -1;
                        gap |= some & (hi >= 0) & ((a > hi + 1) | (b < lo - 1));
                        lo = min(lo, a);
                        hi = max(hi, b);
                    }
                    uint32_t n = (uint32_t)max(hi - lo + 1, 0), key = s_row[i] + (uint32_t)u * s_stx[i];
                    uint4 runs;
                    const bool general = gap || n > kMaxSpan;
                    if (general) {
                        n = (uint32_t)runs_union(rr, [](int, int) {});
                        runs = pack_runs(rr);
                    } else {
                        int fr[kSuper], lr[kSuper];  // first column, 3 - last column; an empty run as 0, 4
#pragma unroll
                        for (int k = 0; k < kSuper; ++k) {
                            const bool some = rr.f[k] <= rr.l[k];
                            fr[k] = some ? rr.f[k] - lo * kSuper : 0;
                            lr[k] = some ? 3 + lo * kSuper - rr.l[k] : 4;
                        }
                        runs = make_uint4(pack16(fr[0], fr[1]), pack16(fr[2], fr[3]), pack16(lr[0], lr[1]),
                                          pack16(lr[2], lr[3]));
                        key += (uint32_t)lo;
                    }
                    s_runs[f] = runs;
                    s_key[f] = key;
                    s_who[f] = (uint16_t)((uint32_t)i | (general ? 0x8000u : 0u));
                    s_p[f] = n;
                    sum += n;
                    if (counting) fine += inst;
                }
            }
            uint32_t batch_sum;
            uint32_t p0 = block_excl_scan<uint32_t, kThreads>(sum, batch_sum, s_warp);
            for (uint32_t f = f0; f < f1; ++f) {
                const uint32_t n = s_p[f];
                s_p[f] = p0;
                p0 += n;
            }
            for (uint32_t f = nu + threadIdx.x; f < 1024; f += kThreads) s_p[f] = 0xffffffffu;
            if (counting) tile_sum += batch_sum;
            __syncthreads();
            const bool staged = batches == 1 && batch_sum <= kStagePairs;
            if (it == batches - 1 && threadIdx.x == 0) st_status(status + tile, tile == 0 ? 2u : 1u, tile_sum);
            // the pairs are made into shared memory before the look-back, while the tiles before
            // this one publish their sums; a tile of more pairs looks back first
#pragma unroll 1
            for (int ph = 0; ph < 2; ++ph) {
                if (writing && (ph == 0) == staged) {
                    const uint32_t room =
                        staged ? batch_sum : at < limit ? (uint32_t)min((uint64_t)batch_sum, limit - at) : 0u;
                    for (uint32_t p = threadIdx.x; p < room; p += kThreads) {
                        uint32_t f = 0;  // the last unit whose first pair is at or before p
#pragma unroll
                        for (uint32_t d = 512; d > 0; d >>= 1)
                            if (s_p[f + d] <= p) f += d;
                        const uint4 runs = s_runs[f];
                        const uint32_t who = s_who[f];
                        uint32_t j = p - s_p[f], key = s_key[f], mask = 0;  // mask: row k's 4 columns in byte k
                        if (who >> 15) {
                            const Runs4 rr = unpack_runs(runs);
                            int left = (int)j;
                            runs_union(rr, [&](int lo, int hi) {
                                if (left >= 0 && left <= hi - lo) j = (uint32_t)(lo + left);
                                left -= hi - lo + 1;
                            });
                            const uint32_t m = runs_mask(rr, (int)j);
                            mask = (m & 0xFu) | (m & 0xF0u) << 4 | (m & 0xF00u) << 8 | (m & 0xF000u) << 12;
                        } else if (pack) {
                            const uint32_t up = kSuper * j * 0x10001u, dn = ((0u - kSuper * j) & 0xFFFFu) * 0x10001u;
                            mask = nibbles(0x080C0E0Fu, runs.x, runs.y, dn) & nibbles(0x0103070Fu, runs.z, runs.w, up);
                        }
                        key += j;
                        if (pack) key = __byte_perm(key, mask | mask >> 4, 0x6410);  // the four nibbles above the id
                        if (staged) {
                            s_pk[p] = key;
                            s_pv[p] = (uint8_t)who;
                        } else {
                            ckey[at + p] = key;
                            cval[at + p] = s_item[who & 0xFFu];
                            count(key);
                        }
                    }
                }
                if (ph == 0 && it == batches - 1) {
                    if (warp == 0) {
                        uint64_t prefix = 0;
                        if (tile > 0) {
                            prefix = lookback_warp(status, tile, 1u, gu);
                            if (lane == 0) st_status(status + tile, 2u, prefix + tile_sum);
                        }
                        if (lane == 0) {
                            s_prefix = prefix;
                            if (base + kDupTile >= n_items) *total = prefix + tile_sum;  // the last tile: the total
                        }
                    }
                    __syncthreads();
                    at = s_prefix;
                    if (coarse_tile > 0) {  // the sort takes at most `limit` pairs: its tiles start below it
                        const uint64_t hi = min(at + tile_sum, limit);
                        for (uint64_t ct = (at + coarse_tile - 1) / coarse_tile; ct * coarse_tile < hi; ++ct)
                            radix_status[ct * 256 + threadIdx.x] = 0ull;
                    }
                }
            }
            if (staged) {
                const uint32_t room = at < limit ? (uint32_t)min((uint64_t)batch_sum, limit - at) : 0u;
                for (uint32_t p = threadIdx.x; p < room; p += kThreads) {
                    const uint32_t key = s_pk[p];
                    ckey[at + p] = key;
                    cval[at + p] = s_item[s_pv[p]];
                    count(key);
                }
            }
            if (writing) at += batch_sum;
            if (batches > 1) __syncthreads();  // the batch has left shared memory
        }
    }
    // every thread left the loop through its barrier: the histograms are complete
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fine += __shfl_xor_sync(0xffffffffu, fine, o);
    if (lane == 0 && fine) atomicAdd(fine_total, fine);
    for (int i = threadIdx.x; i < passes * 256; i += kThreads)
        if (s_h[i]) atomicAdd(&hist[i], s_h[i]);
}

// The same for full rectangles.  An item's supertiles are then a rectangle too,
// so nothing is evaluated per row: persistent blocks take tiles of 256 ITEMS
// depth-ordered items from the ticket (ITEMS consecutive ones per thread),
// scan their supertile counts, publish the sum, look back, and write the
// tile's pairs with consecutive threads on consecutive pairs; a thread finds
// its pair's item by a search over the items' first pairs and the supertile,
// key and 16-bit tile mask from the rectangle.  The digit histograms stay in
// shared memory over all tiles of a block.  It waits for its barriers and the
// chain ticket, items, gather, look-back per tile (48% of the issue slots at 6
// blocks per SM; 4 and 8 blocks, a look-back window of 128 tiles and fetching
// the next tile's items ahead were all slower).  Against the per-row kernel
// above, which full rectangles used to go through: 16 views of 1.5M splats 2.85
// -> 0.87 ms; 1920 x 1080, 1M 128 -> 34 us; 1280 x 720, 200k 43 -> 18 us.
// Counts beyond 32 bits: the starts saturate (no pair past the
// capacity, below 2^32, is written).
// Items per thread: four (half the look-back; 1M small splats, the whole sort 194 us,
// with one 216) where that leaves tiles for most SMs, one up to 2^16 items, where
// large rectangles would otherwise be the work of a few blocks: 2000 splats of
// 20000 tiles each 2.79 -> 0.83 ms, 20k of 2500 each 0.54 -> 0.27; small splats
// take the same time either way (100k: 89 and 91 us).
inline int rect_items(int64_t n) { return n <= 1 << 16 ? 1 : 4; }
template <int ITEMS>
__global__ void __launch_bounds__(kThreads, 6) k_dup_rect(int n_items, const uint32_t* __restrict__ perm,
                                                          const __grid_constant__ SortViews sv,
                                                          const float2* __restrict__ mean2d,
                                                          const int* __restrict__ radius, uint64_t limit, int passes,
                                                          bool pack, uint32_t* tickets, unsigned long long* status,
                                                          uint32_t* __restrict__ ckey, uint32_t* __restrict__ cval,
                                                          uint32_t* __restrict__ hist, uint64_t* __restrict__ total,
                                                          unsigned long long* __restrict__ fine_total,
                                                          unsigned long long* __restrict__ radix_status,
                                                          uint32_t coarse_tile, uint32_t* __restrict__ st_zero,
                                                          int st_n, GiveUp gu) {
    constexpr int TILE = kThreads * ITEMS;
    __shared__ uint64_t s_warp[kThreads / 32 + 1];
    __shared__ uint64_t s_prefix;
    __shared__ unsigned long long s_fine;
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_h[4 * 256];
    __shared__ uint32_t s_start[TILE];  // each item's first pair within the tile
    __shared__ uint2 s_rect[TILE];      // x0 | x1 << 16, y0 | y1 << 16 in tiles
    __shared__ uint32_t s_item[TILE];
    __shared__ uint8_t s_view[TILE];
    if (st_zero != nullptr)  // the supertile counters of k_pair_masks
        for (int i = blockIdx.x * kThreads + threadIdx.x; i < st_n; i += gridDim.x * kThreads) st_zero[i] = 0;
    for (int i = threadIdx.x; i < passes * 256; i += kThreads) s_h[i] = 0;
    if (threadIdx.x == 0) s_fine = 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(&tickets[kMaxPasses], 1u);
        __syncthreads();  // (also: the last tile's pairs have left shared memory)
        const uint32_t tile = s_tile;
        const int64_t base = (int64_t)tile * TILE;
        if (base >= n_items) break;
        uint32_t item[ITEMS];
        float2 m[ITEMS];
        int r[ITEMS];
        const int64_t k0 = base + (int64_t)threadIdx.x * ITEMS;
        if (ITEMS == 4 && k0 + ITEMS <= n_items) {
            const uint4 q = *reinterpret_cast<const uint4*>(perm + k0);  // k0 is a multiple of 4, perm 256-byte aligned
            const uint32_t qi[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) item[i] = qi[i];
        } else {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) item[i] = k0 + i < n_items ? perm[k0 + i] : 0xffffffffu;
        }
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const bool ok = item[i] < (uint32_t)n_items;  // always, unless a look-back gave up (timeout bit set)
            r[i] = ok ? radius[item[i]] : 0;
            m[i] = ok ? mean2d[item[i]] : make_float2(0.f, 0.f);
        }
        uint32_t c[ITEMS];
        uint64_t sum = 0;
        unsigned long long fine = 0;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int v = item[i] < (uint32_t)n_items ? (int)(item[i] / (uint32_t)sv.n_per_view) : 0;
            int x0, x1, y0, y1;
            c[i] = 0;
            if (tile_rect(m[i].x, m[i].y, r[i], sv.views[v].W, sv.views[v].H, x0, x1, y0, y1)) {
                c[i] = (uint32_t)(x1 / kSuper - x0 / kSuper + 1) * (uint32_t)(y1 / kSuper - y0 / kSuper + 1);
                fine += (unsigned long long)(x1 - x0 + 1) * (unsigned long long)(y1 - y0 + 1);
                const int at = threadIdx.x * ITEMS + i;
                s_rect[at] = make_uint2((uint32_t)x0 | ((uint32_t)x1 << 16), (uint32_t)y0 | ((uint32_t)y1 << 16));
                s_item[at] = item[i];
                s_view[at] = (uint8_t)v;
            }
            sum += c[i];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) fine += __shfl_xor_sync(0xffffffffu, fine, o);
        if (lane == 0 && fine) atomicAdd(&s_fine, fine);
        uint64_t tile_sum;
        uint64_t at = block_excl_scan<uint64_t, kThreads>(sum, tile_sum, s_warp);
        if (threadIdx.x == 0) st_status(status + tile, tile == 0 ? 2u : 1u, tile_sum);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            s_start[threadIdx.x * ITEMS + i] = (uint32_t)min(at, (uint64_t)0xffffffffu);
            at += c[i];
        }
        if (warp == 0) {
            uint64_t prefix = 0;
            if (tile > 0) {
                prefix = lookback_warp(status, tile, 1u, gu);
                if (lane == 0) st_status(status + tile, 2u, prefix + tile_sum);
            }
            if (lane == 0) {
                s_prefix = prefix;
                if (base + TILE >= n_items) *total = prefix + tile_sum;  // the last tile: the total
            }
        }
        __syncthreads();
        const uint64_t g0 = s_prefix;
        if (coarse_tile > 0) {  // the sort takes at most `limit` pairs: its tiles start below it
            const uint64_t hi = min(g0 + tile_sum, limit);
            for (uint64_t ct = (g0 + coarse_tile - 1) / coarse_tile; ct * coarse_tile < hi; ++ct)
                radix_status[ct * 256 + threadIdx.x] = 0ull;
        }
        const uint64_t room = g0 < limit ? min(tile_sum, limit - g0) : 0;  // below 2^32
        for (uint64_t p64 = threadIdx.x; p64 < room; p64 += kThreads) {
            const uint32_t p = (uint32_t)p64;
            // the last item whose first pair is at or before p
            int i = 0;
#pragma unroll
            for (int d = TILE / 2; d > 0; d >>= 1)
                if (s_start[i + d] <= p) i += d;
            const uint2 q = s_rect[i];
            const int v = s_view[i];
            const uint32_t x0 = q.x & 0xFFFFu, x1 = q.x >> 16, y0 = q.y & 0xFFFFu, y1 = q.y >> 16;
            const uint32_t w = x1 / kSuper - x0 / kSuper + 1, j = p - s_start[i];
            // below 2^21 the rounded product cannot cross an integer ((j + 1/2) / w is at least
            // 1 / (2 w) away from one)
            const uint32_t row = j < (1u << 21) ? (uint32_t)(((float)j + 0.5f) * __frcp_rn((float)w)) : j / w;
            const uint32_t sx = x0 / kSuper + (j - row * w), sy = y0 / kSuper + row;
            uint32_t key = (uint32_t)sv.st_begin[v] + sy * (uint32_t)sv.st_x[v] + sx;
            for (int d = 0; d < passes; ++d) {
                const uint32_t bin = (key >> (8 * d)) & 0xFFu;
                atomicAdd(&s_h[d * 256 + bin], 1u);
            }
            if (pack) {  // bit 4 k + c: tile (4 sx + c, 4 sy + k) within the rectangle
                const uint32_t cx = sx * kSuper, cy = sy * kSuper;
                const uint32_t a = max(x0, cx) - cx, b = min(x1, cx + kSuper - 1) - cx;
                const uint32_t e = max(y0, cy) - cy, f = min(y1, cy + kSuper - 1) - cy;
                const uint32_t cols = ((2u << b) - (1u << a)) * 0x1111u;
                key |= (cols & ((16u << (4 * f)) - (1u << (4 * e)))) << 16;
            }
            ckey[g0 + p] = key;
            cval[g0 + p] = s_item[i];
        }
    }
    // every thread left the loop through its barrier: the histograms are complete
    if (threadIdx.x == 0 && s_fine) atomicAdd(fine_total, s_fine);
    for (int i = threadIdx.x; i < passes * 256; i += kThreads)
        if (s_h[i]) atomicAdd(&hist[i], s_h[i]);
}

// First position of key >= want in keys[0, n), ascending in (key & kmask).
__device__ __forceinline__ uint32_t lower_bound_u32(const uint32_t* __restrict__ keys, uint32_t n, uint32_t want,
                                                    uint32_t kmask) {
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = lo + ((hi - lo) >> 1);
        if ((keys[mid] & kmask) < want) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The 16-bit mask of an item's instances in the supertile whose first tile
// is (cx0, cy0): bit 4 r + c for tile (cx0 + c, cy0 + r).  The same rule as
// the counts (tile_rect, then tight_row per row with the item's whole
// rectangle), clipped to the supertile.
template <bool TIGHT>
__device__ __forceinline__ uint32_t supertile_mask(const SortViews& sv, const float2* mean2d, const int* radius,
                                                   uint32_t item, const ViewDesc& vd, int cx0, int cy0) {
    const float2 m = mean2d[item];
    int x0, x1, y0, y1;
    if (!tile_rect(m.x, m.y, radius[item], vd.W, vd.H, x0, x1, y0, y1)) return 0u;
    const int a0 = max(x0, cx0), a1 = min(x1, cx0 + kSuper - 1);
    if (a0 > a1) return 0u;
    TightRows t{};
    if constexpr (TIGHT) t = item_tight_rows(sv, mean2d, item);
    uint32_t mask = 0;
#pragma unroll
    for (int r = 0; r < kSuper; ++r) {
        const int y = cy0 + r;
        if (y < y0 || y > y1) continue;
        int f = x0, l = x1;
        if constexpr (TIGHT) tight_row(t, y, x0, x1, f, l);
        f = max(f, a0);
        l = min(l, a1);
        if (f <= l) mask |= ((1u << (l - f + 1)) - 1u) << (r * kSuper + f - cx0);
    }
    return mask;
}

// The instance counts of the supertile's tiles, added into ranges[2 t + 1]
// (cleared by k_keys), from the sorted pairs' 16-bit tile masks: the
// duplication packed them above the supertile id (`pack`), else they are
// computed here and stored to masks[].  Each warp takes segments of
// kPairSeg consecutive pairs; the pairs are sorted by supertile, so a warp's
// 32 pairs mostly share one, and while they do the warp counts each tile's
// bits with four lane reductions (bit j of every mask spread to its own byte)
// into lane j's count, adding it to ranges with one atomic per tile when the
// supertile changes.  32 pairs of several supertiles: one atomic per group
// of equal supertiles and tile.  With st_count (zeroed by the duplication), each
// supertile's total is added there as well, and the ends of its pairs go to
// st_beg / st_end (supertiles without pairs are left alone).  Segments are 128 to 512 pairs
// (the least that gives every warp at most one), loaded 128 pairs at a time
// with the next 128 in flight: the kernel waits for memory, not for its
// arithmetic.
constexpr uint32_t kPairBatch = 128, kPairSegMax = 512;
template <bool TIGHT>
__global__ void __launch_bounds__(kThreads) k_pair_masks(const __grid_constant__ SortViews sv,
                                                         const float2* __restrict__ mean2d,
                                                         const int* __restrict__ radius,
                                                         const uint32_t* __restrict__ ckey,
                                                         const uint32_t* __restrict__ cval, uint32_t n_host,
                                                         const uint64_t* __restrict__ n_dev, uint32_t n_items,
                                                         bool pack, uint16_t* __restrict__ masks,
                                                         uint32_t* __restrict__ ranges, uint32_t* st_count,
                                                         uint32_t* __restrict__ st_beg, uint32_t* __restrict__ st_end,
                                                         const unsigned* __restrict__ gave_up) {
    if (*gave_up != 0) return;  // the pairs are not what the sort was to leave: every list stays empty
    const uint32_t Ic = pass_count(n_host, n_dev);
    const int lane = threadIdx.x & 31;
    // tile j of supertile key (global id) as a global tile index
    auto tile_of = [&](uint32_t key, int j) -> size_t {
        int v = 0;
        while (v + 1 < sv.num_views && sv.st_begin[v + 1] <= (int)key) ++v;
        const int ls = (int)key - sv.st_begin[v];
        const ViewDesc& vd = sv.views[v];
        return (size_t)vd.tile_begin + (size_t)((ls / sv.st_x[v]) * kSuper + (j >> 2)) * vd.tiles_x +
               (size_t)((ls % sv.st_x[v]) * kSuper + (j & 3));
    };
    const uint64_t warp_id = ((uint64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
    const uint64_t warps = ((uint64_t)gridDim.x * kThreads) >> 5;
    const uint64_t want = (Ic + warps - 1) / warps;
    const uint64_t seg =
        min((uint64_t)kPairSegMax, max((want + kPairBatch - 1) / kPairBatch, (uint64_t)1) * kPairBatch);
    constexpr int U = kPairBatch / 32;
    for (uint64_t s0 = warp_id * seg; s0 < Ic; s0 += warps * seg) {
        const uint64_t s1 = min(s0 + seg, (uint64_t)Ic);
        uint32_t cur = 0xffffffffu;  // the supertile being counted (warp-uniform)
        uint32_t acc = 0;            // lane j < 16: its count of tile j
        auto flush = [&]() {
            if (cur != 0xffffffffu && lane < 16 && acc) atomicAdd(&ranges[2 * tile_of(cur, lane) + 1], acc);
            if (st_count != nullptr) {  // the supertile's total
                const uint32_t all = __reduce_add_sync(0xffffffffu, lane < 16 ? acc : 0u);
                if (cur != 0xffffffffu && lane == 0 && all) atomicAdd(&st_count[cur], all);
            }
            acc = 0;
        };
        const uint32_t kmask = pack ? 0xFFFFu : 0xFFFFFFFFu;
        // the supertile of the pair before the group's
        uint32_t last = st_beg != nullptr && s0 > 0 ? ckey[s0 - 1] & kmask : 0xffffffffu;
        uint32_t kn[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t e = s0 + (uint64_t)(32 * u + lane);
            kn[u] = e < s1 ? ckey[e] : 0xffffffffu;
        }
        for (uint64_t b0 = s0; b0 < s1; b0 += kPairBatch) {
            uint32_t kb[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                kb[u] = kn[u];
                const uint64_t e = b0 + kPairBatch + (uint64_t)(32 * u + lane);
                kn[u] = e < s1 ? ckey[e] : 0xffffffffu;
            }
#pragma unroll 1
            for (int u = 0; u < U; ++u) {
                const uint64_t b = b0 + (uint64_t)(32 * u);
                if (b >= s1) break;
                const uint64_t e = b + (uint64_t)lane;
                uint32_t key = 0xffffffffu, m = 0;
                if (e < s1) {
                    key = u == 0 ? kb[0] : u == 1 ? kb[1] : u == 2 ? kb[2] : kb[3];
                    if (pack) {
                        m = key >> 16;
                        key &= 0xFFFFu;
                    } else {
                        int v = 0;
                        while (v + 1 < sv.num_views && sv.st_begin[v + 1] <= (int)key) ++v;
                        const int ls = (int)key - sv.st_begin[v];
                        const uint32_t it = cval[e];
                        m = it < n_items ? supertile_mask<TIGHT>(sv, mean2d, radius, it, sv.views[v],
                                                                 (ls % sv.st_x[v]) * kSuper, (ls / sv.st_x[v]) * kSuper)
                                         : 0u;
                        masks[e] = (uint16_t)m;
                    }
                }
                const uint32_t k0 = __shfl_sync(0xffffffffu, key, 0);  // lane 0 always holds a pair
                const bool same = __all_sync(0xffffffffu, key == k0 || e >= s1);
                if (st_beg != nullptr && (!same || k0 != last || b + 32 >= Ic)) {
                    uint32_t prev = __shfl_up_sync(0xffffffffu, key, 1);
                    if (lane == 0) prev = last;
                    if (e < s1) {
                        if (key != prev) {
                            st_beg[key] = (uint32_t)e;
                            if (prev != 0xffffffffu) st_end[prev] = (uint32_t)e;
                        }
                        if (e + 1 == Ic) st_end[key] = Ic;
                    }
                }
                last = k0;  // (used only if the segment goes on: the group is full then)
                if (!same) {
                    last = __shfl_sync(0xffffffffu, key, 31);
                    // pairs of several supertiles: one atomic per group and tile
                    flush();
                    cur = 0xffffffffu;
                    const unsigned peers = __match_any_sync(0xffffffffu, key);
                    const bool leader = lane == __ffs(peers) - 1 && key != 0xffffffffu;
                    uint32_t all = 0;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const unsigned bj = __ballot_sync(0xffffffffu, (m >> j) & 1u) & peers;
                        if (leader && bj) atomicAdd(&ranges[2 * tile_of(key, j) + 1], (uint32_t)__popc(bj));
                        all += (uint32_t)__popc(bj);
                    }
                    if (st_count != nullptr && leader && all) atomicAdd(&st_count[key], all);
                    continue;
                }
                if (k0 != cur) {
                    flush();
                    cur = k0;
                }
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    // bits 4w .. 4w + 3 of the mask to bytes 0..3, summed over the warp (<= 32 each)
                    const uint32_t spread = (((m >> (4 * w)) & 0xFu) * 0x00204081u) & 0x01010101u;
                    const uint32_t sum = __reduce_add_sync(0xffffffffu, spread);
                    if ((lane >> 2) == w) acc += (sum >> (8 * (lane & 3))) & 0xFFu;
                }
            }
        }
        flush();
    }
}

// One block per supertile s (st_order[blockIdx], the largest first, when
// given), after k_tile_scan: its items are the sorted pairs [cs, ce) with
// key s; every instance's id (and key) goes to its tile's next position, in
// item order, from the pairs' tile masks (in the key's high half when kmask
// is 0xFFFF, else in masks[]).  Rounds of one pair per thread, the next
// round's loads in flight during the current one.  A warp's 32 pairs give one
// ballot per tile; the ballots' counts of all warps (a small table) place the
// warp in each tile's list, and a lane with the tile's bit writes its id at
// the place its lower lanes leave, so that the ids of a warp go to consecutive
// addresses.  Splitting a round by pairs rather than by tiles keeps the chain
// per round short, which is what the kernel waits for: its time is that of the
// longest supertiles, whose rounds follow one another.  The depth a key needs
// is read once per pair, a round ahead.  Against warps that own tiles and walk
// all pairs of a round: 1280 x 720, 200k, full rectangles with keys 114 -> 44
// us; 1920 x 1080, 1M 252 -> 93; opacity-aware lists at 3840 x 2160, 139M
// instances, no keys 225 -> 206 (2.7 TB/s of ids); 16 views 563 -> 524 us.
// With more supertiles than items (no counts or ends then) most blocks find a pair or
// none, so a block is half as large: 20k items on 20000 x 20000 pixels 1.70 -> 1.38 ms
// for the whole sort (four warps 1.23), but 15k items on one supertile of 8000 x 8000
// 276 -> 298 us (four warps 348).
constexpr int kFineWarps = 16;
constexpr int kFineSparseWarps = 8;
template <bool KEYS, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_fine(const __grid_constant__ SortViews sv,
                                                       const float* __restrict__ depth,
                                                       const uint32_t* __restrict__ ckey,
                                                       const uint32_t* __restrict__ cval, uint32_t n_host,
                                                       const uint64_t* __restrict__ n_dev, uint32_t kmask,
                                                       const uint16_t* __restrict__ masks,
                                                       const uint32_t* __restrict__ ranges,
                                                       const uint32_t* __restrict__ st_order,
                                                       const uint32_t* __restrict__ st_count,
                                                       const uint32_t* __restrict__ st_beg,
                                                       const uint32_t* __restrict__ st_end, uint32_t n_items,
                                                       uint32_t* __restrict__ ids_out, uint64_t* __restrict__ keys_out) {
    constexpr int THREADS = 32 * WARPS;
    __shared__ uint32_t s_rng[2];
    __shared__ uint32_t s_beg[16], s_len[16];
    // instances per round (double-buffered), tile and warp, one byte each (<= 32)
    static_assert(WARPS == 8 || WARPS == 16, "the warps' bytes make two words of a tile or four");
    using Counts = std::conditional_t<WARPS == 16, uint4, uint2>;
    __shared__ Counts s_cnt[2][16];
    const int s = st_order != nullptr ? (int)st_order[blockIdx.x] : (int)blockIdx.x;  // largest first
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    int v = 0;
    while (v + 1 < sv.num_views && sv.st_begin[v + 1] <= s) ++v;
    const ViewDesc& vd = sv.views[v];
    const int ls = s - sv.st_begin[v];
    const int cx0 = (ls % sv.st_x[v]) * kSuper, cy0 = (ls / sv.st_x[v]) * kSuper;
    const int tx = vd.tiles_x, ty = tiles_y(vd.H);
    const uint32_t Ic = pass_count(n_host, n_dev);
    if (st_count != nullptr) {  // k_pair_masks left the ends of the supertile's pairs
        if (st_count[s] == 0) return;
        if (threadIdx.x < 2) s_rng[threadIdx.x] = min(threadIdx.x ? st_end[s] : st_beg[s], Ic);
    } else if (threadIdx.x < 2) {
        s_rng[threadIdx.x] = lower_bound_u32(ckey, Ic, (uint32_t)s + threadIdx.x, kmask);
    }
    if (threadIdx.x < 16) {
        const int c = cx0 + (threadIdx.x & 3), r = cy0 + (threadIdx.x >> 2);
        const bool ok = c < tx && r < ty;
        const uint32_t gt = (uint32_t)vd.tile_begin + (uint32_t)r * (uint32_t)tx + (uint32_t)c;
        const uint32_t b = ok ? ranges[2 * gt] : 0u, e = ok ? ranges[2 * gt + 1] : 0u;
        s_beg[threadIdx.x] = b;
        s_len[threadIdx.x] = e - b;
    }
    __syncthreads();
    const uint32_t cs = s_rng[0], ce = s_rng[1];
    if (cs >= ce) return;
    const bool packed = kmask == 0xFFFFu;
    const int tl = lane & 15;
    const uint32_t beg = s_beg[tl], len = s_len[tl];  // lane t (and t + 16): tile t's list
    const uint32_t tile_key = (uint32_t)vd.tile_begin + (uint32_t)(cy0 + (tl >> 2)) * (uint32_t)tx + (uint32_t)(cx0 + (tl & 3));
    uint32_t run = 0;  // lane t: tile t's instances of the rounds before
    // pairs of the next round, and of the one after it: a key's depth is a load that
    // depends on the pair's item
    uint32_t mk = 0, it = 0, dp = 0, mk2 = 0, it2 = 0;
    auto fetch = [&](uint32_t e) {
        mk2 = e < ce ? (packed ? ckey[e] >> 16 : (uint32_t)masks[e]) : 0u;
        it2 = e < ce ? cval[e] : 0u;
    };
    auto advance = [&](uint32_t e) {
        mk = mk2;
        it = it2;
        if constexpr (KEYS) dp = mk != 0 && it < n_items ? __float_as_uint(depth[it]) : 0u;
        fetch(e);
    };
    fetch(cs + threadIdx.x);
    advance(cs + THREADS + threadIdx.x);
    for (uint32_t r0 = cs, round = 0; r0 < ce; r0 += THREADS, round ^= 1u) {
        const uint32_t m = mk, id = it, dep = dp;
        advance(r0 + 2 * THREADS + threadIdx.x);
        // lane t: the warp's instances of tile t in this round, from four lane reductions of
        // the masks' bits spread to bytes
        uint32_t cnt = 0;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const uint32_t spread = (((m >> (4 * w)) & 0xFu) * 0x00204081u) & 0x01010101u;
            const uint32_t sum = __reduce_add_sync(0xffffffffu, spread);
            if ((tl >> 2) == w) cnt = (sum >> (8 * (tl & 3))) & 0xFFu;
        }
        if (lane < 16) reinterpret_cast<uint8_t*>(&s_cnt[round][lane])[warp] = (uint8_t)cnt;
        __syncthreads();  // (a warp two rounds ahead has passed the next barrier: two tables suffice)
        // where the warp's instances of tile t start: after those of the lower warps
        const uint32_t lo = 0xFFFFFFFFu >> (31 - 8 * (warp & 3)) >> 1;  // the bytes of the lower warps in this warp's word
        uint32_t off = run;
        if constexpr (WARPS == 16) {
            const uint4 c4 = s_cnt[round][tl];
            const int wq = warp >> 2;
            off = __dp4a(wq > 0 ? c4.x : c4.x & lo, 0x01010101u, off);
            off = __dp4a(wq > 1 ? c4.y : wq == 1 ? c4.y & lo : 0u, 0x01010101u, off);
            off = __dp4a(wq > 2 ? c4.z : wq == 2 ? c4.z & lo : 0u, 0x01010101u, off);
            off = __dp4a(wq == 3 ? c4.w & lo : 0u, 0x01010101u, off);
            run = __dp4a(c4.x, 0x01010101u, __dp4a(c4.y, 0x01010101u, __dp4a(c4.z, 0x01010101u, __dp4a(c4.w, 0x01010101u, run))));
        } else {
            const uint2 c2 = s_cnt[round][tl];
            off = __dp4a(warp < 4 ? c2.x & lo : c2.x, 0x01010101u, off);
            off = __dp4a(warp < 4 ? 0u : c2.y & lo, 0x01010101u, off);
            run = __dp4a(c2.x, 0x01010101u, __dp4a(c2.y, 0x01010101u, run));
        }
        // whole unless the lists are cut off at the capacity
        const bool whole = __all_sync(0xffffffffu, off + cnt <= len);
        const uint32_t place = beg + off;
        const unsigned any = __reduce_or_sync(0xffffffffu, m);
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            if (!((any >> t) & 1u)) continue;
            bool in = (m >> t) & 1u;
            const uint32_t o = (uint32_t)__popc(__ballot_sync(0xffffffffu, in) & lt);
            const uint32_t p = __shfl_sync(0xffffffffu, place, t) + o;
            if (!whole) {  // (uniform; every lane takes part in the shuffles)
                const uint32_t ot = __shfl_sync(0xffffffffu, off, t) + o, lt_n = __shfl_sync(0xffffffffu, len, t);
                in = in && ot < lt_n;
            }
            uint32_t hi = 0;
            if constexpr (KEYS) hi = __shfl_sync(0xffffffffu, tile_key, t);
            if (in) {
                ids_out[p] = id;
                if constexpr (KEYS) keys_out[p] = ((uint64_t)hi << 32) | dep;
            }
        }
    }
}

// Tile ranges from the per-tile counts in ranges[2 t + 1]: an exclusive scan
// over all tiles (one block), each bound clamped to the capacity.  With
// st_order: the supertiles in decreasing order of their instance counts
// (st_count, from k_pair_masks), by octave buckets
// (st_order, total_st entries), so that the fine writes start the longest
// supertiles first (the order within a bucket is arbitrary; the output does
// not depend on it).  Graph mode: the instance count (fine_total, from
// the duplication) to *count_out, and the capacity bit when it exceeds the
// capacity.
constexpr int kScanThreads = 1024;
constexpr int kStBuckets = 33;  // 0: empty, b: counts in [2^(b-1), 2^b)
__device__ __forceinline__ int octave(uint32_t x) { return x == 0 ? 0 : 32 - __clz(x); }
__global__ void __launch_bounds__(kScanThreads) k_tile_scan(const __grid_constant__ SortViews sv, int num_tiles,
                                                            uint32_t* __restrict__ ranges, uint64_t cap,
                                                            const unsigned long long* fine_total,
                                                            int64_t* count_out, const uint32_t* st_count,
                                                            uint32_t* __restrict__ st_order, unsigned* err) {
    constexpr int PER = 4;                       // consecutive tiles per thread and round
    constexpr int R = kScanThreads * PER;        // tiles per round
    __shared__ uint64_t s_warp[kScanThreads / 32 + 1];
    __shared__ uint32_t s_bk[kStBuckets];
    __shared__ uint32_t s_a[R + R / 32], s_b[R + R / 32];  // counts, then begins and ends (padded)
    auto at = [](int i) { return i + (i >> 5); };
    const int nst = sv.total_st;
    if (threadIdx.x < kStBuckets) s_bk[threadIdx.x] = 0;
    uint64_t run = 0;
    for (int64_t b = 0; b < num_tiles; b += R) {
        // the round's counts, consecutive threads on consecutive tiles
        for (int i = threadIdx.x; i < R; i += kScanThreads)
            s_a[at(i)] = b + i < num_tiles ? ranges[2 * (b + i) + 1] : 0u;
        __syncthreads();
        uint32_t c[PER];
        uint64_t sum = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            c[k] = s_a[at(threadIdx.x * PER + k)];
            sum += c[k];
        }
        uint64_t tot;
        uint64_t pre = run + block_excl_scan<uint64_t, kScanThreads>(sum, tot, s_warp);
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int i = threadIdx.x * PER + k;
            s_a[at(i)] = (uint32_t)(c[k] > 0 ? min(pre, cap) : 0);
            s_b[at(i)] = (uint32_t)(c[k] > 0 ? min(pre + c[k], cap) : 0);
            pre += c[k];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < R; i += kScanThreads)
            if (b + i < num_tiles) {
                ranges[2 * (b + i)] = s_a[at(i)];
                ranges[2 * (b + i) + 1] = s_b[at(i)];
            }
        __syncthreads();  // s_a is reloaded next round
        run += tot;
    }
    if (st_order != nullptr) {
        __syncthreads();
        for (int i = threadIdx.x; i < nst; i += kScanThreads) atomicAdd(&s_bk[octave(__ldcg(st_count + i))], 1u);
        __syncthreads();
        if (threadIdx.x == 0) {  // bucket starts, the largest octave first
            uint32_t acc = 0;
            for (int k = kStBuckets - 1; k >= 0; --k) {
                const uint32_t n = s_bk[k];
                s_bk[k] = acc;
                acc += n;
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nst; i += kScanThreads)
            st_order[atomicAdd(&s_bk[octave(__ldcg(st_count + i))], 1u)] = (uint32_t)i;
    }
    if (threadIdx.x == 0 && count_out != nullptr) {
        const uint64_t all = *fine_total;
        *count_out = (int64_t)all;
        if (all > cap) atomicOr(err, kErrCapacity);
    }
}

// Workspace: per-item arrays, a header cleared by one memset (digit
// histograms, tickets, counts), the look-back status words (cleared by
// k_keys), and the pair key/value double buffers.
struct Layout {
    size_t dk0, dk1, dv0, dv1, hdr, hist, tickets, total, ctotal, gave_up, hdr_bytes, status, status_bytes, tk0, tk1, tv0,
        tv1, total_bytes;
};

Layout make_layout(int n, int64_t capacity) {
    Layout L{};
    size_t o = 0;
    auto take = [&](size_t bytes) {
        size_t at = o;
        o = align256(o + bytes);
        return at;
    };
    const size_t N = (size_t)(n > 0 ? n : 1), C = (size_t)(capacity > 0 ? capacity : 1);
    L.dk0 = take(4 * N);
    L.dk1 = take(4 * N);
    L.dv0 = take(4 * N);
    L.dv1 = take(4 * N);
    L.hdr = o;
    L.hist = take(4 * 256 * kMaxPasses);
    L.tickets = take(4 * (kMaxPasses + 1));
    L.total = take(24);  // instances, then supertile pairs (the duplication), then the give-up flag
    L.ctotal = L.total + 8;
    L.gave_up = L.total + 16;
    L.hdr_bytes = o - L.hdr;
    // status words: 256 per radix tile (the largest tile count of either sort)
    // plus one per duplication tile
    const size_t radix_tiles = (size_t)std::max(radix_tiles_max((int64_t)N), radix_tiles_max((int64_t)C));
    L.status = take(8 * (256 * radix_tiles + (size_t)cdiv((int64_t)N, kDupTile)));
    L.status_bytes = o - L.status;  // a multiple of 256
    L.tk0 = take(4 * C);
    L.tk1 = take(4 * C);
    L.tv0 = take(4 * C);
    L.tv1 = take(4 * C);
    L.total_bytes = o;
    return L;
}

}  // namespace

namespace {
// power_min[g] = ln(1 / (255 o_g)) - kTightMargin: the exponent a splat must reach
// for alpha = o exp(power) >= 1/255, lowered by a margin that covers the
// exponent error of the blend variants (the split tensor-core ones are <= 1e-3);
// +inf for o below the blend's FP32 threshold 1/255 (alpha <= o never reaches
// it; o equal to it still passes where the exponent is 0).
constexpr float kTightMargin = 2e-3f;
__global__ void k_alpha_power_min(int n, const float* __restrict__ opacity, float* __restrict__ out) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    const float o = opacity[g];
    out[g] = o >= 1.0f / 255.0f ? -logf(255.0f * o) - kTightMargin : INFINITY;
}
}  // namespace

cudaError_t launch_alpha_power_min(int n, const float* opacity, float* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_alpha_power_min<<<(n + 255) / 256, 256, 0, s>>>(n, opacity, out);
    count_launches();
    return cudaGetLastError();
}

size_t bin_sort_workspace_bytes(int n_items, int64_t capacity, int /*num_tiles*/) {
    return make_layout(n_items, capacity).total_bytes;
}

gs_status bin_sort_run(const SortViews& sv, const float* mean2d_f, const int* radius, const float* depth,
                       int64_t capacity, void* ws, size_t /*ws_bytes*/, uint64_t* keys_sorted, uint32_t* ids_sorted,
                       uint32_t* tile_ranges, int64_t* n_instances_host, int64_t* n_instances_dev, cudaStream_t s) {
    const int ntiles = sv.total_tiles;
    const int n = sv.num_views * sv.n_per_view;  // items
    const bool graph = n_instances_host == nullptr;
    cudaError_t e;
    if (!graph) *n_instances_host = 0;
    if (n == 0) {
        if ((e = cudaMemsetAsync(tile_ranges, 0, sizeof(uint32_t) * 2 * (size_t)ntiles, s)) != cudaSuccess)
            return cuda_status(e, "gs_bin_sort: clear ranges");
        if (graph && (e = cudaMemsetAsync(n_instances_dev, 0, sizeof(int64_t), s)) != cudaSuccess)
            return cuda_status(e, "gs_bin_sort: count");
        return GS_OK;
    }
    unsigned* err = error_word();
    if (err == nullptr) return cuda_status(cudaGetLastError(), "gs_bin_sort: error word");
    const Layout L = make_layout(n, capacity);
    char* base = static_cast<char*>(ws);
    auto U32 = [&](size_t off) { return reinterpret_cast<uint32_t*>(base + off); };
    const float2* mean2d = reinterpret_cast<const float2*>(mean2d_f);
    uint32_t* hist = U32(L.hist);
    uint32_t* tickets = U32(L.tickets);
    uint64_t* total = reinterpret_cast<uint64_t*>(base + L.total);
    unsigned long long* status = reinterpret_cast<unsigned long long*>(base + L.status);
    const int64_t radix_status_words = (int64_t)(L.status_bytes / 8) - cdiv(n, kDupTile);
    unsigned long long* dup_status = status + radix_status_words;
    unsigned* gave_up = reinterpret_cast<unsigned*>(base + L.gave_up);
    const GiveUp gu{err, gave_up};
    const PassScratch ps{hist, tickets, status, gu};

    // supertiles of every view
    SortViews sv2 = sv;
    {
        int st = 0;
        for (int v = 0; v < sv.num_views; ++v) {
            sv2.st_begin[v] = st;
            sv2.st_x[v] = (int)cdiv(sv.views[v].tiles_x, kSuper);
            st += sv2.st_x[v] * (int)cdiv(tiles_y(sv.views[v].H), kSuper);
        }
        sv2.total_st = st;
    }
    uint64_t* ctotal = reinterpret_cast<uint64_t*>(base + L.ctotal);

    // 1. depth keys and their digit histograms; clears
    if ((e = cudaMemsetAsync(base + L.hdr, 0, L.hdr_bytes, s)) != cudaSuccess)
        return cuda_status(e, "gs_bin_sort: clear header");
    const bool tight = sv.conic != nullptr;
    unsigned long long* fine_total = reinterpret_cast<unsigned long long*>(total);
    // status words: the depth sort's here; the pair sort's by the duplication (graph mode) or a
    // memset sized by the pair count (synchronising mode)
    const size_t depth_status_words = 256 * (size_t)radix_tiles_max(n);
    k_keys<<<(int)cdiv(n, kThreads * kKeyItems), kThreads, 0, s>>>(
        n, depth, U32(L.dk0), U32(L.dv0), hist, reinterpret_cast<uint4*>(status), depth_status_words / 2, dup_status,
        (size_t)cdiv(n, kDupTile), tile_ranges, 2 * (size_t)ntiles);
    count_launches();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_status(e, "gs_bin_sort: keys");

    // 2. depth sort of all items (pass ids 0..3)
    uint32_t* dk[2] = {U32(L.dk0), U32(L.dk1)};
    uint32_t* dv[2] = {U32(L.dv0), U32(L.dv1)};
    int which = 0;
    if ((e = radix_sort(dk, dv, (uint32_t)n, nullptr, 32, 0, ps, &which, s)) != cudaSuccess)
        return cuda_status(e, "gs_bin_sort: depth sort");
    const uint32_t* perm = dv[which];

    // 3. supertile pairs in depth order, the instance count (pass ids 4.. for the supertile-id histograms)
    int st_bits = 1;
    while ((1ll << st_bits) < sv2.total_st) ++st_bits;
    const int st_passes = (st_bits + 7) / 8;
    uint32_t* ck[2] = {U32(L.tk0), U32(L.tk1)};
    uint32_t* cv[2] = {U32(L.tv0), U32(L.tv1)};
    // up to 2^16 supertiles the pairs' tile masks ride in the key's high half
    const bool pack = st_bits <= 16;
    const uint32_t coarse_tile = graph ? (uint32_t)(kThreads * pass_items((uint64_t)capacity)) : 0u;
    // per-supertile instance counts and their order, largest first, in the depth keys'
    // buffers (free once the depth sort is done), when they fit
    const int nst = sv2.total_st;
    uint32_t* st_count = nst <= n ? dk[0] : nullptr;
    uint32_t* st_order = nst <= n ? dk[1] : nullptr;
    // the ends of each supertile's pairs, in the sorted items' buffers (free after the duplication)
    uint32_t* st_beg = nst <= n ? dv[0] : nullptr;
    uint32_t* st_end = nst <= n ? dv[1] : nullptr;
    if ((e = record_kernel_event(GS_KERNEL_DUPLICATE, false, s)) != cudaSuccess)
        return cuda_status(e, "gs_bin_sort: kernel event");
    int dev_sms = 0;
    {
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
            return cuda_status(e, "gs_bin_sort: device");
    }
    if (tight)
        k_dup_coarse<<<(int)std::min<int64_t>(cdiv(n, kDupTile), kDupBlocks * (int64_t)dev_sms), kThreads, 0, s>>>(
            n, perm, sv2, mean2d, radius, (uint64_t)capacity, st_passes, pack, tickets, dup_status, ck[0], cv[0],
            hist + 256 * 4, ctotal, fine_total, status, coarse_tile, st_count, nst, gu);
    else {
        auto dup_rect = rect_items(n) == 1 ? k_dup_rect<1> : k_dup_rect<4>;
        dup_rect<<<(int)std::min<int64_t>(cdiv(n, kThreads * rect_items(n)), 6 * (int64_t)dev_sms), kThreads, 0, s>>>(
            n, perm, sv2, mean2d, radius, (uint64_t)capacity, st_passes, pack, tickets, dup_status, ck[0], cv[0],
            hist + 256 * 4, ctotal, fine_total, status, coarse_tile, st_count, nst, gu);
    }
    count_launches();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_status(e, "gs_bin_sort: duplicate");
    if ((e = record_kernel_event(GS_KERNEL_DUPLICATE, true, s)) != cudaSuccess)
        return cuda_status(e, "gs_bin_sort: kernel event");

    // synchronising mode: the instance and pair counts, before any further work
    uint32_t I_grid = 0;  // pairs the later kernels are sized for
    if (!graph) {
        uint64_t counts[3] = {0, 0, 0};  // instances, supertile pairs, give-up flag (adjacent in the header)
        if ((e = cudaMemcpyAsync(counts, total, sizeof(counts), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
            return cuda_status(e, "gs_bin_sort: read count");
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return cuda_status(e, "gs_bin_sort: synchronize");
        *n_instances_host = (int64_t)counts[0];
        if ((int64_t)counts[0] > capacity) {
            set_error("gs_bin_sort: %llu instances exceed capacity %lld", (unsigned long long)counts[0],
                      (long long)capacity);
            return GS_ERR_CAPACITY;
        }
        if (counts[0] == 0 || counts[2] != 0) return GS_OK;  // k_keys cleared the ranges
        I_grid = (uint32_t)counts[1];
        if ((e = cudaMemsetAsync(status, 0, 8 * 256 * (size_t)radix_tiles_max(I_grid), s)) != cudaSuccess)
            return cuda_status(e, "gs_bin_sort: clear pair-sort status");
    } else {
        if (capacity == 0) {
            k_tile_scan<<<1, kScanThreads, 0, s>>>(sv2, 0, tile_ranges, 0, fine_total, n_instances_dev, nullptr,
                                                   nullptr, err);
            count_launches();
            return cuda_status(cudaGetLastError(), "gs_bin_sort: count");
        }
        I_grid = (uint32_t)capacity;
    }

    // 4. stable sort of the pairs by supertile id: each supertile's items contiguous, in depth order
    if ((e = radix_sort(ck, cv, I_grid, ctotal, st_bits, 4, ps, &which, s)) != cudaSuccess)
        return cuda_status(e, "gs_bin_sort: supertile sort");

    // 5. per-tile counts, tile ranges, then every instance's id at its place
    // the pairs' tile masks go to the free half of the pair buffers (2 bytes per pair)
    uint16_t* masks = reinterpret_cast<uint16_t*>(ck[which ^ 1]);
    auto pair_masks = tight ? k_pair_masks<true> : k_pair_masks<false>;
    const int pair_grid = 8 * dev_sms;  // at most 8 blocks per SM, each warp taking segments of pairs
    pair_masks<<<(int)std::min<int64_t>(pair_grid, cdiv(I_grid, (int64_t)kPairBatch * (kThreads / 32))), kThreads, 0,
                 s>>>(
        sv2, mean2d, radius, ck[which], cv[which], I_grid, ctotal, (uint32_t)n, pack, masks, tile_ranges, st_count,
        st_beg, st_end, gave_up);
    count_launches();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_status(e, "gs_bin_sort: tile counts");
    k_tile_scan<<<1, kScanThreads, 0, s>>>(sv2, ntiles, tile_ranges, (uint64_t)capacity, fine_total,
                                           graph ? n_instances_dev : nullptr, st_count, st_order, err);
    count_launches();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_status(e, "gs_bin_sort: tile ranges");
    const bool sparse = st_count == nullptr;
    auto fine = keys_sorted != nullptr ? (sparse ? k_fine<true, kFineSparseWarps> : k_fine<true, kFineWarps>)
                                       : (sparse ? k_fine<false, kFineSparseWarps> : k_fine<false, kFineWarps>);
    fine<<<nst, 32 * (sparse ? kFineSparseWarps : kFineWarps), 0, s>>>(sv2, depth, ck[which], cv[which], I_grid, ctotal, pack ? 0xFFFFu : 0xFFFFFFFFu,
                                      masks, tile_ranges, st_order, st_count, st_beg, st_end, (uint32_t)n, ids_sorted,
                                      keys_sorted);
    count_launches();
    return cuda_status(cudaGetLastError(), "gs_bin_sort: write lists");
}

}  // namespace gs
