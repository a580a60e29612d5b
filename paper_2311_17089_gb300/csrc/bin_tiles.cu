// Tile lists from a depth order (Sec. 3.1: the Gaussians whose splats touch
// a tile, in the order of their view depth), as one stable counting sort by
// tile over entries that are never stored: entry e of a frame is the e-th
// (Gaussian, covered tile) pair in depth order, and its tile follows from
// its Gaussian's tile rectangle.
//
//   1. tile_items_kernel: per block of the order, each Gaussian's first
//      entry (relative to the block) and its rectangle as (first tile,
//      width); Gaussians without tiles are left out.
//   2. tile_count_kernel: the entries are cut into equal parts, one per
//      warp, at item (Gaussian) boundaries; a warp counts its part's
//      entries per tile in shared memory.  A row of the matrix holds the
//      counts of a CTA's warps together; each warp's offset within the row
//      is kept beside it.
//   3. tile_columns_kernel: the matrix's exclusive column sums plus each
//      tile's start turn every row into the positions where its entries of
//      each tile begin; the tiles' ranges come with them.
//   4. tile_rank_kernel: the parts again, now with running positions: every
//      entry's Gaussian goes straight to its place in the lists.
//
// A list holds a Gaussian at most once, so the order inside a Gaussian's
// entries does not matter.  No kernel waits on another CTA.
//
// Against what it replaced (the pairs written by a duplication pass, sorted
// by one or two 8-bit radix passes, ranges found by a further pass), kernel
// times on GB300: 1256x832, 1.78M entries, 82 -> 58 us; 628x416 at all
// levels, 14.4M entries, 445 -> 201 us; a near/far scene whose nearest
// Gaussians cover every tile, 10.0M entries, 1427 -> 174 us (there one
// block of the duplication emitted most of them alone); 157x104, 0.51M
// entries, 37 -> 30 us; 256x256, 46k entries, 24 -> 20 us.  With many
// entries the rank kernel is the larger half (144 us of the 14.4M), bound by
// the chain of shared-memory counter updates and by the 32-byte sectors its
// scattered 4-byte stores touch; staging a row's entries in shared memory to
// store runs made it 110 us but the counts 62 (shorter rows) from 37.  With
// few, the launches and their first loads are.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "bin_tiles.cuh"
#include "common.cuh"
#include "tma.cuh"

namespace msgs {
namespace {

constexpr uint32_t kAll = 0xffffffffu;
constexpr int kItemThreads = 256;
constexpr int kItemIPT = 4;
constexpr int kItemStep = kItemThreads * kItemIPT;  // order positions a block takes at a time
constexpr int kMaxBlocks = 2048;                    // blocks of the order
constexpr uint32_t kClip = 0x7fffffffu;  // entry counts saturate here, above every capacity
constexpr int kWarps = 8;                // warps of a CTA (fewer where the counters need it)
constexpr int kBatch = 256;              // entries a warp ranks at once
constexpr uint32_t kMinPart = 256;       // fewest entries per part (but for the last)
constexpr int64_t kMaxRow = 65024;       // most entries of a row with 16-bit counts (and 32 a warp)
constexpr int kCtasPerSm = 4;            // 32 warps of 64 registers
constexpr int64_t kRowTiles = 6144;      // frames up to this: a row's positions in shared memory
constexpr int kSmSmem = 224 << 10;
constexpr int kMaxSmem = 160 << 10;      // 65536 tiles: one warp, 128 KB of counts
constexpr int64_t kVecTiles = 32 * kMaxColBlocks;  // above: four columns a lane
constexpr int kColThreads = 1024;
// A matrix of at most this many words (and tiles) is summed by the count
// pass's last CTA instead of a launch of its own.  With 30 tiles and 3 rows
// the launch cost a small frame 3 us of host and device time each.
constexpr int64_t kFusedWords = 16384, kFusedTiles = 1024;

// Per block of the order: its entries, the Gaussians kept, and (written by
// the count pass) the entries before it, saturated.
struct Blocks {
    unsigned long long *sum;  // [blocks]
    uint32_t *kept;           // [blocks]
    uint32_t *pre;            // [blocks + 1]
};

inline int64_t blocks_of(int64_t n, int64_t &size) {
    size = (int64_t)kItemStep * std::max<int64_t>(1, ceil_div(n, (int64_t)kItemStep * kMaxBlocks));
    return std::max<int64_t>(1, ceil_div(n, size));
}

__device__ __forceinline__ uint32_t warp_incl(uint32_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kAll, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

struct ItemsK {
    const uint32_t *order, *n32, *n_tiles;
    const uint2 *rect;
    uint32_t n_max;
    uint32_t tiles_x, tiles;
    uint32_t block_size;
    bool vec;  // the order is 16-byte aligned
    Blocks b;
    uint2 *item;
    uint32_t *idx;
    unsigned long long *err;
};

// Items of block blockIdx.x: item[j] = (entries of the block before it,
// first tile | (width - 1) << 16), idx[j] its Gaussian, packed to the
// block's start.  idx may be the order: a block only writes positions it
// has read.  A block's entry counts saturate at kClip, above every
// capacity.  Bound by the gathers' latency (12 B of n_tiles and rectangle
// per Gaussian, two sectors).
__global__ void __launch_bounds__(kItemThreads) tile_items_kernel(ItemsK a) {
    pdl_wait();
    __shared__ uint32_t s_ent[kItemThreads / 32], s_cnt[kItemThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = min(*a.n32, a.n_max);
    const uint32_t j0 = min(n, blockIdx.x * a.block_size), j1 = min((uint64_t)n, (uint64_t)j0 + a.block_size);
    unsigned long long ents = 0;
    uint32_t kept = 0;
    for (uint32_t base = j0; base < j1; base += kItemStep) {
        uint32_t g[kItemIPT], nt[kItemIPT];
        uint2 rc[kItemIPT];
        const uint32_t j = base + (uint32_t)tid * kItemIPT;
        if (a.vec && j + kItemIPT <= j1) {
            const uint4 q = *reinterpret_cast<const uint4 *>(a.order + j);
            g[0] = q.x;
            g[1] = q.y;
            g[2] = q.z;
            g[3] = q.w;
        } else {
#pragma unroll
            for (int r = 0; r < kItemIPT; r++) g[r] = j + r < j1 ? a.order[j + r] : kAll;
        }
#pragma unroll
        for (int r = 0; r < kItemIPT; r++) {
            nt[r] = 0u;
            rc[r] = make_uint2(0u, 0u);
            if (g[r] < a.n_max) {
                nt[r] = __ldg(a.n_tiles + g[r]);
                rc[r] = __ldg(a.rect + g[r]);
            } else if (g[r] != kAll) {  // only after a wait of the sort gave up
                MS_DCHECK(false, a.err);
                atomicOr(a.err, (unsigned long long)kStatusTimeout);
            }
        }
        uint32_t se = 0, sc = 0;
#pragma unroll
        for (int r = 0; r < kItemIPT; r++) {
            // not a count or a first tile that ms_project wrote for this frame
            // (it writes them for its own camera's): reported, and left out
            if (nt[r] > a.tiles ||
                (nt[r] && (rc[r].x >> 16) * a.tiles_x + (rc[r].x & 0xffffu) >= a.tiles)) {
                MS_DCHECK(false, a.err);
                atomicOr(a.err, (unsigned long long)kStatusTimeout);
                nt[r] = 0u;
            }
            se += nt[r];
            sc += nt[r] != 0u;
        }
        // 1024 items of at most 65536 tiles: the step's entries fit 27 bits
        const uint32_t ie = warp_incl(se, lane), ic = warp_incl(sc, lane);
        if (lane == 31) {
            s_ent[warp] = ie;
            s_cnt[warp] = ic;
        }
        __syncthreads();  // also: every thread has read its part of the order
        uint32_t we = 0, wc = 0, te = 0, tc = 0;
#pragma unroll
        for (int w = 0; w < kItemThreads / 32; w++) {
            we += w < warp ? s_ent[w] : 0u;
            wc += w < warp ? s_cnt[w] : 0u;
            te += s_ent[w];
            tc += s_cnt[w];
        }
        unsigned long long e = ents + we + ie - se;
        uint32_t p = j0 + kept + wc + ic - sc;
#pragma unroll
        for (int r = 0; r < kItemIPT; r++) {
            if (nt[r] == 0u) continue;
            const uint32_t x0 = rc[r].x & 0xffffu, y0 = rc[r].x >> 16;
            const uint32_t w1 = (rc[r].y & 0xffffu) - x0;
            a.item[p] = make_uint2((uint32_t)min(e, (unsigned long long)kClip),
                                   (y0 * a.tiles_x + x0) | (w1 << 16));
            a.idx[p] = g[r];
            p++;
            e += nt[r];
        }
        ents += te;
        kept += tc;
        __syncthreads();  // s_ent / s_cnt are rewritten by the next step
    }
    if (tid == 0) {
        a.b.sum[blockIdx.x] = ents;
        a.b.kept[blockIdx.x] = kept;
    }
}

// A part: its first item (block, index in the block).
struct Part {
    uint32_t block, item;
};

struct PartsK {
    Blocks b;
    const uint2 *item;
    const uint32_t *idx;
    uint32_t block_size, n_max;
    uint32_t cap, tiles, tiles_x;
    uint32_t max_parts;     // rows x warps per row
    uint32_t cnt_words;     // words of a warp's counters, two 16-bit counts each
    uint32_t *matrix;       // element t of row r at matrix[r * stride + t * step]
    uint32_t stride, step;
    uint4 *offsets;         // [parts][cnt_words / 4]: counts of the row's warps before each
    Part *part;             // [max_parts]
    uint32_t *meta;
    bool fused;             // the count pass writes the positions and ranges
    uint32_t *ranges;
    uint32_t *tile_sums;    // [tiles >> sum_shift] zeroed: entries per 32 or 128 tiles
    int sum_shift;
    uint32_t *out;          // gauss_idx
    unsigned long long *err;
    const uint32_t *n32;    // Gaussians of the order

    __device__ uint32_t blocks_of_count() const {
        return (min(__ldg(n32), n_max) + block_size - 1u) / block_size;
    }
};
// meta: entries, parts, entries per part (written by the count pass); CTAs
// of the count pass finished (zeroed)
constexpr int kMetaEntries = 0, kMetaParts = 1, kMetaPart = 2, kMetaDone = 3;

// Walks the items of a part, 32 at a time (a lane an item, the next 32
// loading meanwhile): those from (block b, item i) on whose first entry lies
// below e1 (entries counted from the frame's first); entries from `end` on
// are dropped.  pre: entries before each block.  f(start, n, w, t0, g) per
// group: the lane's item's first entry, its entries (0: no item), width,
// first tile and Gaussian (kIdx).
template <bool kIdx, typename F>
__device__ __forceinline__ void walk_items(const PartsK &a, const uint32_t *pre, uint32_t b,
                                           uint32_t i, uint32_t e1, uint32_t end, F f) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t n_blocks = a.blocks_of_count();
    for (; b < n_blocks && pre[b] < e1; b++, i = 0u) {
        const uint32_t pb = pre[b], total = pre[b + 1] - pb, kept = a.b.kept[b];
        const uint2 *item = a.item + (size_t)b * a.block_size;
        const uint32_t *idx = a.idx + (size_t)b * a.block_size;
        uint2 v1 = make_uint2(kClip, 0u);
        uint32_t n1 = total, g1 = 0u;
        auto load = [&](uint32_t q) {
            v1 = make_uint2(kClip, 0u);
            n1 = total;
            if (q < kept) {
                v1 = item[q];
                if (kIdx) g1 = idx[q];
                if (q + 1u < kept) n1 = item[q + 1u].x;
            }
        };
        load(i + lane);
        for (uint32_t q = i + lane;; q += 32u) {
            const uint2 v = v1;
            const uint32_t next = n1, g = g1;
            load(q + 32u);
            const bool in = q < kept && v.x < e1 - pb;
            // the frame's last entry may cut its item
            const uint32_t n = in ? min(next, end - pb) - v.x : 0u;
            f(pb + v.x, n, (v.y >> 16) + 1u, v.y & 0xffffu, g);
            if (!__all_sync(kAll, in)) break;
        }
    }
}

// Items of more tiles than this are taken by the whole warp, a lane a tile.
constexpr uint32_t kBigItem = 16;

// The row and column of tile m of an item of width w (inv = 1 / w): exact,
// since m < 2^16 keeps the quotient's error below half a tile's 1 / w.
__device__ __forceinline__ uint32_t item_tile(uint32_t t0, uint32_t m, uint32_t w, float inv,
                                              uint32_t tiles_x) {
    const uint32_t y = (uint32_t)(((float)m + 0.5f) * inv);
    return t0 + y * tiles_x + (m - y * w);
}

// CTA c counts parts c W .. c W + W - 1, W its warps, which share row c.
__global__ void __launch_bounds__(32 * kWarps, kCtasPerSm) tile_count_kernel(PartsK a) {
    pdl_wait();
    extern __shared__ __align__(16) uint32_t s_mem[];
    __shared__ uint32_t s_pre[kMaxBlocks + 1];
    __shared__ unsigned long long s_scan[kWarps];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5, W = blockDim.x >> 5;
    uint32_t *cnt = s_mem + w * a.cnt_words;
    {
        uint4 *c4 = reinterpret_cast<uint4 *>(cnt);
        for (uint32_t k = lane; k < a.cnt_words / 4u; k += 32u) c4[k] = make_uint4(0u, 0u, 0u, 0u);
    }
    // entries before every block of the order that holds any: consecutive
    // blocks per thread, one scan
    const uint32_t n_blocks = a.blocks_of_count();
    {
        const uint32_t per = (n_blocks + blockDim.x - 1u) / blockDim.x;
        const uint32_t b0 = min(n_blocks, tid * per), b1 = min(n_blocks, b0 + per);
        unsigned long long sum = 0;
#pragma unroll 8
        for (uint32_t b = b0; b < b1; b++) sum += a.b.sum[b];
        unsigned long long x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kAll, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31u) s_scan[w] = x;
        __syncthreads();
        unsigned long long run = x - sum;
        for (uint32_t k = 0; k < w; k++) run += s_scan[k];
        for (uint32_t b = b0; b < b1; b++) {
            s_pre[b] = (uint32_t)min(run, (unsigned long long)kClip);
            run += a.b.sum[b];
        }
        if (tid == blockDim.x - 1u) s_pre[n_blocks] = (uint32_t)min(run, (unsigned long long)kClip);
        __syncthreads();
    }
    const uint32_t E = min(s_pre[n_blocks], a.cap);
    const uint32_t part = (max(kMinPart, (E + a.max_parts - 1u) / a.max_parts) + 31u) & ~31u;
    const uint32_t parts = (E + part - 1u) / part;
    if (blockIdx.x == 0) {
        for (uint32_t b = tid; b <= n_blocks; b += blockDim.x) a.b.pre[b] = s_pre[b];
        if (tid == 0) {
            a.meta[kMetaEntries] = E;
            a.meta[kMetaParts] = parts;
            a.meta[kMetaPart] = part;
        }
    }
    const uint32_t rows = (parts + W - 1u) / W;
    if (blockIdx.x >= rows) {
        if (rows == 0u && a.fused && blockIdx.x == 0)  // no entry at all
            for (uint32_t t = tid; t < 2u * a.tiles; t += blockDim.x) a.ranges[t] = 0u;
        return;
    }
    const uint32_t p = blockIdx.x * W + w;
    if (p < parts) {
        // the first item that starts at or past the part's first entry
        const uint32_t e0 = p * part, e1 = min(E, e0 + part);
        uint32_t b = 0, hi = n_blocks;  // s_pre[b] <= e0 < s_pre[hi]
        while (hi - b > 1u) {
            const uint32_t mid = (b + hi) >> 1;
            if (s_pre[mid] <= e0) b = mid;
            else hi = mid;
        }
        uint32_t i = 0u;
        const uint32_t f0 = e0 - s_pre[b];
        if (f0 > 0u) {
            const uint2 *item = a.item + (size_t)b * a.block_size;
            uint32_t l = 0, h = a.b.kept[b];  // item[l] starts before f0
            while (h - l > 1u) {
                const uint32_t step = (h - l + 31u) / 32u, q = l + (lane + 1u) * step;
                const uint32_t c = __popc(__ballot_sync(kAll, q < h && item[q].x < f0));
                l += c * step;
                h = min(h, l + step);
            }
            i = l + 1u;
        }
        if (lane == 0) a.part[p] = {b, i};
        auto add = [&](uint32_t t) {
            if (t < a.tiles) {
                atomicAdd(cnt + (t >> 1), 1u << (16u * (t & 1u)));
            } else {  // not a rectangle ms_project wrote for this frame
                MS_DCHECK(false, a.err);
                atomicOr(a.err, (unsigned long long)kStatusTimeout);
            }
        };
        walk_items<false>(a, s_pre, b, i, e1, E,
                          [&](uint32_t, uint32_t n, uint32_t wd, uint32_t t0, uint32_t) {
            if (n <= kBigItem) {
                uint32_t t = t0, x = 0u;
                for (uint32_t m = 0; m < n; m++) {
                    add(t);
                    t++;
                    if (++x == wd) {
                        x = 0u;
                        t += a.tiles_x - wd;
                    }
                }
            }
            const float inv = 1.0f / (float)wd;
            for (uint32_t big = __ballot_sync(kAll, n > kBigItem); big; big &= big - 1u) {
                const int l = __ffs(big) - 1;
                const uint32_t bn = __shfl_sync(kAll, n, l), bw = __shfl_sync(kAll, wd, l);
                const uint32_t bt = __shfl_sync(kAll, t0, l);
                const float bi = __shfl_sync(kAll, inv, l);
                for (uint32_t m = lane; m < bn; m += 32u) add(item_tile(bt, m, bw, bi, a.tiles_x));
            }
        });
    }
    __syncthreads();
    // two tiles a word: the counts of the row's warps before each warp, and
    // the row's own (a row's entries fit 16 bits)
    uint32_t *row = a.matrix + (size_t)blockIdx.x * a.stride;
    uint32_t *off = reinterpret_cast<uint32_t *>(a.offsets) + (size_t)blockIdx.x * W * a.cnt_words;
    for (uint32_t k0 = 0; k0 < a.cnt_words; k0 += blockDim.x) {
        const uint32_t k = k0 + tid;
        uint32_t run = 0;
        if (k < a.cnt_words) {
            for (uint32_t v = 0; v < W; v++) {
                if (W > 1u) off[v * a.cnt_words + k] = run;
                run += s_mem[v * a.cnt_words + k];
            }
            if (2u * k < a.tiles) row[(size_t)(2u * k) * a.step] = run & 0xffffu;
            if (2u * k + 1u < a.tiles) row[(size_t)(2u * k + 1u) * a.step] = run >> 16;
        }
        // 16 lanes hold 32 tiles
        uint32_t sum = (run & 0xffffu) + (run >> 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(kAll, sum, o);
        if (!a.fused && (lane & 15u) == 0u && sum)
            atomicAdd(a.tile_sums + ((2u * k) >> a.sum_shift), sum);
    }
    if (!a.fused) return;
    // the last CTA: every tile's rows, then the tiles' starts (consecutive
    // tiles per thread), then the positions
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(a.meta + kMetaDone, 1u) == rows - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (2u * a.tiles <= blockDim.x) {
        // few tiles, so up to 16384 / tiles rows: G threads share a tile's,
        // a run of them each (one thread per tile took 50 of this kernel's
        // 63-76 us for 1M entries in 1 to 15 tiles)
        const uint32_t G = min(32u, blockDim.x / a.tiles);
        const uint32_t g = tid / a.tiles, t = tid - g * a.tiles;
        const uint32_t len = (rows + G - 1u) / G, r0 = min(rows, g * len);
        const uint32_t r1 = g < G ? min(rows, r0 + len) : r0;
        uint32_t *part = s_pre + 32, *start = part + 256;  // [G][tiles], [tiles]
        uint32_t c = 0, before = 0, total = 0;
#pragma unroll 8
        for (uint32_t r = r0; r < r1; r++)
            c += __ldcg(a.matrix + (size_t)r * a.stride + (size_t)t * a.step);
        if (g < G) part[tid] = c;
        __syncthreads();
        if (g < G) {
            for (uint32_t k = 0; k < G; k++) {
                const uint32_t v = part[k * a.tiles + t];
                before += k < g ? v : 0u;
                total += v;
            }
        }
        const uint32_t mine = g == 0u ? total : 0u, incl = warp_incl(mine, (int)lane);
        if (lane == 31u) s_pre[w] = incl;
        __syncthreads();
        if (g == 0u) {
            uint32_t run = incl - mine;
            for (uint32_t k = 0; k < w; k++) run += s_pre[k];
            start[t] = run;
            a.ranges[2u * t] = total ? run : 0u;
            a.ranges[2u * t + 1u] = total ? run + total : 0u;
        }
        __syncthreads();
        if (a.step != 1u || g >= G) return;
        uint32_t at = start[t] + before;
        for (uint32_t q = r0; q < r1; q += 8u) {
            uint32_t v[8];
#pragma unroll
            for (uint32_t i = 0; i < 8u; i++)
                v[i] = q + i < r1 ? __ldcg(a.matrix + (size_t)(q + i) * a.stride + t) : 0u;
#pragma unroll
            for (uint32_t i = 0; i < 8u; i++)
                if (q + i < r1) {
                    a.matrix[(size_t)(q + i) * a.stride + t] = at;
                    at += v[i];
                }
        }
        return;
    }
    const uint32_t per = (a.tiles + blockDim.x - 1u) / blockDim.x;
    const uint32_t t0 = min(a.tiles, tid * per), t1 = min(a.tiles, t0 + per);
    uint32_t sum = 0;
    for (uint32_t t = t0; t < t1; t++) {
        uint32_t c = 0;
#pragma unroll 8
        for (uint32_t r = 0; r < rows; r++)
            c += __ldcg(a.matrix + (size_t)r * a.stride + (size_t)t * a.step);
        s_mem[t] = c;
        sum += c;
    }
    const uint32_t incl = warp_incl(sum, (int)lane);
    if (lane == 31u) s_pre[w] = incl;
    __syncthreads();
    uint32_t run = incl - sum;
    for (uint32_t k = 0; k < w; k++) run += s_pre[k];
    for (uint32_t t = t0; t < t1; t++) {
        const uint32_t c = s_mem[t];
        if (a.step == 1u) {
            uint32_t at = run;
            for (uint32_t r0 = 0; r0 < rows; r0 += 8u) {
                uint32_t v[8];
#pragma unroll
                for (uint32_t i = 0; i < 8u; i++)
                    v[i] = r0 + i < rows ? __ldcg(a.matrix + (size_t)(r0 + i) * a.stride + t) : 0u;
#pragma unroll
                for (uint32_t i = 0; i < 8u; i++)
                    if (r0 + i < rows) {
                        a.matrix[(size_t)(r0 + i) * a.stride + t] = at;
                        at += v[i];
                    }
            }
        }
        a.ranges[2u * t] = c ? run : 0u;
        a.ranges[2u * t + 1u] = c ? run + c : 0u;
        run += c;
    }
}

struct ColK {
    uint32_t *matrix;
    uint32_t stride, step, tiles, row_warps;
    const uint32_t *meta;
    const uint32_t *tile_sums;
    uint32_t *ranges;
};

// 32 columns of the matrix per block, a lane per column (kVec = 1), or 128,
// four a lane (kVec = 4), its 32 warps a thirty-second of the rows each:
// column sums, the block's start (the sum of the blocks' entries before it),
// then the rows again, each count replaced by its position.  Bound by the
// latency of its two rounds of loads; kColAhead rows are in flight per warp.
constexpr int kColAhead = 8;

template <int kVec>
__global__ void __launch_bounds__(kColThreads) tile_columns_kernel(ColK a) {
    pdl_wait();
    constexpr int kColWarps = kColThreads / 32;
    constexpr int kAhead = kColAhead / kVec;
    __shared__ uint32_t s_sum[kColWarps][32 * kVec];
    __shared__ uint32_t s_start;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t col = (blockIdx.x * 32u + lane) * kVec;
    const uint32_t parts = a.meta[kMetaParts];
    const uint32_t rows = (parts + a.row_warps - 1u) / a.row_warps;
    const uint32_t per = (rows + kColWarps - 1) / kColWarps;
    const uint32_t r0 = min(rows, warp * per), r1 = col < a.tiles ? min(rows, r0 + per) : r0;
    uint32_t *m = a.matrix + (size_t)col * a.step;
    if (threadIdx.x == 0) s_start = 0u;
    // rows r .. r + kAhead - 1 of this lane's columns
    uint32_t v[kAhead][kVec];
    auto load = [&](uint32_t r) {
#pragma unroll
        for (int i = 0; i < kAhead; i++) {
            const uint32_t *p = m + (size_t)(r + i) * a.stride;
            if (r + i < r1) {
                if (kVec == 4 && a.step == 1u) {
                    // a row's columns past the tiles, up to its stride, are not used
                    const uint4 q = __ldcg(reinterpret_cast<const uint4 *>(p));
                    v[i][0] = q.x;
                    v[i][1 % kVec] = q.y;
                    v[i][2 % kVec] = q.z;
                    v[i][3 % kVec] = q.w;
                } else {
#pragma unroll
                    for (int c = 0; c < kVec; c++)
                        v[i][c] = col + c < a.tiles ? __ldcg(p + c * a.step) : 0u;
                }
            } else {
#pragma unroll
                for (int c = 0; c < kVec; c++) v[i][c] = 0u;
            }
        }
    };
    uint32_t sum[kVec];
#pragma unroll
    for (int c = 0; c < kVec; c++) sum[c] = 0u;
    for (uint32_t r = r0; r < r1; r += kAhead) {
        load(r);
#pragma unroll
        for (int i = 0; i < kAhead; i++)
#pragma unroll
            for (int c = 0; c < kVec; c++) sum[c] += v[i][c];
    }
#pragma unroll
    for (int c = 0; c < kVec; c++) s_sum[warp][lane * kVec + c] = col + c < a.tiles ? sum[c] : 0u;
    // entries of the blocks before this one (kMaxColBlocks <= kColThreads)
    const uint32_t prev = __reduce_add_sync(
        kAll, threadIdx.x < blockIdx.x ? __ldcg(a.tile_sums + threadIdx.x) : 0u);
    __syncthreads();
    if (lane == 0 && prev) atomicAdd(&s_start, prev);
    uint32_t before[kVec], total[kVec], mine = 0;
#pragma unroll
    for (int c = 0; c < kVec; c++) {
        before[c] = total[c] = 0u;
#pragma unroll 8
        for (int w = 0; w < kColWarps; w++) {
            const uint32_t x = s_sum[w][lane * kVec + c];
            before[c] += w < (int)warp ? x : 0u;
            total[c] += x;
        }
        mine += total[c];
    }
    const uint32_t incl = warp_incl(mine, (int)lane);
    __syncthreads();
    uint32_t run[kVec];
    uint32_t begin = s_start + incl - mine;  // the first column's first position
#pragma unroll
    for (int c = 0; c < kVec; c++) {
        run[c] = begin + before[c];
        if (warp == 0 && col + c < a.tiles) {
            a.ranges[2 * (col + c)] = total[c] ? begin : 0u;
            a.ranges[2 * (col + c) + 1] = total[c] ? begin + total[c] : 0u;
        }
        begin += total[c];
    }
    // a matrix of one row that lies in the ranges is its positions now
    if (a.step != 1u) return;
    for (uint32_t r = r0; r < r1; r += kAhead) {
        load(r);
#pragma unroll
        for (int i = 0; i < kAhead; i++) {
            if (r + i >= r1) break;
            uint32_t o[kVec];
#pragma unroll
            for (int c = 0; c < kVec; c++) {
                o[c] = run[c];
                run[c] += v[i][c];
            }
            uint32_t *p = m + (size_t)(r + i) * a.stride;
            if constexpr (kVec == 4) *reinterpret_cast<uint4 *>(p) = make_uint4(o[0], o[1], o[2], o[3]);
            else *p = o[0];
        }
    }
}

// The parts again, in order.  A group of 32 items with at most kBatch
// entries writes its entries (tile | lane << 16) to shared memory and ranks
// them 32 at a time: lanes with the same tile (warp match) take consecutive
// positions.  A group of more entries goes item by item, a lane a tile,
// where no two lanes meet.  A tile's next position is the row's plus the
// warp's 16-bit running offset; kRowSmem: the row lies in shared memory.
template <bool kRowSmem>
__global__ void __launch_bounds__(32 * kWarps, kCtasPerSm) tile_rank_kernel(PartsK a) {
    pdl_wait();
    extern __shared__ __align__(16) uint32_t s_mem[];
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, W = blockDim.x >> 5;
    const uint32_t parts = a.meta[kMetaParts];
    if (blockIdx.x * W >= parts) return;
    const uint32_t p = blockIdx.x * W + w;
    const uint32_t E = a.meta[kMetaEntries], part = a.meta[kMetaPart];
    uint16_t *cnt = reinterpret_cast<uint16_t *>(s_mem + w * a.cnt_words);
    uint32_t *entry = s_mem + W * a.cnt_words + w * kBatch;
    uint32_t *s_row = s_mem + W * (a.cnt_words + kBatch);  // [tiles]
    const uint32_t *row = a.matrix + (size_t)blockIdx.x * a.stride;
    // the row and the warps' offsets arrive by bulk copies (every size and
    // address a multiple of 16 bytes); a row in the ranges has its words two
    // apart, and a row of one warp no offsets
    __shared__ __align__(8) uint64_t s_bar;
    const uint32_t off_bytes = W > 1u ? W * a.cnt_words * 4u : 0u;
    const uint32_t row_bytes = kRowSmem && a.step == 1u ? a.stride * 4u : 0u;
    if (threadIdx.x == 0) {
        mbar_init(&s_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(&s_bar, off_bytes + row_bytes);
        if (row_bytes) bulk_copy_g2s(s_row, row, row_bytes, &s_bar);
        if (off_bytes)
            bulk_copy_g2s(s_mem, a.offsets + (size_t)blockIdx.x * W * (a.cnt_words / 4u), off_bytes,
                          &s_bar);
    }
    if (kRowSmem && a.step != 1u)
        for (uint32_t k = threadIdx.x; k < a.tiles; k += blockDim.x)
            s_row[k] = __ldcg(row + (size_t)k * a.step);
    if (W == 1u)
        for (uint32_t k = lane; k < a.cnt_words; k += 32u) s_mem[k] = 0u;
    const Part first = p < parts ? a.part[p] : Part{0u, 0u};
    __syncthreads();
    bool landed = false;
    for (uint32_t spins = 0; spins < kSpinLimit && !landed; spins++) landed = mbar_try_wait(&s_bar, 0u);
    if (!landed) {  // the copies are still out: the lists are not valid
        atomicOr(a.err, (unsigned long long)kStatusTimeout);
        for (uint32_t spins = 0; spins < kSpinLimit && !landed; spins++)
            landed = mbar_try_wait(&s_bar, 0u);
        return;
    }
    if (p < parts) {
        const uint32_t le = kAll >> (31u - lane);  // lanes up to this one
        auto base_of = [&](uint32_t t) {
            return kRowSmem ? s_row[t] : __ldcg(row + (size_t)t * a.step);
        };
        auto put = [&](uint32_t to, uint32_t g) {
            if (to < E) {
                a.out[to] = g;
            } else {  // the lists' order was not one
                MS_DCHECK(false, a.err);
                atomicOr(a.err, (unsigned long long)kStatusTimeout);
            }
        };
        walk_items<true>(a, a.b.pre, first.block, first.item, min(E, p * part + part), E,
                         [&](uint32_t start, uint32_t n, uint32_t wd, uint32_t t0, uint32_t g) {
            const uint32_t s0 = __shfl_sync(kAll, start, 0);
            const uint32_t most = __reduce_max_sync(kAll, n);
            const uint32_t total = __reduce_max_sync(kAll, n ? start - s0 + n : 0u);
            if (total <= kBatch && most <= 32u) {
                uint32_t t = t0, x = 0u;
                for (uint32_t m = 0; m < n; m++) {
                    entry[start - s0 + m] = min(t, a.tiles - 1u) | (lane << 16);
                    t++;
                    if (++x == wd) {
                        x = 0u;
                        t += a.tiles_x - wd;
                    }
                }
                __syncwarp();
#pragma unroll 2
                for (uint32_t k = lane; k - lane < total; k += 32u) {
                    const bool ok = k < total;
                    const uint32_t v = ok ? entry[k] : 0u;
                    const uint32_t tile = v & 0xffffu;
                    const uint32_t gk = __shfl_sync(kAll, g, (int)(v >> 16));
                    const uint32_t peers = __match_any_sync(kAll, ok ? tile : kAll);
                    uint32_t at = 0u, from = 0u;
                    if (ok) {
                        at = cnt[tile];
                        from = base_of(tile);
                    }
                    __syncwarp();
                    // the last of the peers moves the tile's offset on
                    if (ok && (peers & ~le) == 0u) cnt[tile] = (uint16_t)(at + __popc(peers));
                    __syncwarp();
                    if (ok) put(from + at + __popc(peers & (le >> 1)), gk);
                }
                __syncwarp();
                return;
            }
            // four items at a time: their tiles and bases first, then their
            // offsets in order
            const float inv = 1.0f / (float)wd;
            const uint32_t items = __popc(__ballot_sync(kAll, n != 0u));
            for (uint32_t l = 0; l < items; l += 4u) {
                uint32_t bn[4], bw[4], bt[4], bg[4], t[4], to[4];
                float bi[4];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int src = (int)((l + j) & 31u);
                    bn[j] = __shfl_sync(kAll, n, src);
                    bw[j] = __shfl_sync(kAll, wd | (t0 << 16), src);
                    bg[j] = __shfl_sync(kAll, g, src);
                    bi[j] = __shfl_sync(kAll, inv, src);
                    bt[j] = bw[j] >> 16;
                    bw[j] &= 0xffffu;
                    if (l + j >= items) bn[j] = 0u;
                }
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    t[j] = min(item_tile(bt[j], lane, bw[j], bi[j], a.tiles_x), a.tiles - 1u);
                    to[j] = lane < bn[j] ? base_of(t[j]) : 0u;
                }
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    if (lane < bn[j]) {
                        const uint32_t at = cnt[t[j]];
                        cnt[t[j]] = (uint16_t)(at + 1u);
                        put(to[j] + at, bg[j]);
                    }
                    for (uint32_t m = lane + 32u; m < bn[j]; m += 32u) {
                        const uint32_t tm =
                            min(item_tile(bt[j], m, bw[j], bi[j], a.tiles_x), a.tiles - 1u);
                        const uint32_t at = cnt[tm];
                        cnt[tm] = (uint16_t)(at + 1u);
                        put(base_of(tm) + at, bg[j]);
                    }
                    __syncwarp();
                }
            }
        });
    }
}

// How a frame's entries are cut and counted.
struct Cut {
    bool in_ranges, row_smem;
    int warps;          // per CTA and row
    int64_t rows;       // at most
    uint32_t cnt_words;
    int64_t stride;
    size_t count_smem, rank_smem;
};

// Warps per row: kWarps, or what leaves two CTAs per SM their shared memory
// (16-bit counters: 2 bytes a tile and warp).  Rows: what the SMs hold at
// once, but enough of them that a row's entries fit 16-bit counts, no more
// than minimal parts of the capacity fill (CTAs without a row kept the other
// frames' kernels of an 8-frame sweep waiting), and no more than the matrix
// has room for; with room for none (a capacity below
// about a quarter of the tiles) one row of one warp lies in the ranges.
Cut cut_of(int64_t tiles, int64_t cap, size_t matrix_bytes) {
    Cut c;
    c.stride = (tiles + 3) & ~(int64_t)3;
    c.cnt_words = (uint32_t)(((tiles + 1) / 2 + 3) & ~(int64_t)3);
    c.row_smem = tiles <= kRowTiles;
    const size_t row_b = c.row_smem ? (size_t)c.stride * 4 : 0;
    const size_t warp_b = ((size_t)c.cnt_words + kBatch) * 4;
    c.warps = (int)std::max<size_t>(
        1, std::min<size_t>(kWarps, ((size_t)(kSmSmem / 2 - 1024) - row_b) / warp_b));
    int64_t want = 0, room = 0;
    for (;;) {
        c.rank_smem = c.warps * warp_b + row_b;
        const int64_t ctas = std::max<int64_t>(
            1, std::min<int64_t>(kCtasPerSm, (int64_t)(kSmSmem / (c.rank_smem + 1024))));
        want = std::max<int64_t>(ctas * num_sms(), ceil_div(cap, kMaxRow));
        // a row: its counts, its warps' offsets and parts
        const size_t row_bytes = (size_t)c.stride * 4 +
                                 (c.warps > 1 ? (size_t)c.warps * c.cnt_words * 4 : 0) +
                                 (size_t)c.warps * sizeof(Part);
        room = (int64_t)(matrix_bytes / row_bytes);
        if (room >= 1 || c.warps == 1) break;
        c.warps = 1;  // little room: a row of one warp needs no offsets
    }
    c.in_ranges = room < 1;
    c.rows = c.in_ranges ? 1 : std::min({want, room, ceil_div(cap, (int64_t)kMinPart * c.warps)});
    // (and, where the count pass sums the columns, a word per tile)
    c.count_smem = std::max<size_t>((size_t)c.warps * c.cnt_words,
                                    tiles <= kFusedTiles ? (size_t)c.stride : 0) * 4;
    return c;
}

}  // namespace

int64_t tile_block_count(int64_t n) {
    int64_t size;
    return blocks_of(n, size);
}

int launch_tile_lists(const TileListArgs &t, cudaStream_t st) {
    int rc;
    int64_t size;
    const int64_t nb = blocks_of(t.n, size);
    const Cut cut = cut_of(t.tiles, t.cap, t.matrix_bytes);
    Blocks b;
    b.sum = t.block_sums;
    b.kept = t.block_words;
    b.pre = b.kept + nb;
    ItemsK ik;
    ik.order = t.order;
    ik.n32 = t.n32;
    ik.n_tiles = t.n_tiles;
    ik.rect = t.rect;
    ik.n_max = (uint32_t)t.n;
    ik.tiles_x = (uint32_t)t.tiles_x;
    ik.tiles = (uint32_t)t.tiles;
    ik.block_size = (uint32_t)size;
    ik.vec = aligned(t.order, 16);
    ik.b = b;
    ik.item = t.item;
    ik.idx = t.idx;
    ik.err = t.err;
    if ((rc = cuda_check(launch_after(tile_items_kernel, (unsigned)nb, kItemThreads, 0, st, ik), "tile items")))
        return rc;
    PartsK pk;
    pk.b = b;
    pk.item = t.item;
    pk.idx = t.idx;
    pk.block_size = (uint32_t)size;
    pk.n_max = (uint32_t)t.n;
    pk.n32 = t.n32;
    pk.cap = (uint32_t)t.cap;
    pk.tiles = (uint32_t)t.tiles;
    pk.tiles_x = (uint32_t)t.tiles_x;
    pk.max_parts = (uint32_t)(cut.rows * cut.warps);
    pk.cnt_words = cut.cnt_words;
    pk.matrix = cut.in_ranges ? t.ranges : t.matrix;
    pk.stride = (uint32_t)cut.stride;
    pk.step = cut.in_ranges ? 2u : 1u;
    // behind the matrix: the rows' warps' offsets, then the parts; the one
    // part of a row in the ranges has its words behind the blocks'
    uint32_t *behind = t.matrix + cut.rows * cut.stride;
    pk.offsets = reinterpret_cast<uint4 *>(behind);
    if (cut.warps > 1) behind += cut.rows * cut.warps * cut.cnt_words;
    pk.part = reinterpret_cast<Part *>(cut.in_ranges ? t.block_words + 2 * nb + 2 : behind);
    pk.meta = t.meta;
    pk.tile_sums = t.tile_sums;
    pk.sum_shift = t.tiles > kVecTiles ? 7 : 5;
    pk.out = t.gauss_idx;
    pk.err = t.err;
    void (*rank)(PartsK) = cut.row_smem ? tile_rank_kernel<true> : tile_rank_kernel<false>;
    if ((rc = ensure_smem_attr(reinterpret_cast<const void *>(tile_count_kernel), kMaxSmem)) ||
        (rc = ensure_smem_attr(reinterpret_cast<const void *>(rank), kMaxSmem)))
        return rc;
    const unsigned grid = (unsigned)cut.rows, threads = 32u * (unsigned)cut.warps;
    pk.fused = t.tiles <= kFusedTiles && cut.rows * t.tiles <= kFusedWords;
    pk.ranges = t.ranges;
    if ((rc = cuda_check(launch_after(tile_count_kernel, grid, threads, cut.count_smem, st, pk), "tile counts")))
        return rc;
    ColK ck;
    ck.matrix = pk.matrix;
    ck.stride = pk.stride;
    ck.step = pk.step;
    ck.tiles = pk.tiles;
    ck.row_warps = (uint32_t)cut.warps;
    ck.meta = t.meta;
    ck.tile_sums = t.tile_sums;
    ck.ranges = t.ranges;
    if (!pk.fused) {
        const bool vec = t.tiles > kVecTiles;
        if ((rc = cuda_check(launch_after(vec ? tile_columns_kernel<4> : tile_columns_kernel<1>,
                                          (unsigned)ceil_div(t.tiles, vec ? 128 : 32), kColThreads, 0,
                                          st, ck),
                             "tile columns")))
            return rc;
    }
    return cuda_check(launch_after(rank, grid, threads, cut.rank_smem, st, pk), "tile ranks");
}

}  // namespace msgs
