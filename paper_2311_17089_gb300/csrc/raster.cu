// Front-to-back blending per 16x16 tile (Sec. 3.1; Eq. 3 with incremental
// transmittance T_k): a 256-thread CTA walks a segment of a tile's sorted
// list, one thread per pixel.
//
// Load balance: low resolutions put thousands of splats on a few tiles
// (Sec. 3.2, item 2), so one CTA per tile would leave most SMs idle.  Each
// tile's list is cut into segments of seg_len = max(kMinSegment, D /
// resident CTAs) entries; only tiles longer than a fair share of the work
// are split.
// A CTA walks its segment in sub-batches of kChunk records, double-buffered:
// the next sub-batch arrives in shared memory (cp.async, a record per
// thread, on an mbarrier) while the current one is blended.  A sub-batch's
// records are first tested against the tile's sixteen 4x4 pixel blocks; each
// half warp then blends only those that reach its block, four at a time.
//
// Bound by instruction issue where the SMs are full (1256x832: 175M warp
// instructions, 74% of the issue slots), by a deep tile's serial walk where
// they are not.  GB300, kernel times before (8x4 blocks by box test, record
// pairs regrouped through shared memory, per-record bulk copies) and now:
// 1256x832 of 1M Gaussians 242 -> 206 us, 628x416 at all levels 88 -> 72,
// 256x256 of 10k 42 -> 38, near/far 3M 700 -> 631.  The copies alone made
// 241 -> 219 and 820 -> 726 (the bulk engine takes 48-byte copies one by
// one).  Two pixels per thread (8x8 blocks per warp, packed arithmetic)
// issued as much and lengthened the deep walks (3M: 870 to 1130 us).
//
// The blend stays exactly sequential across segments (decoupled look-back):
//   - a segment whose predecessor has published its inclusive prefix
//     starts from that per-pixel (C, T) and applies the termination rule
//     directly;
//   - otherwise it blends from T = 1 into a local aggregate (C_l, T_l),
//     publishes it, and folds forward from the nearest published prefix
//     over the aggregates after it to get its exact (C_in, T_in).  If no
//     termination can fall inside the segment (T_in T_l >= 1e-4, T being
//     monotone) the result is C_in + T_in C_l, T_in T_l; otherwise the pixel
//     terminates inside the segment: it is handed on as terminated at once,
//     and the segment is walked again from T_in to find the exact stopping
//     point.
// Each pixel is written by the segment it terminates in, or by its tile's
// last segment.  A segment after which every pixel has terminated marks
// the tile done; later segments of that tile stop as soon as they see the
// mark.  Every wait is bounded; a wait that gives
// up sets a status bit and the CTA carries on.
#include <cuda_runtime.h>

#include <atomic>
#include <stdint.h>

#include "common.cuh"
#include "tma.cuh"
#include "raster_ws.cuh"
#include "raster_list.cuh"
#include "reach.cuh"

namespace msgs {

constexpr int kRecBytes = 48;                // one raster record
constexpr int kBufBytes = kChunk * kRecBytes;  // staged records, as copied
constexpr float kAlphaMax = 0.99f;
constexpr float kTStop = 1e-4f;
#ifndef MS_RASTER_WINDOW
#define MS_RASTER_WINDOW 16
#endif
// Segments of one tile walked at once: segment k starts when segment k - W
// has published its result (or the tile is done).  Pixels of low-resolution
// frames terminate long before the end of their tile's list, and every
// segment started past that point is wasted work.
constexpr uint32_t kWindow = MS_RASTER_WINDOW;
constexpr uint32_t kAgg = 1u;                // segment flag: local aggregate published
constexpr uint32_t kPre = 2u;                // segment flag: inclusive prefix published
// ms_raster (AUTO) launches both blend kernels for frames with at least as
// many tiles as SMs and fewer than kListBandSms times as many, and the list
// kernel takes the frame when its mean list length lies in kListMeanMin ..
// kListMeanMax.
constexpr int64_t kListBandSms = 4;
constexpr uint32_t kListMeanMin = 1024;
constexpr uint32_t kListMeanMax = 8192;

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Loads from shared memory at a 32-bit address plus a constant ("memory":
// after the stores that wrote it, in the compiler's order too).
template <int kOff>
__device__ __forceinline__ float4 lds4(uint32_t p) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4 + %5];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(p), "n"(kOff)
                 : "memory");
    return v;
}
template <int kOff>
__device__ __forceinline__ float2 lds2(uint32_t p) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2 + %3];"
                 : "=f"(v.x), "=f"(v.y)
                 : "r"(p), "n"(kOff)
                 : "memory");
    return v;
}

__device__ __forceinline__ uint2 lds_offsets(uint32_t p) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                 : "=r"(v.x), "=r"(v.y)
                 : "r"(p)
                 : "memory");
    return v;
}

struct RasterArgs {
    const uint32_t *ranges;
    const uint32_t *gidx;
    const float4 *rec;
    uint32_t n_rec;
    int W, H, tiles_x, tiles;
    float bg0, bg1, bg2;
    float *image;
    float *final_t;
    uint32_t *n_contrib;
    uint32_t *n_eval;
    uint32_t *seg_off;    // [tiles + 1] exclusive prefix of segments per tile
    uint32_t *seg_len;    // [1] entries per segment (a multiple of kChunk)
    uint32_t *ticket;
    uint32_t *flags;      // [max_segs] 0, kAgg (local aggregate), kPre (prefix)
    uint32_t *tile_done;  // [tiles] every pixel terminated, image written
    float4 *agg;          // [max_segs][256] local (C0, C1, C2, T) from T = 1
    uint2 *agg2;          // [max_segs][256] (n_contrib, n_eval | term bit)
    float4 *pre;          // [max_segs][256] inclusive (C0, C1, C2, T)
    uint2 *pre2;          // [max_segs][256] (n_contrib, n_eval | term bit)
    const uint32_t *use_list;  // NULL, or nonzero when the list kernel blends this frame instead
    unsigned long long *err;
};

struct Seg {
    uint32_t t, k, nk, start, len;
};

// Segment c's tile and list entries; called by whole warps, whose lanes
// search together.
__device__ __forceinline__ Seg seg_of(const RasterArgs &a, uint32_t c, uint32_t L) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t lo = 0, hi = (uint32_t)a.tiles;  // seg_off[lo] <= c < seg_off[hi]
    while (hi - lo > 1u) {
        const uint32_t step = (hi - lo + 31u) / 32u, q = lo + (lane + 1u) * step;
        const uint32_t n =
            __popc(__ballot_sync(0xffffffffu, q < hi && a.seg_off[q] <= c));
        lo += n * step;
        hi = min(hi, lo + step);
    }
    Seg sg;
    sg.t = lo;
    sg.k = c - a.seg_off[lo];
    sg.nk = a.seg_off[lo + 1] - a.seg_off[lo];
    uint32_t s = a.ranges[2 * lo], e = a.ranges[2 * lo + 1];
    sg.start = s + sg.k * L;
    uint32_t stop = min(e, sg.start + L);
    sg.len = stop > sg.start ? stop - sg.start : 0;
    return sg;
}

// One block: D = sum of list lengths, segment length L = max(kChunk,
// ceil(D / resident) rounded up to kChunk), then the number of segments of
// every tile (at least one, so empty tiles still write the background),
// exclusive-scanned.  It also zeroes the n_zero16 16-byte words at zero (the
// tile kernel's ticket, segment flags and tile marks; none for the list
// kernel), which the raster launch after it reads.  With use_list, it
// writes there which blend kernel takes the frame: the list kernel when the
// mean list length D / tiles lies in list_mean_min .. list_mean_max, else
// the tile kernel.
__global__ void __launch_bounds__(1024)
segment_offsets_kernel(const uint32_t *ranges, int tiles, uint32_t resident,
                       uint32_t *__restrict__ off, uint32_t *__restrict__ seg_len,
                       uint4 *__restrict__ zero, uint32_t n_zero16,
                       uint32_t *__restrict__ use_list, uint32_t list_mean_min,
                       uint32_t list_mean_max) {
    __shared__ uint32_t s_warp[32];
    __shared__ unsigned long long s_total;
    pdl_wait<false>();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (tiles + 1023) / 1024;
    const int t0 = tid * per;
    // the thread's list lengths, the first kKeep of them read once (frames
    // of up to 8192 tiles); the ranges are read beside the zeroing's stores
    constexpr int kKeep = 8;
    uint32_t keep[kKeep];
#pragma unroll
    for (int k = 0; k < kKeep; k++) {
        const int t = t0 + k;
        keep[k] = k < per && t < tiles ? ranges[2 * t + 1] - ranges[2 * t] : 0u;
    }
    auto rest = [&](int t) { return ranges[2 * t + 1] - ranges[2 * t]; };
    const int t1 = min(tiles, t0 + per);
    for (uint32_t i = tid; i < n_zero16; i += 1024) zero[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) s_total = 0;
    __syncthreads();
    unsigned long long d = 0;
#pragma unroll
    for (int k = 0; k < kKeep; k++) d += keep[k];
    for (int t = t0 + kKeep; t < t1; t++) d += rest(t);
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if (lane == 0 && d) atomicAdd(&s_total, d);
    __syncthreads();
    unsigned long long share = (s_total + resident - 1) / (resident > 0 ? resident : 1);
    uint32_t L = (uint32_t)(((share + kChunk - 1) / kChunk) * kChunk);
    if (L < kMinSegment) L = kMinSegment;
    auto segs = [&](uint32_t len) { return len > L ? (len + L - 1) / L : 1u; };
    uint32_t sum = 0;
#pragma unroll
    for (int k = 0; k < kKeep; k++)
        if (t0 + k < t1) sum += segs(keep[k]);
    for (int t = t0 + kKeep; t < t1; t++) sum += segs(rest(t));
    uint32_t x = sum;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t v = s_warp[lane];
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        s_warp[lane] = v;
    }
    __syncthreads();
    uint32_t run = x - sum + (warp > 0 ? s_warp[warp - 1] : 0u);
#pragma unroll
    for (int k = 0; k < kKeep; k++)
        if (t0 + k < t1) {
            off[t0 + k] = run;
            run += segs(keep[k]);
        }
    for (int t = t0 + kKeep; t < t1; t++) {
        off[t] = run;
        run += segs(rest(t));
    }
    pdl_next();
    if (tid == 1023) {
        off[tiles] = run;
        seg_len[0] = L;
        if (use_list)
            use_list[0] = s_total >= (unsigned long long)list_mean_min * (unsigned long long)tiles &&
                          s_total <= (unsigned long long)list_mean_max * (unsigned long long)tiles;
    }
}

struct PixelState {
    float C0, C1, C2, T;
    uint32_t last, evals;
    bool term;
};

// A warp covers an 8x4 block of pixels, each half warp a 4x4 one with its
// own list of the records that reach it.  (Of the lane slots of an 8x4
// block's records, about 37% are accepted by their pixel on the 1M-Gaussian
// scene at 1256x832, of a 4x4 block's half.)
constexpr int kWarps = kRasterThreads / 32;
constexpr int kGroup = 4;  // records blended at a time; a list is padded to it
constexpr int kListLen = kChunk + 2 * kGroup;  // (and read a group ahead)
// Dynamic shared memory: two staging buffers, a record that no pixel accepts
// (the lists' padding), the records' block masks, and the half warps' lists.
constexpr int kMaskOff = 2 * kBufBytes + kRecBytes;
constexpr int kListOff = kMaskOff + kChunk * 2;
constexpr int kSmemBytes = kListOff + kWarps * 2 * kListLen * 2;
// The chords and extents below bound the pixels a record is accepted at
// (reach.cuh); the margin covers the rounding of their own last operations
// and of the distances (a few 2^-24 of the record's extents: 0.06 px at 10^5).
#ifndef MS_CULL_MARGIN
#define MS_CULL_MARGIN 0.0625f
#endif
constexpr float kInf = __builtin_huge_valf();

// Bits 4 k + j, k = 0, 1: some pixel centre of the tile's 4x4 block (j, row
// band b0 + k) may have alpha >= 1/255.  (x, y): the record's centre relative
// to the tile's corner.  Over a band of pixel rows the rows' intervals of
// reach.cuh span an x interval whose ends are chords' ends: the right end
// is largest at the row of the ellipse's rightmost point (dx = ex, dy = -B ex /
// 2C), so over the band at the nearest row to that; the left end likewise
// with the signs turned.  Without an ellipse a chord's end is a convex
// function of its row, largest at the band's first or last.  A conic without
// usable curvature, or NaN, keeps every block.
__device__ __forceinline__ uint32_t blocks_reached(float x, float y, float A, float B, float C,
                                                   float thr, int b0) {
    if (!reach_curved(A, C)) return 0xffu;
    float ex, ey;
    const bool bounded = reach_extents(A, B, C, thr, ex, ey);
    const float den = reach_det(A, B, C), top = A * reach_thr(thr);
    const float yr = -0.5f * ex * __fdividef(B, C);  // dy of the rightmost point
    const float ia = __fdividef(-0.5f, A), slope = ia * B;
    uint32_t bits = 0u;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        // the band's pixel centres relative to the record's
        const float yl = (float)(4 * (b0 + k)) + 0.5f - y, yh = yl + 3.0f;
        auto chord = [&](float dy, float side) {  // the end of the chord at dy
            return fmaf(side, sqrt_approx(fmaxf(fmaf(-den, dy * dy, top), 0.0f)), slope * dy);
        };
        float x1, x0;
        if (bounded) {
            if (yl > ey + MS_CULL_MARGIN || yh < -ey - MS_CULL_MARGIN) continue;
            const float r = fminf(yh, fmaxf(yl, yr)), l = fminf(yh, fmaxf(yl, -yr));
            x1 = r != yr ? chord(r, ia) : ex;
            x0 = l != -yr ? chord(l, -ia) : -ex;
        } else {
            x1 = fmaxf(chord(yl, ia), chord(yh, ia));
            x0 = fminf(chord(yl, -ia), chord(yh, -ia));
        }
        x1 += x + MS_CULL_MARGIN;
        x0 += x - MS_CULL_MARGIN;
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (!(4.0f * j + 0.5f > x1) && !(4.0f * j + 3.5f < x0)) bits |= 1u << (4 * k + j);
    }
    return bits;
}

// The records of the staged sub-batch whose block mask has the half warp's
// bit, as byte offsets in list order, for both halves of the warp (bits
// `bit` and bit + 1), padded with the record at `pad` to a common multiple
// of kGroup, which is returned.  Any other record has alpha < 1/255 at every pixel of the
// block, so skipping it changes nothing.
__device__ __forceinline__ uint32_t compact(const uint16_t *__restrict__ masks, uint32_t bit,
                                            uint16_t *lists, uint32_t pad) {
    const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
    uint32_t n[2] = {0u, 0u};
#pragma unroll
    for (int k = 0; k < kChunk / 32; k++) {
        const uint32_t i = (uint32_t)k * 32u + lane;
        const uint32_t bits = (uint32_t)masks[i] >> bit;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint32_t m = __ballot_sync(0xffffffffu, (bits >> h) & 1u);
            if ((bits >> h) & 1u) lists[h * kListLen + n[h] + __popc(m & lt)] = (uint16_t)(i * kRecBytes);
            n[h] += __popc(m);
        }
    }
    const uint32_t len = (max(n[0], n[1]) + kGroup - 1u) & ~(uint32_t)(kGroup - 1);
#pragma unroll
    for (int h = 0; h < 2; h++)
        for (uint32_t k = n[h] + lane; k < len; k += 32u) lists[h * kListLen + k] = (uint16_t)pad;
    __syncwarp();
    return len;
}

// A pixel being blended: y is its row's centre, or +inf once it has ended
// (or lies outside the image): every power is then -inf or NaN and no record
// is accepted.
struct Pix {
    float T, C0, C1, C2, y;
    uint32_t last, evals;
};

// power * log2(e) = A dx^2 + B dx dy + C dy^2 of a record at the pixel.
__device__ __forceinline__ float power_of(const float4 r0, float C, float fx, float y) {
    const float dx = __fsub_rn(fx, r0.x), dy = __fsub_rn(y, r0.y);
    const float u = __fmaf_rn(r0.w, dy, __fmul_rn(r0.z, dx));
    return __fmaf_rn(__fmul_rn(C, dy), dy, __fmul_rn(dx, u));
}

// One record: skipped if the power is positive or alpha below 1/255 (power *
// log2(e) < thr); stop before a Gaussian that would bring T below 1e-4, else
// accumulate and advance T.  pos: 1 + its list position.
__device__ __forceinline__ void blend_one(const float4 *__restrict__ r, float fx, uint32_t pos,
                                          Pix &s) {
    const float4 r1 = r[1], r2 = r[2];
    const float p = power_of(r[0], r1.x, fx, s.y);
    if (!(p <= 0.0f && p >= r2.y)) return;
    const float al = fminf(kAlphaMax, __fmul_rn(r1.y, ex2_approx(p)));
    const float Tn = __fmaf_rn(-al, s.T, s.T);
    if (Tn < kTStop) {
        s.y = kInf;
        s.evals = pos;
        return;
    }
    const float w = __fmul_rn(al, s.T);
    s.C0 = __fmaf_rn(w, r1.z, s.C0);
    s.C1 = __fmaf_rn(w, r1.w, s.C1);
    s.C2 = __fmaf_rn(w, r2.x, s.C2);
    s.T = Tn;
    s.last = pos;
}

// Blend the half warp's listed records (n, the same for both halves) into
// the thread's pixel; pos0 is the list position of the sub-batch's first
// record.  kGroup records at a time: all their alphas (0 where not accepted,
// which leaves T and the colour as they are; independent of T, so their
// loads and arithmetic overlap), then T through the group and one test
// whether it ends a pixel of the warp, whose weights are then formed again
// up to the record that ends it; then the colours.  About 27 instructions a
// record.  `odd`: some record's colour is not finite (it must not meet a
// zero weight) or its power may round above 0: one record at a time.
__device__ __forceinline__ void blend_list(const unsigned char *__restrict__ aos,
                                           const uint16_t *__restrict__ list, uint32_t n, bool odd,
                                           uint32_t pos0, float fx, Pix &s) {
    if (odd) {
        for (uint32_t m = 0; m < n; m++) {
            const uint32_t o = list[m];
            blend_one(reinterpret_cast<const float4 *>(aos + o), fx,
                      pos0 + o / (uint32_t)kRecBytes + 1u, s);
        }
        return;
    }
    const uint32_t base = smem_addr(aos);
    uint32_t last = 0xffffu;  // offset of the last blended record
    const uint32_t at = smem_addr(list);
    static_assert(kGroup == 4, "a group's offsets are one 8-byte load");
    uint2 next = lds_offsets(at);
    for (uint32_t m = 0; m < n; m += kGroup) {
        const uint2 ii = next;
        next = lds_offsets(at + 2u * (m + kGroup));  // of the next group
        const uint32_t o[kGroup] = {ii.x & 0xffffu, ii.x >> 16, ii.y & 0xffffu, ii.y >> 16};
        float al[kGroup], w[kGroup], c[kGroup][3];
#pragma unroll
        for (int k = 0; k < kGroup; k++) {
            const uint32_t r = base + o[k];
            const float4 r1 = lds4<16>(r);
            const float2 r2 = lds2<32>(r);
            const float p = power_of(lds4<0>(r), r1.x, fx, s.y);
            const float a = fminf(kAlphaMax, __fmul_rn(r1.y, ex2_approx(p)));
            al[k] = p >= r2.y ? a : 0.0f;
            c[k][0] = r1.z;
            c[k][1] = r1.w;
            c[k][2] = r2.x;
        }
        float T = s.T;
#pragma unroll
        for (int k = 0; k < kGroup; k++) {
            w[k] = __fmul_rn(al[k], T);
            T = __fmaf_rn(-al[k], T, T);
        }
        const bool ends = T < kTStop;
        const uint32_t any = __ballot_sync(0xffffffffu, ends);
        if (any) {
            if (ends) {
                T = s.T;
#pragma unroll
                for (int k = 0; k < kGroup; k++) {
                    const float Tn = __fmaf_rn(-al[k], T, T);
                    if (s.y != kInf && Tn < kTStop) {
                        s.y = kInf;
                        s.evals = pos0 + o[k] / (uint32_t)kRecBytes + 1u;
                    }
                    const bool on = s.y != kInf;
                    w[k] = on ? __fmul_rn(al[k], T) : 0.0f;
                    T = on ? Tn : T;
                }
            }
            __syncwarp();
        }
#pragma unroll
        for (int k = 0; k < kGroup; k++) {
            s.C0 = __fmaf_rn(w[k], c[k][0], s.C0);
            s.C1 = __fmaf_rn(w[k], c[k][1], s.C1);
            s.C2 = __fmaf_rn(w[k], c[k][2], s.C2);
            if (w[k] != 0.0f) last = o[k];
        }
        s.T = T;
        if (any && !__any_sync(0xffffffffu, s.y != kInf)) break;
    }
    if (last != 0xffffu) s.last = pos0 + last / (uint32_t)kRecBytes + 1u;
}

// The first kChunk threads copy their records (g: a thread's list entry)
// into the buffer and arrive on its mbarrier once their copies have landed
// (a thread without a record at once); the caller guarantees that every warp
// is done reading the buffer.
__device__ __forceinline__ void issue_batch(const RasterArgs &a, uint32_t g, uint32_t cnt,
                                            float4 *buf, uint64_t *bar) {
    MS_DCHECK(cnt <= (uint32_t)kChunk, a.err);
    if (threadIdx.x < (uint32_t)kChunk) {
        if (threadIdx.x < cnt) {
            MS_DCHECK(g < a.n_rec, a.err);
            if (g >= a.n_rec) g = 0;  // unreachable unless binning reported an error
            const float4 *src = a.rec + 3 * (size_t)g;
            float4 *dst = buf + 3 * threadIdx.x;
            cp_async16(dst, src);
            cp_async16(dst + 1, src + 1);
            cp_async16(dst + 2, src + 2);
        }
        cp_async_arrive(bar);
    }
}

__device__ __forceinline__ bool wait_batch(const RasterArgs &a, uint64_t *bar, uint32_t parity) {
    for (uint32_t spins = 0; spins < kSpinLimit; spins++)
        if (mbar_try_wait(bar, parity)) return true;
    atomicOr(a.err, (unsigned long long)kStatusTimeout);
    for (uint32_t spins = 0; spins < kSpinLimit; spins++)  // copies still in flight
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// The state of tile pixel slot `i` (fwd_index) after segment c.
__device__ __forceinline__ PixelState load_state(const float4 *v, const uint2 *v2, uint32_t c,
                                                 int i) {
    float4 st = __ldcg(v + (size_t)c * kRasterThreads + i);
    uint2 st2 = __ldcg(v2 + (size_t)c * kRasterThreads + i);
    PixelState s = {st.x, st.y, st.z, st.w, st2.x, st2.y & ~kTermBit, (st2.y & kTermBit) != 0};
    return s;
}

__device__ __forceinline__ void store_state(float4 *v, uint2 *v2, uint32_t c, int i,
                                            const PixelState &s) {
    v[(size_t)c * kRasterThreads + i] = make_float4(s.C0, s.C1, s.C2, s.T);
    v2[(size_t)c * kRasterThreads + i] = make_uint2(s.last, s.evals | (s.term ? kTermBit : 0u));
}

// The exact state after one more segment, from the state P before it and
// the segment's local result X (blended from T = 1).  A pixel terminates in
// the segment when X terminated locally or P.T X.T < 1e-4 (T is monotone);
// its colour then needs a re-walk, the fold only records the termination.
// Every segment folds with this one function in list order, so all of them
// reach bit-identical prefixes and the same termination decisions.
__device__ __forceinline__ PixelState fold(const PixelState &P, const PixelState &X) {
    if (P.term) return P;
    PixelState r = P;
    if (X.term || P.T * X.T < kTStop) {
        r.term = true;
        return r;
    }
    r.C0 = fmaf(P.T, X.C0, P.C0);
    r.C1 = fmaf(P.T, X.C1, P.C1);
    r.C2 = fmaf(P.T, X.C2, P.C2);
    r.T = P.T * X.T;
    r.last = X.last != 0 ? X.last : P.last;
    r.evals = X.evals;
    return r;
}

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t *p) {
    return *reinterpret_cast<const volatile uint32_t *>(p);
}

// Walk one segment in sub-batches through two staging buffers: while the
// warps mask, list and blend the records of sub-batch j in one buffer, the
// cp.async copies of sub-batch j + 1 land in the other and the list entries of
// sub-batch j + 2 are read.  Two CTA barriers per sub-batch: after the block
// masks, and with the termination test, when every warp is done with
// sub-batch j.  In local mode (`exact` false) the walk stops as soon as the
// tile is marked done.  The CTA stops early once every pixel has
// terminated.  Returns kWalked, kAborted.  A copy wait that gives up sets
// the status word and ends the waiting warps' pixels; the walk stays in
// step across the CTA.
constexpr int kWalked = 0, kAborted = 1;
__device__ __forceinline__ int run_segment(const RasterArgs &a, const Seg &sg, uint32_t L,
                                           bool exact, bool active, float fx, float fy, int tx,
                                           int ty, PixelState &s, unsigned char *smem,
                                           uint64_t *bar, uint32_t &par, uint32_t *s_abort) {
    const uint32_t pos0 = sg.k * L;
    if (sg.len == 0) return kWalked;
    const uint32_t nb = (sg.len + kChunk - 1) / kChunk;
    const uint32_t tid = threadIdx.x, wid = tid >> 5;
    float4 *aos = reinterpret_cast<float4 *>(smem);
    unsigned char *masks = smem + kMaskOff;
    uint16_t *lists = reinterpret_cast<uint16_t *>(smem + kListOff) + wid * 2u * kListLen;
    auto entry = [&](uint32_t j) {  // this thread's list entry of sub-batch j
        const uint32_t i = j * kChunk + tid;
        return tid < (uint32_t)kChunk && i < sg.len ? __ldg(a.gidx + sg.start + i) : 0u;
    };
    Pix q = {s.T, s.C0, s.C1, s.C2, active && !s.term ? fy : kInf, s.last, s.evals};
    issue_batch(a, entry(0), min(sg.len, (uint32_t)kChunk), aos, &bar[0]);
    uint32_t next = entry(1);
    bool abort = false;
    for (uint32_t j = 0; j < nb; j++) {
        const uint32_t b = j & 1u, off = j * kChunk;
        const uint32_t cnt = min(sg.len - off, (uint32_t)kChunk);
        const bool ok = wait_batch(a, &bar[b], (par >> b) & 1u);
        par ^= 1u << b;
        const bool more = j + 1 < nb;
        if (more) {
            issue_batch(a, next, min(sg.len - off - kChunk, (uint32_t)kChunk),
                        aos + (b ^ 1u) * 3 * kChunk, &bar[b ^ 1u]);
            next = entry(j + 2);
        }
        // a copy wait that gave up has set the status word: the warp's pixels
        // stop here (their result is reported wrong), the walk goes on in
        // step with the other warps
        if (!__all_sync(0xffffffffu, ok)) q.y = kInf;
        // the block masks: a thread takes one record and two of the tile's
        // four row bands
        const float4 *buf = aos + b * 3 * kChunk;
        bool bad = false;
        {
            const uint32_t i = tid & (uint32_t)(kChunk - 1), band = (tid / kChunk) * 2u;
            uint32_t bits = 0u;
            if (i < cnt) {
                const float4 r0 = buf[3 * i], r1 = buf[3 * i + 1];
                const float2 r2 = *reinterpret_cast<const float2 *>(buf + 3 * i + 2);
                bits = blocks_reached(r0.x - (float)(tx * 16), r0.y - (float)(ty * 16), r0.z, r0.w,
                                      r1.x, r2.y, (int)band);
                // B^2 below 4 A C by more than the power's rounding, a few
                // 2^-24 of its terms: it cannot come out positive
                bad = !((r1.z + r1.w + r2.x) * 0.0f == 0.0f) ||
                      !(r0.w * r0.w < 3.99998474f * r0.z * r1.x);
            }
            masks[2u * i + tid / kChunk] = (unsigned char)bits;
        }
        const bool odd = __syncthreads_or(bad) != 0;
        // warps whose pixels have all terminated skip their share
        if (__any_sync(0xffffffffu, q.y != kInf)) {
            const uint32_t n = compact(reinterpret_cast<const uint16_t *>(masks),
                                       (wid >> 1) * 4u + (wid & 1u) * 2u, lists, (2u - b) * kBufBytes);
            blend_list(reinterpret_cast<const unsigned char *>(buf),
                       lists + ((tid >> 4) & 1u) * kListLen, n, odd, pos0 + off, fx, q);
            if (q.y != kInf) q.evals = pos0 + off + cnt;
        }
        // two slots: a warp may still be reading sub-batch j's value while
        // thread 0 writes sub-batch j + 1's
        if (tid == 0) s_abort[b] = exact ? 0u : ld_volatile(a.tile_done + sg.t);
        const int ended = __syncthreads_and(q.y == kInf);
        abort = s_abort[b] != 0;
        if (ended || abort) {
            if (more) {  // drain the copies already issued
                wait_batch(a, &bar[b ^ 1u], (par >> (b ^ 1u)) & 1u);
                par ^= 1u << (b ^ 1u);
            }
            break;
        }
    }
    if (active) s = {q.C0, q.C1, q.C2, q.T, q.last, q.evals, q.y == kInf};
    return abort ? kAborted : kWalked;
}

__global__ void __launch_bounds__(kRasterThreads, 4)  // 64 registers: 4 CTAs per SM
raster_kernel(RasterArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t s_next;
    __shared__ uint32_t s_flag;
    __shared__ uint32_t s_wait;
    __shared__ uint32_t s_abort[2];
    pdl_wait();
    if (a.use_list && *a.use_list) return;  // the list kernel blends this frame
    const int tid = threadIdx.x;
    if (tid < kRecBytes / 4)  // the padding record: no power reaches its threshold
        reinterpret_cast<float *>(smem + 2 * kBufBytes)[tid] = tid == 9 ? kInf : 0.0f;
    if (tid == 0) {
        mbar_init(&bar[0], kChunk);
        mbar_init(&bar[1], kChunk);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const uint32_t total = a.seg_off[a.tiles];
    const uint32_t L = a.seg_len[0];
    uint32_t parity = 0u;  // phase parity of bar[0] (bit 0) and bar[1] (bit 1)
    for (;;) {
        __syncthreads();
        if (tid == 0) s_next = atomicAdd(a.ticket, 1u);
        __syncthreads();
        const uint32_t c = s_next;
        if (c >= total) break;
        const Seg sg = seg_of(a, c, L);
        if (sg.k >= kWindow) {
            // wait for the segment kWindow places earlier in this tile; it
            // holds an earlier ticket, so its CTA is running
            if (tid == 0) {
                uint32_t skip = 0, spins = 0;
                for (;;) {
                    if (ld_volatile(a.flags + c - kWindow) != 0) break;
                    if (ld_volatile(a.tile_done + sg.t)) {
                        skip = 1;
                        break;
                    }
                    if (++spins > kSpinLimit) {
                        atomicOr(a.err, (unsigned long long)kStatusTimeout);
                        break;
                    }
                    __nanosleep(64);
                }
                s_wait = skip;
            }
            __syncthreads();
            if (s_wait) continue;  // an earlier segment finished the tile
        }
        const uint32_t prev = c - 1;
        bool exact = sg.k == 0;
        if (!exact) {
            if (tid == 0)
                s_flag = ld_volatile(a.tile_done + sg.t) ? 3u : ld_acquire(a.flags + prev);
            __syncthreads();
            if (s_flag == 3u) continue;  // an earlier segment finished the tile
            exact = s_flag == kPre;
        }
        const int tx = sg.t % a.tiles_x, ty = sg.t / a.tiles_x;
        // each warp covers an 8x4 pixel block (2 x 4 blocks per tile), each
        // half of it a 4x4 one: close pixels accept and terminate alike
        const int wid = tid >> 5, lid = tid & 31;
        const int lx = (wid & 1) * 8 + (lid >> 4) * 4 + (lid & 3);
        const int ly = (wid >> 1) * 4 + ((lid >> 2) & 3);
        const int slot = fwd_index(lx, ly);
        const int px = tx * 16 + lx, py = ty * 16 + ly;
        const bool inside = px < a.W && py < a.H;
        const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
        PixelState s = {0.0f, 0.0f, 0.0f, 1.0f, 0u, sg.k * L, false};
        bool was_term = false;  // terminated in an earlier segment (already written)
        if (sg.k > 0 && exact) {
            s = load_state(a.pre, a.pre2, prev, slot);
            was_term = s.term;
        }
        // pass 0 walks the segment (exact from the predecessor's prefix, or
        // locally from T = 1); pass 1 re-walks it from the exact prefix for
        // the pixels that terminate inside it, after the prefix is published
        bool active = inside, skip = false, redone = false;
        const bool last_seg = sg.k + 1 == sg.nk;
        for (int pass = 0; pass < 2; pass++) {
            const int rc = run_segment(a, sg, L, exact || pass == 1, active, fx, fy, tx, ty, s,
                                       smem, bar, parity, s_abort);
            if (rc == kAborted) {
                skip = true;  // an earlier segment finished the tile
                break;
            }
            if (pass == 1) break;
            bool redo = false;
            PixelState in = s;
            if (!exact) {
                // publish the local aggregate, then look back: the nearest
                // predecessor with a published prefix, and the aggregates
                // after it
                store_state(a.agg, a.agg2, c, slot, s);
                __threadfence();
                __syncthreads();
                if (tid == 0) {
                    st_release(a.flags + c, kAgg);
                    // batched look-back over the flags of up to 16
                    // predecessors; the tile's first segment never publishes
                    // an aggregate, so the walk ends there at the latest
                    const uint32_t c0 = c - sg.k;
                    uint32_t j = prev, spins = 0, res = 0;
                    for (;;) {
                        uint32_t pre_mask = 0, agg_mask = 0;
#pragma unroll
                        for (int i = 0; i < 16; i++) {
                            const uint32_t f = (j >= c0 + i) ? ld_relaxed(a.flags + j - i) : 0u;
                            pre_mask |= (uint32_t)(f == kPre) << i;
                            agg_mask |= (uint32_t)(f == kAgg) << i;
                        }
                        // leading run of aggregates, then a prefix or a gap
                        const uint32_t run = __ffs(~agg_mask) - 1;
                        j -= run;
                        if (run < 16 && ((pre_mask >> run) & 1u)) {
                            fence_acquire();  // the states behind the flags seen
                            break;
                        }
                        if (run < 16) {
                            // j has published nothing yet
                            if (ld_volatile(a.tile_done + sg.t)) {
                                res = 1u;
                                break;
                            }
                            if (++spins > kSpinLimit) {
                                atomicOr(a.err, (unsigned long long)kStatusTimeout);
                                res = 1u;
                                break;
                            }
                            __nanosleep(32);
                        }
                    }
                    s_flag = res;
                    s_next = j;
                }
                __syncthreads();
                if (s_flag) {
                    skip = true;
                    break;
                }
                const uint32_t j = s_next;
                in = load_state(a.pre, a.pre2, j, slot);
                // fold the aggregates after j, four loads in flight at a time;
                // stop once every pixel is known to have terminated before this
                // segment (the segments it terminated in write it)
                uint32_t i = j + 1;
                for (; i + 4 <= c; i += 4) {
                    PixelState x0 = load_state(a.agg, a.agg2, i, slot);
                    PixelState x1 = load_state(a.agg, a.agg2, i + 1, slot);
                    PixelState x2 = load_state(a.agg, a.agg2, i + 2, slot);
                    PixelState x3 = load_state(a.agg, a.agg2, i + 3, slot);
                    in = fold(fold(fold(fold(in, x0), x1), x2), x3);
                    if (__syncthreads_and(in.term || !inside)) {
                        i = c;
                        break;
                    }
                }
                for (; i < c; i++) in = fold(in, load_state(a.agg, a.agg2, i, slot));
                if (in.term) {
                    s = in;
                    was_term = true;
                } else if (!s.term && in.T * s.T >= kTStop) {
                    s = fold(in, s);
                } else {
                    // the pixel terminates inside this segment: successors
                    // only need to know that; its exact result comes next
                    redo = inside;
                    s.term = true;
                }
            }
            // publish the inclusive prefix before any re-walk, so no
            // successor ever waits for one
            const bool all_done = __syncthreads_and(s.term || !inside);
            if (!last_seg) {
                if (!all_done) store_state(a.pre, a.pre2, c, slot, s);
                __threadfence();
                __syncthreads();
                if (tid == 0) st_release(all_done ? a.tile_done + sg.t : a.flags + c,
                                         all_done ? 1u : kPre);
            }
            if (!__syncthreads_or(redo)) break;
            if (redo) s = in;
            active = redo;
            redone = redo;
        }
        if (skip) continue;
        // every pixel is written once: by the segment it terminates in, or
        // by the tile's last segment
        if (inside && !was_term && (s.term || last_seg || redone)) {
            const size_t p = (size_t)py * a.W + px, plane = (size_t)a.W * a.H;
            MS_DCHECK(p < plane, a.err);
            a.image[p] = fmaf(s.T, a.bg0, s.C0);
            a.image[plane + p] = fmaf(s.T, a.bg1, s.C1);
            a.image[2 * plane + p] = fmaf(s.T, a.bg2, s.C2);
            if (a.final_t) a.final_t[p] = s.T;
            if (a.n_contrib) a.n_contrib[p] = s.last;
            if (a.n_eval) a.n_eval[p] = s.evals;
        }
    }
}

static int raster_blocks_per_sm() {
    // the same for every device of the one architecture this library targets
    static std::atomic<int> blocks_per_sm{0};
    int b = blocks_per_sm.load(std::memory_order_relaxed);
    if (b == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, raster_kernel, kRasterThreads,
                                                          kSmemBytes) != cudaSuccess ||
            b < 1)
            b = 1;
        blocks_per_sm.store(b, std::memory_order_relaxed);
    }
    return b;
}

}  // namespace msgs

using namespace msgs;

extern "C" size_t ms_raster_workspace_bytes(int64_t tiles, int64_t dup_capacity) {
    RasterLayout L;
    if (!raster_layout(tiles, dup_capacity, L)) return 0;
    return L.total;
}

extern "C" int ms_raster_ex2(const ms_proj_t *proj, const ms_bins_t *bins,
                             const ms_camera_t *cam, float *image, float *final_t,
                             uint32_t *n_contrib, uint32_t *n_eval, void *ws, size_t ws_bytes,
                             int strategy, int32_t max_ctas_per_sm, void *stream) {
    if (strategy < MS_RASTER_AUTO || strategy > MS_RASTER_GROUP32)
        return fail(MS_ERR_INVALID_ARG, "unknown raster strategy");
    if (max_ctas_per_sm < 0) return fail(MS_ERR_INVALID_ARG, "max_ctas_per_sm must be >= 0");
    if (!proj || !bins || !cam || !image) return fail(MS_ERR_INVALID_ARG, "NULL argument");
    if (cam->width < 1 || cam->height < 1 || cam->width > 32768 || cam->height > 32768)
        return fail(MS_ERR_INVALID_ARG, "image size must be 1..32768");
    if (!proj->rec || !aligned(proj->rec, 16)) return fail(MS_ERR_INVALID_ARG, "rec NULL or misaligned");
    if (!bins->gauss_idx || !bins->ranges || !bins->counts)
        return fail(MS_ERR_INVALID_ARG, "bins buffers NULL");
    if (proj->n < 1 || proj->n > INT32_MAX)
        return fail(MS_ERR_INVALID_ARG, "ms_proj_t n must be 1..2^31-1");
    const int tiles_x = (cam->width + 15) / 16, tiles_y = (cam->height + 15) / 16;
    const int64_t tiles = (int64_t)tiles_x * tiles_y;
    RasterLayout L;
    if (!raster_layout(tiles, bins->dup_capacity, L))
        return fail(MS_ERR_INVALID_ARG, "tiles or dup_capacity out of range");
    if (!ws || ws_bytes < L.total || !aligned(ws, 16))
        return fail(MS_ERR_INVALID_ARG, "raster workspace missing, too small or misaligned");
    cudaStream_t st = as_stream(stream);
    char *w = static_cast<char *>(ws);
    int rc;
    if ((rc = ensure_smem_attr(reinterpret_cast<const void *>(raster_kernel), kSmemBytes)))
        return rc;
    // the tile kernel's persistent CTAs: as many as fit, or at most
    // max_ctas_per_sm per SM so that other frames' kernels find room beside it
    const int per_sm = max_ctas_per_sm > 0 ? std::min(raster_blocks_per_sm(), (int)max_ctas_per_sm)
                                           : raster_blocks_per_sm();
    const int resident = (int)std::min<int64_t>((int64_t)per_sm * num_sms(), kMaxResident);
    // A frame with fewer tiles than SMs would leave SMs without a tile: the
    // tile kernel then splits every list into many segments, most of them
    // blended speculatively, and the list kernel is faster.  Up to
    // kListBandSms x SMs tiles (and no cap on the tile kernel's CTAs), the
    // frame's mean list length decides on the device (both kernels are
    // launched, the one not chosen returns at once): lists of
    // kListMeanMin .. kListMeanMax entries per tile (selective frames, whose
    // pixels walk deep into them) go to the list kernel; short ones, which
    // the tile kernel walks quickly, and long ones (all levels, whose
    // pixels end early in lists whose first kMaskPrefix entries the list
    // kernel's mask pass covers whole) to the tile kernel.  Measured on
    // GB300, this call alone on two 1M-Gaussian scenes: 314x208 selective
    // (260 tiles, 3.5-4.0k entries each) list 130 and 139 us against tile
    // 175 and 169; 157x104 (70 tiles) list 66 against tile 117 and 126; all
    // levels at 314x208 (18k entries) tile 67 and 81 against list 195 and
    // 221; the 256x256 single-level frame (180 entries) tile 48 against
    // list 65.  The limits were chosen with an earlier, slower tile kernel:
    // at 418x277 (486 tiles, 2.5-3.1k entries) the present one would take
    // 143 and 156 us where the list kernel takes 207 and 198.
    // The group kernels are chosen only explicitly: on selective frames they
    // are slower than the kernel chosen here (8 lanes at 314x208: 171 to 191
    // us).
    const int64_t sms = num_sms();
    const int group = strategy == MS_RASTER_GROUP8    ? 8
                      : strategy == MS_RASTER_GROUP16 ? 16
                      : strategy == MS_RASTER_GROUP32 ? 32
                                                      : 0;
    const bool auto_list = strategy == MS_RASTER_AUTO && tiles < sms;
    // a cap on the tile kernel's CTAs (frames blended side by side) keeps
    // the tile kernel: the list kernel cannot leave SMs to other frames; so
    // does a duplicate capacity below kListMeanMin entries per tile, which
    // rules the list kernel out before the lists are known
    const bool band = strategy == MS_RASTER_AUTO && !auto_list && max_ctas_per_sm == 0 &&
                      tiles < kListBandSms * sms &&
                      bins->dup_capacity >= (int64_t)kListMeanMin * tiles;
    const bool list = group > 0 || strategy == MS_RASTER_LIST || auto_list;
    RasterArgs a;
    a.ranges = bins->ranges;
    a.gidx = bins->gauss_idx;
    a.rec = reinterpret_cast<const float4 *>(proj->rec);
    a.n_rec = (uint32_t)proj->n;
    a.W = cam->width;
    a.H = cam->height;
    a.tiles_x = tiles_x;
    a.tiles = (int)tiles;
    a.bg0 = cam->bg[0];
    a.bg1 = cam->bg[1];
    a.bg2 = cam->bg[2];
    a.image = image;
    a.final_t = final_t;
    a.n_contrib = n_contrib;
    a.n_eval = n_eval;
    a.seg_off = reinterpret_cast<uint32_t *>(w + L.seg_off);
    a.seg_len = reinterpret_cast<uint32_t *>(w + L.seg_len);
    a.ticket = reinterpret_cast<uint32_t *>(w + L.ticket);
    a.flags = reinterpret_cast<uint32_t *>(w + L.flags);
    a.tile_done = reinterpret_cast<uint32_t *>(w + L.tile_done);
    a.agg = reinterpret_cast<float4 *>(w + L.agg);
    a.agg2 = reinterpret_cast<uint2 *>(w + L.agg2);
    a.pre = reinterpret_cast<float4 *>(w + L.pre);
    a.pre2 = reinterpret_cast<uint2 *>(w + L.pre2);
    uint32_t *use_list = band ? reinterpret_cast<uint32_t *>(w + L.use_list) : nullptr;
    a.use_list = use_list;
    a.err = reinterpret_cast<unsigned long long *>(bins->counts) + kCntStatus;
    // the segmentation is the same for both kernels: the backward walks it
    // the tile kernel's ticket, flags and tile marks are zeroed by the first
    // kernel (the workspace and zero_bytes are 256-byte aligned)
    if ((rc = cuda_check(launch_after(segment_offsets_kernel, 1, 1024, 0, st, bins->ranges, (int)tiles,
                                      (uint32_t)resident, a.seg_off, a.seg_len,
                                      reinterpret_cast<uint4 *>(w),
                                      list ? 0u : (uint32_t)(L.zero_bytes / 16), use_list,
                                      kListMeanMin, kListMeanMax),
                         "segment offsets launch")))
        return rc;
    if (list || band) {
        ListArgs la;
        la.ranges = a.ranges;
        la.gidx = a.gidx;
        la.rec = a.rec;
        la.n_rec = a.n_rec;
        la.W = a.W;
        la.H = a.H;
        la.tiles_x = a.tiles_x;
        la.tiles = a.tiles;
        la.bg0 = a.bg0;
        la.bg1 = a.bg1;
        la.bg2 = a.bg2;
        la.image = a.image;
        la.final_t = a.final_t;
        la.n_contrib = a.n_contrib;
        la.n_eval = a.n_eval;
        la.seg_off = a.seg_off;
        la.seg_len = a.seg_len;
        la.pre = a.pre;
        la.rowmask = reinterpret_cast<uint32_t *>(w + L.rowmask);
        la.use_list = use_list;
        la.max_segs = (uint32_t)L.max_segs;
        la.err = a.err;
        if (group > 0) return cuda_check(launch_raster_group(la, group, st), "raster group launch");
        if ((rc = cuda_check(launch_raster_list(la, st), "raster list launch"))) return rc;
        if (!band) return MS_OK;
    }
    return cuda_check(launch_after(raster_kernel, resident, kRasterThreads, kSmemBytes, st, a),
                      "raster launch");
}

extern "C" int ms_raster_ex(const ms_proj_t *proj, const ms_bins_t *bins,
                            const ms_camera_t *cam, float *image, float *final_t,
                            uint32_t *n_contrib, uint32_t *n_eval, void *ws, size_t ws_bytes,
                            int strategy, void *stream) {
    return ms_raster_ex2(proj, bins, cam, image, final_t, n_contrib, n_eval, ws, ws_bytes,
                         strategy, 0, stream);
}

extern "C" int ms_raster(const ms_proj_t *proj, const ms_bins_t *bins, const ms_camera_t *cam,
                         float *image, float *final_t, uint32_t *n_contrib, uint32_t *n_eval,
                         void *ws, size_t ws_bytes, void *stream) {
    return ms_raster_ex(proj, bins, cam, image, final_t, n_contrib, n_eval, ws, ws_bytes,
                        MS_RASTER_AUTO, stream);
}
