// Binning and depth sort (the step between "preprocess" and "rasterize" in RGBAvatar Sec. 3.2;
// the paper's renderer inherits it from 3DGS): every kept Gaussian is listed in every screen
// tile of its rectangle and each (frame, tile) list is ordered by (depth bits, Gaussian index).
//
// Design: a kernel counts the rectangles' tiles, a three-phase scan (per-CTA
// partials, one CTA over the partials, per-CTA writes; one CTA in all for few tiles) turns the counts into list offsets and a work list, a scatter
// kernel drops (depth << 32 | index) keys, with a mask of the pixel blocks each splat reaches in
// the low byte of the index word, into their tile's segment, and
// one CTA per non-empty tile sorts its list: in shared memory by one bucket pass on the top depth bits and a placement of every key by its rank in its bucket,
// or, for long segments, by the same bucket pass with the keys in L2; buckets too crowded for it
// fall back to a stable LSD radix sort of the keys compressed to (depth - segment minimum) << 32 |
// index. Because the key carries the index, the result is unique.
#include <algorithm>

#include "reach.cuh"
#include "rgba_internal.cuh"

namespace rgba {
namespace {

constexpr int kScanTile = 1024;  // tiles per CTA of the three-phase scan

// Exclusive scan over the CTA (kScanTile threads) of one (u64 value, u32 count) pair per
// thread: warp shuffles, then the 32 warp totals scanned by warp 0. Also returns the totals.
__device__ __forceinline__ void block_scan(unsigned long long v, unsigned e, unsigned long long &ex_v,
                                           unsigned &ex_e, unsigned long long &tot_v, unsigned &tot_e) {
    __shared__ unsigned long long s_v[32];
    __shared__ unsigned s_e[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long xv = v;
    unsigned xe = e;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long yv = __shfl_up_sync(0xffffffffu, xv, o);
        const unsigned ye = __shfl_up_sync(0xffffffffu, xe, o);
        if (lane >= o) {
            xv += yv;
            xe += ye;
        }
    }
    if (lane == 31) {
        s_v[warp] = xv;
        s_e[warp] = xe;
    }
    __syncthreads();
    if (warp == 0) {
        unsigned long long wv = s_v[lane];
        unsigned we = s_e[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long yv = __shfl_up_sync(0xffffffffu, wv, o);
            const unsigned ye = __shfl_up_sync(0xffffffffu, we, o);
            if (lane >= o) {
                wv += yv;
                we += ye;
            }
        }
        s_v[lane] = wv;
        s_e[lane] = we;
    }
    __syncthreads();
    ex_v = (warp ? s_v[warp - 1] : 0ull) + xv - v;
    ex_e = (warp ? s_e[warp - 1] : 0u) + xe - e;
    tot_v = s_v[31];
    tot_e = s_e[31];
    __syncthreads();  // s_v / s_e free for the next call
}

// The scan's per-CTA partials: [nb] sums, [nb] non-empty counts, [nb][32] bucket counts and
// the [32] bucket offsets, in the workspace.
struct ScanAux {
    unsigned long long *bsum;
    unsigned *bne, *bhist, *bucket;
};

__device__ __forceinline__ ScanAux scan_aux(const Ctx &c) {
    const long long nb = (c.T + kScanTile - 1) / kScanTile;
    ScanAux a;
    a.bsum = reinterpret_cast<unsigned long long *>(c.scan_aux);
    a.bne = reinterpret_cast<unsigned *>(a.bsum + nb);
    a.bhist = a.bne + nb;
    a.bucket = a.bhist + nb * 32;
    return a;
}

__device__ __forceinline__ unsigned bucket_of(unsigned v) { return 31u - __clz(v); }

// Counting and scattering take one (frame, Gaussian) per thread and give each CTA a piece of one frame. Its
// touches of tiles are counted in shared memory, one counter per tile of the frame, and each tile a CTA
// touched then costs one global atomic: 16 frames of 60,000 Gaussians make 3.3 M touches, mostly of a few
// hundred tiles, and a global atomic per touch (returning the places, in the preprocess, or counting there
// and taking the places here) made the L2's atomic units and the wait for them the bound. Projection, count,
// scan and scatter together, one atomic per touch in the projection, then this: 16 frames 148 -> 125 us, ten frames
// 112 -> 87, 64 frames of eight avatars 661 -> 535, 15 frames of five 275 -> 220, one frame 60 -> 53. Frames of more
// than kHistTiles tiles (1,773 pixels square) are taken in windows of whole tile rows, one after the other. Touch by
// touch with global atomics, then this, count, scan and scatter: one frame of 1,800 x 1,800 (N = 60,000) 128 -> 41 us,
// of 4,096 x 4,096 223 -> 143, of 2,048 x 2,048 under 2,000 splats of its size 14.2 -> 2.4 ms.
constexpr int kBinThreads = 256;
constexpr int kHistTiles = 12288;

// The CTA's frame and Gaussian. Neighbouring CTAs take different frames, so that the atomics under way
// spread over all frames' tiles.
struct BinItem {
    FrameInfo f;
    int i;
    bool valid;
};
__device__ __forceinline__ BinItem bin_item(const Ctx &c) {
    BinItem b;
    b.f = c.frames[blockIdx.x];
    b.i = (int)((blockIdx.y + blockIdx.z * gridDim.y) * kBinThreads + threadIdx.x);
    b.valid = b.i < b.f.n;
    return b;
}

// Calls f(y0, y1, tiles) for every window of the frame's tile rows, [y0, y1), whose tiles have a counter each, by the
// whole CTA. WINDOWS: some frame of the batch has more than kHistTiles tiles (a row has at most 512); of several
// windows those that no rectangle of the CTA meets are passed over, and the barrier in the vote keeps a window's
// counters from the next one's. Otherwise the only window is the frame, and its bounds are compiled out: they cost
// the scatter up to 15 registers, and 477 us instead of 448 on one frame of 1,024 x 1,024 with 64 splats of its size.
template <bool WINDOWS, typename F>
__device__ __forceinline__ void each_window(const FrameInfo &fr, const ushort4 &rc, F f) {
    const int all = fr.tiles_x * fr.tiles_y;
    if (!WINDOWS) return f(0, 0x7fffffff, all);
    const int rows = all <= kHistTiles ? fr.tiles_y : kHistTiles / fr.tiles_x;
    for (int y0 = 0; y0 < fr.tiles_y; y0 += rows) {
        const int y1 = min(fr.tiles_y, y0 + rows);
        if (rows < fr.tiles_y && !__syncthreads_or(rc.y < y1 && rc.w > y0 && rc.x < rc.z)) continue;
        f(y0, y1, (y1 - y0) * fr.tiles_x);
    }
}
static_assert(RGBA_MAX_DIM / 8 <= kHistTiles, "a window holds a row of tiles");

// Calls f(t) for the rectangle's tiles in rows [y0, y1), t counted from row y0.
template <typename F>
__device__ __forceinline__ void each_tile(const ushort4 &rc, int tiles_x, int y0, int y1, F f) {
    for (int ty = max((int)rc.y, y0); ty < min((int)rc.w, y1); ++ty)
        for (int tx = rc.x; tx < rc.z; ++tx) f((ty - y0) * tiles_x + tx);
}

template <bool WINDOWS>
__global__ void __launch_bounds__(kBinThreads) k_count(Ctx c) {
    extern __shared__ unsigned s_hist[];
    pdl_enter();
    const BinItem b = bin_item(c);
    if (b.i - (int)threadIdx.x >= b.f.n || b.i < 0) return;  // the whole CTA
    const ushort4 rc = b.valid ? c.rects[b.f.rec_base + b.i] : make_ushort4(0, 0, 0, 0);
    each_window<WINDOWS>(b.f, rc, [&](int y0, int y1, int tiles) {
        unsigned *count = c.tile_count + b.f.tile_base + y0 * b.f.tiles_x;
        for (int t = threadIdx.x; t < tiles; t += kBinThreads) s_hist[t] = 0u;
        __syncthreads();
        each_tile(rc, b.f.tiles_x, y0, y1, [&](int t) { atomicAdd(s_hist + t, 1u); });
        __syncthreads();
        for (int t = threadIdx.x; t < tiles; t += kBinThreads)
            if (s_hist[t]) atomicAdd(count + t, s_hist[t]);
    });
}

// Phase 1, one thread per tile: the tile's total count into tile_start, and per CTA the sum, the number of
// non-empty tiles and the histogram of floor(log2(length)).
__global__ void __launch_bounds__(kScanTile) k_scan_blocks(Ctx c) {
    __shared__ unsigned s_hist[32];
    pdl_enter();
    const ScanAux a = scan_aux(c);
    if (threadIdx.x < 32) s_hist[threadIdx.x] = 0;
    __syncthreads();
    const long long t = (long long)blockIdx.x * kScanTile + threadIdx.x;
    unsigned v = 0;
    if (t < c.T) {
        v = c.tile_count[t];
        c.tile_count[t] = 0u;  // the next binning of the same projection counts from zero again
        c.tile_start[t] = v;
        if (v) atomicAdd(&s_hist[bucket_of(v)], 1u);
    }
    unsigned long long ex, tot;
    unsigned exe, tote;
    block_scan(v, v > 0, ex, exe, tot, tote);
    if (threadIdx.x == 0) {
        a.bsum[blockIdx.x] = tot;
        a.bne[blockIdx.x] = tote;
    }
    if (threadIdx.x < 32) a.bhist[blockIdx.x * 32 + threadIdx.x] = s_hist[threadIdx.x];
}

// Phase 2, one CTA: exclusive scans over the CTAs of phase 1 (sums, non-empty counts, and per
// bucket the counts, warp w taking bucket w), the bucket offsets with the longest bucket first,
// the pair total, the capacity check and the work-list length.
__global__ void __launch_bounds__(kScanTile) k_scan_top(Ctx c) {
    __shared__ unsigned s_btot[32];
    pdl_enter();
    const ScanAux a = scan_aux(c);
    const long long nb = (c.T + kScanTile - 1) / kScanTile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long carry = 0;
    unsigned carry_e = 0;
    for (long long b0 = 0; b0 < nb; b0 += kScanTile) {
        const long long b = b0 + threadIdx.x;
        const unsigned long long v = b < nb ? a.bsum[b] : 0ull;
        const unsigned e = b < nb ? a.bne[b] : 0u;
        unsigned long long ex, tot;
        unsigned exe, tote;
        block_scan(v, e, ex, exe, tot, tote);
        if (b < nb) {
            a.bsum[b] = carry + ex;
            a.bne[b] = carry_e + exe;
        }
        carry += tot;
        carry_e += tote;
    }
    {
        unsigned run = 0;  // warp w: bucket w, lane = CTA within a chunk of 32
        for (long long b0 = 0; b0 < nb; b0 += 32) {
            const long long b = b0 + lane;
            const unsigned h = b < nb ? a.bhist[b * 32 + warp] : 0u;
            unsigned x = h;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (b < nb) a.bhist[b * 32 + warp] = run + x - h;
            run += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) s_btot[warp] = run;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned off = 0;
        for (int k = 31; k >= 0; --k) {
            a.bucket[k] = off;
            off += s_btot[k];
        }
        c.tile_start[c.T] = carry > 0xffffffffull ? 0xffffffffu : (unsigned)carry;
        c.cnt->pairs = carry > 0xffffffffull ? 0xffffffffu : (unsigned)carry;
        c.cnt->overflow = carry > (unsigned long long)c.cap ? 1u : 0u;
        c.cnt->n_work = carry_e;
    }
}

// Phase 3, one thread per tile: the list start (exclusive scan of the totals), also as the scatter's
// cursor, and the tile's place in the work list: non-empty tiles by bucket, longest bucket first (in any order within
// a bucket), then the empty tiles in tile order.
__global__ void __launch_bounds__(kScanTile) k_scan_write(Ctx c) {
    __shared__ unsigned s_off[32];
    pdl_enter();
    const ScanAux a = scan_aux(c);
    const long long t = (long long)blockIdx.x * kScanTile + threadIdx.x;
    const unsigned v = t < c.T ? c.tile_start[t] : 0u;
    if (threadIdx.x < 32) s_off[threadIdx.x] = a.bucket[threadIdx.x] + a.bhist[blockIdx.x * 32 + threadIdx.x];
    const bool empty = t < c.T && v == 0;
    unsigned long long ex, tot;
    unsigned exe, tote;
    block_scan(v, empty, ex, exe, tot, tote);  // its syncs also publish s_off
    if (t < c.T) {
        const unsigned long long st = a.bsum[blockIdx.x] + ex;
        c.tile_start[t] = st > 0xffffffffull ? 0xffffffffu : (unsigned)st;
        if (v) {
            c.work[atomicAdd(&s_off[bucket_of(v)], 1u)] = (unsigned)t;
            c.cursor[t] = (unsigned)st;  // meaningless past 2^32 pairs, and then unused
        } else {
            // empty tiles before this CTA: its first tile index minus the non-empty ones
            const unsigned e0 = (unsigned)((long long)blockIdx.x * kScanTile) - a.bne[blockIdx.x];
            c.work[c.cnt->n_work + e0 + exe] = (unsigned)t;
        }
    }
}

// The three phases by one CTA, kScanOne / kScanTile tiles per thread, for batches of few tiles, where the
// launches are most of the phases' time: count and scan 12.2 -> 8.8 us at 64 tiles, 13.7 -> 8.8 at 1,024, 14.1 ->
// 9.2 at 2,268. With 16 tiles per thread one CTA takes 25 us at 10,240 tiles and the phases 17.
constexpr int kScanOne = 4 * kScanTile;

__global__ void __launch_bounds__(kScanTile) k_scan_one(Ctx c) {
    constexpr int PER = kScanOne / kScanTile;
    __shared__ unsigned s_hist[32], s_off[32];
    pdl_enter();
    const int tid = threadIdx.x;
    if (tid < 32) s_hist[tid] = 0u;
    __syncthreads();
    const int t0 = tid * PER, T = (int)c.T;
    unsigned v[PER], ne = 0u;
    unsigned long long sum = 0ull;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        v[q] = 0u;
        if (t0 + q < T) {
            v[q] = c.tile_count[t0 + q];
            c.tile_count[t0 + q] = 0u;  // as k_scan_blocks
        }
        sum += v[q];
        if (v[q]) {
            ++ne;
            atomicAdd(&s_hist[bucket_of(v[q])], 1u);
        }
    }
    unsigned long long st, tot;
    unsigned exe, tote;
    block_scan(sum, ne, st, exe, tot, tote);  // its syncs also publish s_hist
    if (tid < 32) {  // bucket offsets, the longest bucket first
        const unsigned h = s_hist[31 - tid];
        unsigned x = h;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (tid >= o) x += y;
        }
        s_off[31 - tid] = x - h;
    }
    __syncthreads();
    unsigned empty = (unsigned)t0 - exe;  // empty tiles before this thread's
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        if (t0 + q >= T) break;
        const unsigned at = st > 0xffffffffull ? 0xffffffffu : (unsigned)st;
        c.tile_start[t0 + q] = at;
        if (v[q]) {
            c.cursor[t0 + q] = at;
            c.work[atomicAdd(&s_off[bucket_of(v[q])], 1u)] = (unsigned)(t0 + q);
        } else {
            c.work[tote + empty++] = (unsigned)(t0 + q);
        }
        st += v[q];
    }
    if (tid == 0) {
        c.tile_start[T] = tot > 0xffffffffull ? 0xffffffffu : (unsigned)tot;
        c.cnt->pairs = tot > 0xffffffffull ? 0xffffffffu : (unsigned)tot;
        c.cnt->overflow = tot > (unsigned long long)c.cap ? 1u : 0u;
        c.cnt->n_work = tote;
    }
}

// One thread per (frame, Gaussian): drops its key into the list of every tile of its rectangle,
// with the tile's block mask. The masks cost one ellipse extent per four pixel rows of the
// rectangle and two compares per block; computed here they are paid once per (Gaussian, tile),
// where every compositing warp of a tile (eight, forwards and again backwards) would test every
// entry of its list. TW: the tile width (16 or 8).
// In shared memory the counts of the CTA's touches become, with one global atomic per touched tile, the
// places its keys take in the lists.
template <int TW, bool WINDOWS>
__global__ void __launch_bounds__(kBinThreads) k_scatter(Ctx c) {
    extern __shared__ unsigned s_hist[];
    constexpr int TH = kTilePix / TW, NBX = TW / 8, BANDS = TH / 4;
    pdl_enter();
    if (c.cnt->overflow) return;
    const BinItem b = bin_item(c);
    if (b.i - (int)threadIdx.x >= b.f.n || b.i < 0) return;  // the whole CTA
    const FrameInfo &f = b.f;
    const long long r = f.rec_base + (b.valid ? b.i : 0);
    // every load of the record at once (few Gaussians are culled)
    ushort4 rc = c.rects[r];
    const unsigned bits = __float_as_uint(c.depth[r]);
    const float4 r0 = c.records[r * 3];
    const float2 r1 = *reinterpret_cast<const float2 *>(c.records + r * 3 + 1);
    if (!b.valid) rc = make_ushort4(0, 0, 0, 0);
    const Reach e = reach_of(r0, r1);
    each_window<WINDOWS>(f, rc, [&](int y0, int y1, int tiles) {
        unsigned *cur = c.cursor + f.tile_base + y0 * f.tiles_x;
        for (int t = threadIdx.x; t < tiles; t += kBinThreads) s_hist[t] = 0u;
        __syncthreads();
        each_tile(rc, f.tiles_x, y0, y1, [&](int t) { atomicAdd(s_hist + t, 1u); });
        __syncthreads();
        for (int t = threadIdx.x; t < tiles; t += kBinThreads)
            if (s_hist[t]) s_hist[t] = atomicAdd(cur + t, s_hist[t]);
        __syncthreads();
        if (rc.z <= rc.x) return;
        for (int ty = max((int)rc.y, y0); ty < min((int)rc.w, y1); ++ty) {
            float xl[BANDS], xr[BANDS];
#pragma unroll
            for (int k = 0; k < BANDS; ++k) reach_rows(e, (float)(ty * TH + 4 * k) + 0.5f, (float)(ty * TH + 4 * k) + 3.5f, xl[k], xr[k]);
            unsigned *place = s_hist + (ty - y0) * f.tiles_x;
            for (int tx = rc.x; tx < rc.z; ++tx) {
                unsigned mask = 0u;
#pragma unroll
                for (int k = 0; k < BANDS; ++k)
#pragma unroll
                    for (int q = 0; q < NBX; ++q) {
                        const float x0 = (float)(tx * TW + 8 * q) + 0.5f;
                        if (xr[k] >= x0 && xl[k] <= x0 + 7.0f) mask |= 1u << (k * NBX + q);
                    }
                if (e.all) mask = 0xffu;
                if (e.none) mask = 0u;
                const unsigned pos = atomicAdd(place + tx, 1u);
                c.keys[pos] = ((unsigned long long)bits << 32) | pack_low(c.masked, (unsigned)b.i, mask);
            }
        }
    });
}

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
// Shared memory of the sort: 96 KB, so that two CTAs share an SM. The bucket sort takes kSmemCap keys
// and 2^kMaxBits 2-byte bucket counts; the radix sort kSmemCap keys, their ranks and the digit counts;
// the sort of long lists 2^kStreamBits 4-byte bucket counts.
constexpr int kSmemCap = 16 * kSortThreads;
constexpr int kMaxBits = 14;
constexpr int kSortSmem = kSmemCap * 8 + (2 << kMaxBits) + 16;
static_assert(kSmemCap * (8 + 2) + kSortWarps * 256 * 4 <= kSortSmem, "radix sort fits");
constexpr int kDigitParts = kSortThreads / 256;  // threads sharing one digit's column of warp counts
static_assert(kSortThreads % 256 == 0 && 32 % kDigitParts == 0, "whole digits per warp");

// Lanes of `act` holding the same 8-bit digit as this lane: one ballot per digit bit (a warp
// multi-split), all on the full-rate vote path.
__device__ __forceinline__ unsigned digit_peers(unsigned act, unsigned d) {
    unsigned m = act;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const unsigned bit = (d >> b) & 1u;
        const unsigned v = __ballot_sync(act, bit);
        m &= bit ? v : ~v;
    }
    return m;
}

// Stable LSD radix sort of L keys on the bits [shift0, shift_end), 8-bit digits; a and b are both in
// global memory, or a is in shared memory and b unused (kInPlace, L <= kSmemCap). Warp w owns the contiguous run [w S, (w+1) S) of the
// input; within a warp, rounds of 32 keys go in order and lanes are ranked by lane index among
// equal digits (digit_peers), so the order of equal digits is kept and the result after the
// last pass is fully sorted. In place, each key's rank within its warp's run of equal digits is kept from
// the counting sweep (s_rank, L entries); the scatter sweep takes the keys into registers, all of the CTA's
// before any is written, and only adds the digit base. Otherwise it ranks again. Returns the buffer
// holding the result. A second shared-memory buffer in place of the registers holds 4,544 keys beside two CTAs
// per SM; longer crowded lists then sort in global memory: one list of 8,192 keys, 900 of them at one depth,
// 133 us, of 4,545 86, 300 lists of 6,000 172; in place 55, 35 and 70.
constexpr int kRounds = 4;  // rounds of 32 keys whose loads the radix sweeps issue together

template <bool kInPlace>
__device__ unsigned long long *radix_sort(unsigned long long *a, unsigned long long *b, int L,
                                          int shift0, int shift_end, unsigned *s_cnt /* [kSortWarps][256] */,
                                          unsigned *s_sum /* [kSortWarps] */, unsigned short *s_rank) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int S = ((L + kSortWarps - 1) / kSortWarps + 31) & ~31;
    const int lo = warp * S, hi = min(L, lo + S);
    unsigned *cnt = s_cnt + warp * 256;
    const unsigned lt_mask = (1u << lane) - 1u;
    // thread (digit d, part q) owns the counts of digit d in warps [q W/P, (q+1) W/P)
    const int d_own = threadIdx.x / kDigitParts, w_own = (threadIdx.x % kDigitParts) * (kSortWarps / kDigitParts);
    for (int shift = shift0; shift < shift_end; shift += 8) {
        for (int d = lane; d < 256; d += 32) cnt[d] = 0;
        __syncwarp();
        // rounds of 32 keys, the keys of kRounds rounds loaded at once (in global memory each
        // round would otherwise wait for its own load)
        for (int base0 = lo; base0 < hi; base0 += kRounds * 32) {
            unsigned long long kk[kRounds];
#pragma unroll
            for (int u = 0; u < kRounds; ++u) {
                const int e = base0 + 32 * u + lane;
                kk[u] = e < hi ? a[e] : 0ull;
            }
#pragma unroll
            for (int u = 0; u < kRounds; ++u) {
                const int base = base0 + 32 * u;
                if (base >= hi) break;  // warp-uniform
                const int e = base + lane;
                const bool ok = e < hi;
                const unsigned act = __ballot_sync(0xffffffffu, ok);
                unsigned d = 0, peers = 0, before = 0;
                if (ok) {
                    d = (unsigned)(kk[u] >> shift) & 255u;
                    peers = digit_peers(act, d);
                    before = cnt[d];
                    if (kInPlace) s_rank[e] = (unsigned short)(before + __popc(peers & lt_mask));
                }
                __syncwarp();
                if (ok && (peers & lt_mask) == 0) cnt[d] = before + __popc(peers);
                __syncwarp();
            }
        }
        __syncthreads();
        // the scatter base of (digit d, warp w) is the count of all (digit, warp) pairs before it
        // in digit-major order: an exclusive scan over the CTA's threads, which are ordered the
        // same way, of each thread's sum over its warps, plus the running sum within them
        {
            unsigned run = 0;
#pragma unroll
            for (int w = w_own; w < w_own + kSortWarps / kDigitParts; ++w) {
                const unsigned c = s_cnt[w * 256 + d_own];
                s_cnt[w * 256 + d_own] = run;
                run += c;
            }
            unsigned x = run;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) s_sum[warp] = x;
            __syncthreads();
            unsigned off = x - run;
#pragma unroll
            for (int q = 0; q < kSortWarps; ++q) off += q < warp ? s_sum[q] : 0u;
#pragma unroll
            for (int w = w_own; w < w_own + kSortWarps / kDigitParts; ++w) s_cnt[w * 256 + d_own] += off;
        }
        __syncthreads();
        if (kInPlace) {
            constexpr int KPT = kSmemCap / kSortThreads;
            unsigned long long k[KPT];
#pragma unroll
            for (int u = 0; u < KPT; ++u) {
                const int e = lo + 32 * u + lane;
                k[u] = e < hi ? a[e] : 0ull;
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < KPT; ++u) {
                const int e = lo + 32 * u + lane;
                if (e < hi) a[cnt[(unsigned)(k[u] >> shift) & 255u] + s_rank[e]] = k[u];
            }
            __syncthreads();
            continue;
        } else {
            for (int base0 = lo; base0 < hi; base0 += kRounds * 32) {
                unsigned long long kk[kRounds];
#pragma unroll
                for (int u = 0; u < kRounds; ++u) {
                    const int e = base0 + 32 * u + lane;
                    kk[u] = e < hi ? a[e] : 0ull;
                }
#pragma unroll
                for (int u = 0; u < kRounds; ++u) {
                    const int base = base0 + 32 * u;
                    if (base >= hi) break;  // warp-uniform
                    const int e = base + lane;
                    const bool ok = e < hi;
                    const unsigned act = __ballot_sync(0xffffffffu, ok);
                    unsigned d = 0, peers = 0, pos = 0;
                    const unsigned long long k = kk[u];
                    if (ok) {
                        d = (unsigned)(k >> shift) & 255u;
                        peers = digit_peers(act, d);
                        pos = cnt[d] + __popc(peers & lt_mask);
                    }
                    __syncwarp();
                    if (ok) {
                        b[pos] = k;
                        if ((peers & lt_mask) == 0) cnt[d] += __popc(peers);
                    }
                    __syncwarp();
                }
            }
        }
        __syncthreads();
        unsigned long long *t = a;
        a = b;
        b = t;
    }
    return a;
}

constexpr int kTieRun = 32;  // longest run of equal depths the tie pass orders by itself

constexpr int kBucketRun = 64;  // longest bucket the rank placement orders by itself

// Sort of L <= KPT kSortThreads keys at g by one bucket pass: each thread keeps its KPT keys in registers,
// a shared-memory atomic per key counts the 2^BITS buckets of the depth spread (two 16-bit counts to a
// word) and gives the key its slot in its bucket, an exclusive scan turns the counts into starts, the
// keys go to their bucket's run in s_keys (in any order inside), and every key there counts the smaller
// keys of its bucket (keys are distinct: the index differs) and writes its Gaussian index and block
// mask straight to its rank in the tile's lists `out` and `out_mask`. Per key that is one shared-memory
// write and, with about two buckets per key, two or three reads in the last step: the
// shared-memory passes over the keys are what bounds the sort of a list. Returns false, with nothing
// written, when some bucket is longer than kBucketRun.
template <int KPT, int BITS>
__device__ __forceinline__ bool bucket_sort(const unsigned long long *g, int L, unsigned long long *s_keys, unsigned *s_cnt,
                                            unsigned *s_sum /* [kSortWarps] */, unsigned *s_dmin, unsigned *s_dmax,
                                            bool masked, unsigned *__restrict__ out, unsigned char *out_mask) {
    constexpr int NW = 1 << (BITS - 1), PER = NW / kSortThreads;  // words, words per thread
    static_assert(PER % 4 == 0, "whole 16-byte groups per thread");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long k[KPT];
#pragma unroll
    for (int i = 0; i < KPT; ++i) k[i] = tid + i * kSortThreads < L ? g[tid + i * kSortThreads] : 0ull;
    uint4 *cnt4 = reinterpret_cast<uint4 *>(s_cnt);
#pragma unroll
    for (int i = 0; i < PER / 4; ++i) cnt4[tid + i * kSortThreads] = make_uint4(0u, 0u, 0u, 0u);
    unsigned dmin = 0xffffffffu, dmax = 0u;
#pragma unroll
    for (int i = 0; i < KPT; ++i)
        if (tid + i * kSortThreads < L) {
            dmin = min(dmin, (unsigned)(k[i] >> 32));
            dmax = max(dmax, (unsigned)(k[i] >> 32));
        }
    dmin = __reduce_min_sync(0xffffffffu, dmin);
    dmax = __reduce_max_sync(0xffffffffu, dmax);
    if (lane == 0) {
        atomicMin(s_dmin, dmin);
        atomicMax(s_dmax, dmax);
    }
    __syncthreads();
    const unsigned d0 = *s_dmin;
    const int bshift = max(0, 32 - __clz(*s_dmax - d0) - BITS);
    auto bucket = [&](unsigned long long key) { return ((unsigned)(key >> 32) - d0) >> bshift; };
    unsigned slot[KPT / 4], crowd = 0u;  // slots below kBucketRun, a byte each
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        unsigned s = 0u;
        if (tid + i * kSortThreads < L) {
            const unsigned b = bucket(k[i]), sh = 16u * (b & 1u);
            s = (atomicAdd(&s_cnt[b >> 1], 1u << sh) >> sh) & 0xffffu;
        }
        crowd = max(crowd, s);
        slot[i / 4] = (i & 3 ? slot[i / 4] : 0u) | s << (8 * (i & 3));
    }
    if (__syncthreads_or(crowd >= (unsigned)kBucketRun)) return false;
    {  // exclusive scan of the counts; thread t owns words [t PER, (t + 1) PER)
        unsigned w[PER], run = 0u;
#pragma unroll
        for (int i = 0; i < PER / 4; ++i) {
            const uint4 q = cnt4[tid * (PER / 4) + i];
            w[4 * i] = q.x;
            w[4 * i + 1] = q.y;
            w[4 * i + 2] = q.z;
            w[4 * i + 3] = q.w;
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const unsigned c0 = w[i] & 0xffffu, c1 = w[i] >> 16;
            w[i] = run | ((run + c0) << 16);
            run += c0 + c1;
        }
        unsigned x = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_sum[warp] = x;
        __syncthreads();
        unsigned off = x - run;
#pragma unroll
        for (int q = 0; q < kSortWarps; ++q) off += q < warp ? s_sum[q] : 0u;
        off |= off << 16;  // both halves: no start exceeds kSmemCap
#pragma unroll
        for (int i = 0; i < PER / 4; ++i)
            cnt4[tid * (PER / 4) + i] = make_uint4(w[4 * i] + off, w[4 * i + 1] + off, w[4 * i + 2] + off, w[4 * i + 3] + off);
        if (tid == 0) s_cnt[NW] = (unsigned)L;  // the last bucket's end
    }
    __syncthreads();
    const unsigned short *start = reinterpret_cast<const unsigned short *>(s_cnt);
#pragma unroll
    for (int i = 0; i < KPT; ++i)
        if (tid + i * kSortThreads < L) s_keys[start[bucket(k[i])] + ((slot[i / 4] >> (8 * (i & 3))) & 0xffu)] = k[i];
    __syncthreads();
#pragma unroll 2
    for (int p = tid; p < L; p += kSortThreads) {
        const unsigned long long key = s_keys[p];
        const unsigned b = bucket(key);
        const int lo = start[b], hi = start[b + 1];
        int rank = lo;
        for (int q = lo; q < hi; ++q) rank += s_keys[q] < key;
        out[rank] = low_index(masked, (unsigned)key);
        out_mask[rank] = low_mask(masked, (unsigned)key);
    }
    return true;
}

constexpr int kStreamBits = 14;  // buckets of the sort of long lists
constexpr int kStreamLoads = 8;  // keys per thread in flight in its sweeps
constexpr int kStreamChunk = kStreamLoads * kSortThreads - 2 * kBucketRun;  // keys ranked at a time
static_assert((4 << kStreamBits) + 8 * kStreamLoads * kSortThreads <= kSortSmem, "bucket counts and a chunk fit");

// Calls f(key) for the L keys at g, kStreamLoads of each thread's loads in flight at once.
template <typename F>
__device__ __forceinline__ void sweep(const unsigned long long *g, int L, F f) {
    for (int e0 = threadIdx.x; e0 < L; e0 += kStreamLoads * kSortThreads) {
        unsigned long long k[kStreamLoads];
#pragma unroll
        for (int u = 0; u < kStreamLoads; ++u) {
            const int e = e0 + u * kSortThreads;
            k[u] = e < L ? g[e] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kStreamLoads; ++u)
            if (e0 + u * kSortThreads < L) f(k[u]);
    }
}

// Sort of a list too long for shared memory: the same bucket pass with the keys in global memory
// (L2) and only the bucket counts in shared memory. One sweep counts the 2^kStreamBits buckets of
// the depth spread, a scan turns the counts into starts, a second sweep moves every key to its
// bucket's run in tmp (a shared-memory atomic gives the place; any order within the bucket), and a
// third ranks each key among its bucket's (a few neighbours in tmp) and writes its index and mask.
// Every sweep keeps kStreamLoads loads per thread in flight; a list of 24,000 keys takes three
// sweeps instead of the radix sort's four passes of two dependent sweeps each with a warp-wide digit
// match per key. Returns false, with nothing written, when some bucket is longer than kBucketRun.
__device__ bool bucket_sort_stream(const unsigned long long *g, unsigned long long *tmp, int L, unsigned d0, int db,
                                   unsigned *s_cnt /* [2^kStreamBits] */, unsigned *s_sum /* [kSortWarps] */,
                                   bool masked, unsigned *__restrict__ out, unsigned char *__restrict__ out_mask) {
    constexpr int NB = 1 << kStreamBits, PER = NB / kSortThreads;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int bshift = max(0, db - kStreamBits);
    auto bucket = [&](unsigned long long k) { return ((unsigned)(k >> 32) - d0) >> bshift; };
    for (int i = tid; i < NB; i += kSortThreads) s_cnt[i] = 0u;
    __syncthreads();
    sweep(g, L, [&](unsigned long long k) { atomicAdd(&s_cnt[bucket(k)], 1u); });
    __syncthreads();
    // exclusive scan of the counts; warp w owns buckets [w NB/W, (w+1) NB/W) and walks them 32 at a
    // time (neighbouring lanes, neighbouring banks)
    unsigned longest = 0u, run = 0u;
    for (int i = 0; i < PER; ++i) {
        unsigned *p = s_cnt + warp * (PER * 32) + 32 * i + lane;
        const unsigned v = *p;
        unsigned x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        *p = run + x - v;
        run += __shfl_sync(0xffffffffu, x, 31);
        longest = max(longest, v);
    }
    if (lane == 0) s_sum[warp] = run;
    if (__syncthreads_or(longest > (unsigned)kBucketRun)) return false;
    unsigned off = 0u;
    for (int w = 0; w < warp; ++w) off += s_sum[w];
    for (int i = 0; i < PER; ++i) s_cnt[warp * (PER * 32) + 32 * i + lane] += off;
    __syncthreads();
    sweep(g, L, [&](unsigned long long k) { tmp[atomicAdd(&s_cnt[bucket(k)], 1u)] = k; });
    __syncthreads();  // s_cnt[b] is now the end of bucket b; the keys at g are no longer needed
    // the grouped keys come back to shared memory a chunk at a time, with the keys around it that a bucket
    // can reach into, the next chunk's loads under way while this one's keys are ranked
    unsigned long long *s_k = reinterpret_cast<unsigned long long *>(s_cnt + NB);
    unsigned long long k[kStreamLoads];
    auto load = [&](int c0) {
        const int at = max(0, c0 - kBucketRun), n = min(L, c0 + kStreamChunk + kBucketRun) - at;
#pragma unroll
        for (int u = 0; u < kStreamLoads; ++u) k[u] = tid + u * kSortThreads < n ? tmp[at + tid + u * kSortThreads] : 0ull;
    };
    load(0);
    for (int c0 = 0; c0 < L; c0 += kStreamChunk) {
#pragma unroll
        for (int u = 0; u < kStreamLoads; ++u) s_k[tid + u * kSortThreads] = k[u];
        __syncthreads();
        if (c0 + kStreamChunk < L) load(c0 + kStreamChunk);
        const int at = max(0, c0 - kBucketRun);  // s_k[q - at] is tmp[q]
        for (int p = c0 + tid; p < min(L, c0 + kStreamChunk); p += kSortThreads) {
            const unsigned long long key = s_k[p - at];
            const unsigned b = bucket(key);
            const int lo = b ? (int)s_cnt[b - 1] : 0, hi = (int)s_cnt[b];
            int rank = lo;
            for (int q = lo; q < hi; ++q) rank += s_k[q - at] < key;
            out[rank] = low_index(masked, (unsigned)key);
            out_mask[rank] = low_mask(masked, (unsigned)key);
        }
        __syncthreads();
    }
    return true;
}

// Persistent: CTAs take (frame, tile) segments from the LPT-ordered work list. A key is
// (depth, Gaussian index), "index" standing here for the word that also holds the block mask below
// the index. A segment of up to kSmemCap keys is sorted by bucket_sort, with more keys per thread and
// more buckets the longer it is, a longer one by bucket_sort_stream with its keys in
// global memory (mostly L2). A bucket longer than kBucketRun sends a segment of up to kSmemCap keys to a
// full-key radix sort in shared memory (index bits, then depth bits), and a longer one to a radix sort in
// global memory on the depth bits only, which leaves runs of equal depth in list order; a tie pass orders
// each such run by index (insertion sort by the run's first thread), a run longer than kTieRun the full key.
// The radix sorts take keys compressed to (depth - min depth) << 32 | index.
// Bound by the shared-memory passes over the keys and, for short lists, by the load and the barriers
// between them, so two CTAs share an SM, at 64 registers with 136 bytes spilled. Keys moved between two shared-memory buffers with 2^12 buckets
// whatever the length (one CTA per SM, lists of 8,193 to 12,288 keys by positions), then this: one frame with lists
// of up to 6,321 keys 35 -> 16 us, 15 frames of five avatars 145 -> 80, 16 frames 55 -> 43, ten frames 43 -> 31,
// 64 frames of eight avatars with lists of up to 24,552 keys 268 -> 188. The same with one CTA of 1,024
// threads: 14, 68, 49, 35 and 256 us. A list of 12,289 to 24,552 keys through L2 by buckets instead of radix passes:
// 475 -> 147 us on the 15 frames.
// Thread 0 claims work items three ahead and, one stage per item, loads the claimed item's tile id and
// then its list bounds while the CTA sorts the current segment.
__global__ void __launch_bounds__(kSortThreads, 2) k_tile_sort(Ctx c) {
    extern __shared__ __align__(16) unsigned long long s_keys[];
    unsigned *s_cnt = reinterpret_cast<unsigned *>(s_keys + kSmemCap);  // bucket_sort's counts
    __shared__ unsigned s_cur, s_st, s_L, s_dmin, s_dmax, s_imax, s_long, s_sum[kSortWarps];
    pdl_enter();
    if (c.cnt->overflow) return;
    const unsigned n_work = c.cnt->n_work;
    // thread 0's pipeline: w1 / t1 the next item and its tile, w2 the item after it
    unsigned w1 = 0, t1 = 0, w2 = 0;
    if (threadIdx.x == 0) {
        // the first two items by CTA, the one with the longest list taking the shortest next
        const unsigned w0 = blockIdx.x;
        w1 = 2 * gridDim.x - 1 - w0;
        w2 = 2 * gridDim.x + atomicAdd(&c.cnt->next_sort, 1u);
        const unsigned t0 = w0 < n_work ? c.work[w0] : 0u;
        t1 = w1 < n_work ? c.work[w1] : 0u;
        s_cur = w0 < n_work ? 1u : 0u;
        s_st = w0 < n_work ? c.tile_start[t0] : 0u;
        s_L = w0 < n_work ? c.tile_start[t0 + 1] - s_st : 0u;
        s_dmin = 0xffffffffu;
        s_dmax = 0u;
        s_imax = 0u;
        s_long = 0u;
    }
    __syncthreads();
    while (s_cur) {
        const unsigned st = s_st, L = s_L;
        unsigned nst = 0, nend = 0, t2 = 0, w3 = 0;
        if (threadIdx.x == 0) {  // consumed at the end of this segment and at the next one
            if (w1 < n_work) {
                nst = c.tile_start[t1];
                nend = c.tile_start[t1 + 1];
            }
            t2 = w2 < n_work ? c.work[w2] : 0u;
            w3 = 2 * gridDim.x + atomicAdd(&c.cnt->next_sort, 1u);
        }
        const unsigned long long *g = c.keys + st;
        unsigned *out = c.sorted + st;
        unsigned char *masks = c.list_masks(st);  // over the list's keys, once nobody reads them
        const bool in_smem = L <= (unsigned)kSmemCap;
        bool done;
        if (L <= 4u * kSortThreads) {
            done = bucket_sort<4, 12>(g, (int)L, s_keys, s_cnt, s_sum, &s_dmin, &s_dmax, c.masked, out, masks);
        } else if (L <= 8u * kSortThreads) {
            done = bucket_sort<8, 13>(g, (int)L, s_keys, s_cnt, s_sum, &s_dmin, &s_dmax, c.masked, out, masks);
        } else if (in_smem) {
            done = bucket_sort<16, 14>(g, (int)L, s_keys, s_cnt, s_sum, &s_dmin, &s_dmax, c.masked, out, masks);
        } else {
            unsigned dmin = 0xffffffffu, dmax = 0u;
            sweep(g, (int)L, [&](unsigned long long k) {
                dmin = min(dmin, (unsigned)(k >> 32));
                dmax = max(dmax, (unsigned)(k >> 32));
            });
            dmin = __reduce_min_sync(0xffffffffu, dmin);
            dmax = __reduce_max_sync(0xffffffffu, dmax);
            if ((threadIdx.x & 31) == 0) {
                atomicMin(&s_dmin, dmin);
                atomicMax(&s_dmax, dmax);
            }
            __syncthreads();
            done = bucket_sort_stream(g, c.keys2 + st, (int)L, s_dmin, 32 - __clz(s_dmax - s_dmin),
                                      reinterpret_cast<unsigned *>(s_keys), s_sum, c.masked, out, masks);
        }
        if (!done) {  // a crowded bucket; the keys at g are untouched and s_dmin, s_dmax set
            unsigned imax = 0u;
            sweep(g, (int)L, [&](unsigned long long k) { imax = max(imax, (unsigned)k); });
            imax = __reduce_max_sync(0xffffffffu, imax);
            if ((threadIdx.x & 31) == 0) atomicMax(&s_imax, imax);
            const unsigned d0 = s_dmin;
            const int db = 32 - __clz(s_dmax - d0);  // bits of the depth spread
            unsigned long long *a = in_smem ? s_keys : c.keys2 + st, *bb = in_smem ? nullptr : c.keys + st;
            unsigned short *rank = reinterpret_cast<unsigned short *>(s_keys + kSmemCap);
            unsigned *cnt = reinterpret_cast<unsigned *>(rank + kSmemCap);
            const int shift0 = c.masked ? 8 : 0;  // of the index below its mask
            for (unsigned e = threadIdx.x; e < L; e += blockDim.x) {
                const unsigned long long k = g[e];
                a[e] = ((unsigned long long)((unsigned)(k >> 32) - d0) << 32) | (unsigned)k;
            }
            __syncthreads();
            const int ib = 32 - __clz(s_imax);  // bits of the largest index (0 if 0)
            unsigned long long *res;
            if (in_smem) {
                res = radix_sort<true>(a, bb, (int)L, shift0, ib, cnt, s_sum, rank);
                res = radix_sort<true>(a, bb, (int)L, 32, 32 + db, cnt, s_sum, rank);
            } else {
                res = radix_sort<false>(a, bb, (int)L, 32, 32 + db, cnt, s_sum, nullptr);
                // ties: a run keeps its depth under any reordering, so run starts found by other
                // threads do not change while a run is being ordered
                for (unsigned e = threadIdx.x; e + 1 < L; e += blockDim.x) {
                    const unsigned dep = (unsigned)(res[e] >> 32);
                    if ((unsigned)(res[e + 1] >> 32) != dep || (e > 0 && (unsigned)(res[e - 1] >> 32) == dep))
                        continue;
                    unsigned end = e + 2;
                    while (end < L && end - e <= (unsigned)kTieRun && (unsigned)(res[end] >> 32) == dep) ++end;
                    if (end - e > (unsigned)kTieRun) {
                        s_long = 1u;
                        continue;
                    }
                    for (unsigned i = e + 1; i < end; ++i) {
                        const unsigned long long k = res[i];
                        unsigned j = i;
                        for (; j > e && res[j - 1] > k; --j) res[j] = res[j - 1];
                        res[j] = k;
                    }
                }
                __syncthreads();
                if (s_long) {
                    unsigned long long *other = res == a ? bb : a;
                    res = radix_sort<false>(res, other, (int)L, shift0, ib, cnt, s_sum, nullptr);
                    other = res == a ? bb : a;
                    res = radix_sort<false>(res, other, (int)L, 32, 32 + db, cnt, s_sum, nullptr);
                }
            }
            if (res == g) {  // the masks go over this buffer: finish from the other one
                for (unsigned e = threadIdx.x; e < L; e += blockDim.x) a[e] = res[e];
                __syncthreads();
                res = a;
            }
            for (unsigned e = threadIdx.x; e < L; e += blockDim.x) {
                const unsigned low = (unsigned)res[e];
                out[e] = low_index(c.masked, low);
                masks[e] = low_mask(c.masked, low);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            s_cur = w1 < n_work ? 1u : 0u;
            s_st = nst;
            s_L = nend - nst;
            w1 = w2;
            t1 = t2;
            w2 = w3;
            s_dmin = 0xffffffffu;
            s_dmax = 0u;
            s_imax = 0u;
            s_long = 0u;
        }
        __syncthreads();
    }
    // the last CTA out puts the work counter back to zero for the next launch
    if (threadIdx.x == 0 && atomicAdd(&c.cnt->done_sort, 1u) == gridDim.x - 1) {
        c.cnt->next_sort = 0u;
        c.cnt->done_sort = 0u;
    }
}

}  // namespace

cudaError_t launch_scan(const Ctx &c, cudaStream_t s) {
    if (c.T <= kScanOne) return launch_pdl(k_scan_one, dim3(1), dim3(kScanTile), 0, s, c);
    const unsigned nb = (unsigned)((c.T + kScanTile - 1) / kScanTile);
    cudaError_t e = launch_pdl(k_scan_blocks, dim3(nb), dim3(kScanTile), 0, s, c);
    if (e != cudaSuccess) return e;
    if ((e = launch_pdl(k_scan_top, dim3(1), dim3(kScanTile), 0, s, c)) != cudaSuccess) return e;
    return launch_pdl(k_scan_write, dim3(nb), dim3(kScanTile), 0, s, c);
}

int scan_kernels(long long T) { return T <= kScanOne ? 1 : 3; }

size_t scan_aux_bytes(long long T) {
    const long long nb = (T + kScanTile - 1) / kScanTile;
    return (size_t)nb * 8 + (size_t)nb * 4 + (size_t)nb * 32 * 4 + 32 * 4;
}

namespace {
dim3 bin_grid(const Ctx &c, int max_n) {
    const unsigned chunks = (unsigned)(max_n - 1) / kBinThreads + 1, z = (chunks - 1) / 65535u + 1;
    return dim3((unsigned)c.B, (chunks - 1) / z + 1, z);
}
size_t bin_smem(int max_tiles) { return 4 * (size_t)std::min(max_tiles, kHistTiles); }
}  // namespace

cudaError_t launch_count(const Ctx &c, int max_n, int max_tiles, cudaStream_t s) {
    if (c.B == 0 || max_n == 0) return cudaSuccess;
    return launch_pdl(max_tiles > kHistTiles ? k_count<true> : k_count<false>, bin_grid(c, max_n), dim3(kBinThreads), bin_smem(max_tiles), s, c);
}

cudaError_t launch_scatter(const Ctx &c, int max_n, int max_tiles, cudaStream_t s) {
    if (c.B == 0 || max_n == 0) return cudaSuccess;
    const bool w = max_tiles > kHistTiles;
    return launch_pdl(c.tw == 16 ? (w ? k_scatter<16, true> : k_scatter<16, false>) : (w ? k_scatter<8, true> : k_scatter<8, false>),
                      bin_grid(c, max_n), dim3(kBinThreads), bin_smem(max_tiles), s, c);
}

cudaError_t launch_tile_sort(const Ctx &c, int sms, cudaStream_t s) {
    static int attr_device = -1, per_sm = 1;
    const int smem = kSortSmem;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (attr_device != dev) {
        e = cudaFuncSetAttribute(k_tile_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tile_sort, kSortThreads, smem);
        if (e != cudaSuccess) return e;
        per_sm = per_sm < 1 ? 1 : per_sm;
        attr_device = dev;
    }
    return launch_pdl(k_tile_sort, dim3(sms * per_sm), dim3(kSortThreads), (size_t)smem, s, c);
}

}  // namespace rgba
