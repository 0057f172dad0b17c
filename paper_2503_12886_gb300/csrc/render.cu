// Front-to-back alpha compositing ("rasterize", RGBAvatar Sec. 3.2 on the 3DGS renderer) and
// its exact reverse. The binning tile (16x16 or 8x32 pixels) fixes the lists; the compositing
// work is split finer: every warp is an independent persistent worker that takes (tile, pixel
// block) items from one counter, so the few heavy tiles of a face-centred frame spread over
// many warps and no warp ever waits at a CTA barrier. A block is 8 x 4 pixels, one per lane.
//
// Every list entry comes with a byte that says which of the tile's eight blocks its splat can
// reach (made once per (Gaussian, tile) by the scatter). A warp scans its tile's list 128 entries
// at a time, four mask bytes per lane, and queues the positions whose bit for its block is set. It
// stages 32 S of the queued entries at a time: each lane loads the records of S of them (one step
// ahead of the compositing, the Gaussian indices two), tests which half of the block (4 x 4 pixels) the splat
// reaches and writes the entry, in the form the pixel loop reads, to the shared-memory slots of those
// halves. The two halves of the warp then walk their own slots side by side, in list order (in
// reverse in the backward): on 16 frames of 512 x 512 (N = 60,000) a quarter of the splats that meet a
// block miss one of its halves, which leaves 9 % fewer steps after the fuller half of each stage. The
// pixel step has no branches (lanes that do not take part keep their state; skipping an entry that no
// pixel takes saved less than the vote and the broken-up schedule cost), so that several entries' steps
// overlap, and the power is evaluated for two entries at a time in packed FP32. The forward
// stops once every pixel of the block is saturated.
//
// Per pixel, with d = pixel centre - mean:
//   power = -(a dx^2 + c dy^2) / 2 - b dx dy  (skip if > 0)
//   alpha = min(0.99, o exp(power))            (skip if < 1/255)
//   stop, without blending, once T (1 - alpha) < 1e-4
// The backward recomputes each alpha with the same instruction sequence as the forward, walks
// the list backwards from the stored contributor count, and recovers T by division by
// (1 - alpha). Per-Gaussian gradient sums are formed 16 entries at a time with the warp turned
// round: lanes hold entries instead of pixels and add up their rows of a shared-memory matrix
// that the visits filled; the sums reach global memory as atomic reductions.
#include "reach.cuh"
#include "rgba_internal.cuh"

namespace rgba {
namespace {

constexpr float kAlphaMax = 0.99f;
constexpr float kTMin = 1e-4f;

__device__ __forceinline__ int find_frame(const Ctx &c, long long t) {
    int lo = 0, hi = c.B - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (c.frames[mid].tile_base <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// power = -(a dx^2 + c dy^2)/2 - b dx dy = dx ((-a/2) dx + (-b) dy) + (-c/2) dy dy for a pair of staged
// entries: A = (-u, -v), B = (-a/2, -b), hc = -c/2, one entry in each component. Both kernels evaluate
// through this function and cut with skip(), so their decisions agree bit for bit.
__device__ __forceinline__ float2 power_of(float pxc, float pyc, const float4 &A, const float4 &B, float2 hc) {
    const float2 dx = __fadd2_rn(make_float2(pxc, pxc), make_float2(A.x, A.y));
    const float2 dy = __fadd2_rn(make_float2(pyc, pyc), make_float2(A.z, A.w));
    const float2 t = __ffma2_rn(make_float2(B.x, B.y), dx, __fmul2_rn(make_float2(B.z, B.w), dy));
    return __ffma2_rn(dx, t, __fmul2_rn(__fmul2_rn(hc, dy), dy));
}

// the skip decision: a positive power (never, for a positive definite conic, but kept as the
// definition) or alpha below 1/255 (alpha_cut): most pairs, the far tail of a splat, are rejected
// before the exponential and before the colour is read
__device__ __forceinline__ bool skip(float power, float tau) { return power > 0.0f || power < tau; }

// e^x for the compositing, as 2^(x log2 e) on the hardware's base-2 exponential in its
// flush-to-zero form: no weight that counts (alpha >= 1/255) is near the subnormal range.
__device__ __forceinline__ float exp_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__fmul_rn(x, 1.44269504088896341f)));
    return y;
}

struct PixF {
    float pxc, pyc, T, C0, C1, C2;
    int last;
    bool inside, done;
};

// One list entry for one pixel (forward), once the caller has evaluated the entry's power at
// the pixel: live = the pixel is still compositing and the entry passes the alpha cutoff. A live
// entry that would take T (1 - alpha) below 1e-4 marks the pixel done without blending;
// otherwise it blends. Branch-free, so a warp whose lanes disagree runs it once: a lane that is
// not live keeps its state whatever its exponential gives. The colour is added under the same
// condition and not with a weight of 0, which would carry an infinite or undefined colour to
// every pixel the entry was staged for. Returns the splatting weight alpha T at the pixel (0 when the
// entry does not blend).
__device__ __forceinline__ float composite(PixF &p, bool live, float power, const float4 &Cc, int pos) {
    const float alpha = fminf(kAlphaMax, __fmul_rn(Cc.x, exp_ftz(power)));
    const float testT = p.T * (1.0f - alpha);
    const bool sat = testT < kTMin;
    p.done = p.done || (live && sat);
    const bool blend = live && !sat;
    const float w = alpha * p.T;
    // predicated instructions: selects of the results cost the walks of few blocks 1 to 4 %
    asm("{\n\t.reg .pred q;\n\t"
        "setp.ne.s32 q, %5, 0;\n\t"
        "@q fma.rn.f32 %0, %6, %9, %0;\n\t"
        "@q fma.rn.f32 %1, %7, %9, %1;\n\t"
        "@q fma.rn.f32 %2, %8, %9, %2;\n\t"
        "@q mov.f32 %3, %10;\n\t"
        "@q mov.s32 %4, %11;\n\t}"
        : "+f"(p.C0), "+f"(p.C1), "+f"(p.C2), "+f"(p.T), "+r"(p.last)
        : "r"((int)blend), "f"(Cc.y), "f"(Cc.z), "f"(Cc.w), "f"(w), "f"(testT), "r"(pos));
    return blend ? w : 0.0f;
}

constexpr int kWarpsPerCta = 4;  // independent warps per CTA (they share nothing but the loss sum)

// Two staged entries, slots 2 p and 2 p + 1, as the pixel loop reads them:
//   A = (-u, -u', -v, -v')  B = (-a/2, -a'/2, -b, -b')  H = (-c/2, -c'/2, tau, tau')
//   c = (opacity, r, g, b)  pos = list position + 1   idx = Gaussian index
struct __align__(16) Pair {
    float4 A, B, H, c[2];
    int pos[2];
    unsigned idx[2];
};

// A warp's shared memory: the queue of list positions that reach its block, and for each half of
// the block its staged slots, up to 32 S (the loop looks one pair ahead, past the end at whatever follows). The
// halves lie 64 bytes apart modulo the banks' 128, so that both halves' reads are one pass.
template <int S>
struct WarpMem {
    static constexpr int kQueue = 256;  // holds a stage's worth and one scan
    static_assert(32 * S - 1 + 128 <= kQueue, "queue");
    static constexpr int kHalf = 16 * S * (int)sizeof(Pair) + 64, kSlots = kHalf + 16 * S * (int)sizeof(Pair);
    __align__(16) unsigned char mem[kSlots + 4 * kQueue];  // the halves' slots, then the queue
    __device__ __forceinline__ Pair *half(int h) { return reinterpret_cast<Pair *>(mem + h * kHalf); }
    __device__ __forceinline__ const Pair *half(int h) const { return reinterpret_cast<const Pair *>(mem + h * kHalf); }
    __device__ __forceinline__ unsigned &queue(unsigned i) { return reinterpret_cast<unsigned *>(mem + kSlots)[i & (kQueue - 1)]; }
    __device__ __forceinline__ unsigned queue(unsigned i) const { return reinterpret_cast<const unsigned *>(mem + kSlots)[i & (kQueue - 1)]; }
};

// One compositing warp's view of a (tile, pixel block) item: the tile's list and the block.
struct Walk {
    const unsigned *list;        // the tile's sorted Gaussian indices
    const unsigned char *masks;  // and their block masks (8-byte aligned)
    int len;
    unsigned blk;
    const float4 *rec;  // the frame's render records
    float bx0, by0;     // the block's first pixel centre
    bool masked;        // the lists carry masks
};

// The entries of list positions [0, hi) that reach the block, front to back (DIR = 1) or back to
// front (DIR = -1). A chunk is 128 list positions, four neighbouring ones per lane (their mask bytes
// are one word); fill() appends a chunk's hits to the queue in walking order, with the words of the two
// chunks after it in flight.
template <int S, int DIR>
struct Feed {
    int hi, next, left;   // entries; the next chunk to load; chunks not scanned yet
    unsigned head, count; // the queue's first element and length
    unsigned w0, w1;      // this lane's mask bytes of the next two chunks, as loaded: a warp waits for a
                          // load at the first instruction that reads it, so nothing does before the scan

    // this lane's first list position of chunk k
    static __device__ __forceinline__ int first(int k) {
        const int lane = threadIdx.x & 31;
        return k * 128 + 4 * (DIR > 0 ? lane : 31 - lane);
    }
    __device__ __forceinline__ unsigned load(const Walk &w) {
        const int e = first(next);
        next += DIR;
        unsigned m = 0u;  // bytes past the list's end lie in its own key segment
        if (e >= 0 && e < hi) m = *reinterpret_cast<const unsigned *>(w.masks + e);
        return m;
    }
    __device__ __forceinline__ void start(const Walk &w, int hi_) {
        hi = hi_;
        left = (hi + 127) / 128;
        next = DIR > 0 ? 0 : left - 1;
        head = count = 0u;
        w0 = load(w);
        w1 = load(w);
    }
    // until the queue holds a stage's worth (or the list is done); returns the entries scanned
    __device__ __forceinline__ int fill(const Walk &w, WarpMem<S> &m) {
        const int lane = threadIdx.x & 31;
        const unsigned lt = (1u << lane) - 1u;
        int scanned = 0;
        while (count < 32u * S && left > 0) {
            const int e = first(next - 2 * DIR);
            unsigned hits = (w0 >> w.blk) & 0x01010101u;  // bit 8 i: byte i
            if (hi - e < 4) hits = hi > e ? hits & ((1u << (8 * (hi - e))) - 1u) : 0u;
            const unsigned n = __popc(hits);
            const unsigned b0 = __ballot_sync(0xffffffffu, n & 1u), b1 = __ballot_sync(0xffffffffu, n & 2u),
                           b2 = __ballot_sync(0xffffffffu, n & 4u);
            unsigned at = head + count + __popc(b0 & lt) + 2u * __popc(b1 & lt) + 4u * __popc(b2 & lt);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = DIR > 0 ? i : 3 - i;
                if ((hits >> (8 * k)) & 1u) m.queue(at++) = (unsigned)(e + k + 1);
            }
            count += __popc(b0) + 2u * __popc(b1) + 4u * __popc(b2);
            --left;
            scanned += min(128, hi - (next - 2 * DIR) * 128);
            w0 = w1;
            w1 = load(w);
        }
        __syncwarp();
        return scanned;
    }
};

// Up to 32 S queued entries on their way to the slots: lane l takes entries l, l + 32, ... First
// their list positions and Gaussian indices, a step later their records.
template <int S>
struct Ids {
    unsigned pos[S], idx[S];
    int n;  // entries
};
template <int S>
struct Stage {
    Ids<S> id;
    float4 r0[S], r1[S];
    float r2[S];
};

template <int S, int DIR>
__device__ __forceinline__ void load_ids(const Walk &w, const WarpMem<S> &m, Feed<S, DIR> &f, Ids<S> &d) {
    const int lane = threadIdx.x & 31;
    d.n = min((int)f.count, 32 * S);
#pragma unroll
    for (int s = 0; s < S; ++s) {
        if (lane + 32 * s < d.n) {
            d.pos[s] = m.queue(f.head + lane + 32 * s);
            d.idx[s] = w.list[d.pos[s] - 1u];
        }
    }
    f.head += d.n;
    f.count -= d.n;
}

template <int S>
__device__ __forceinline__ void load_stage(const Walk &w, const Ids<S> &d, Stage<S> &g) {
    const int lane = threadIdx.x & 31;
    g.id = d;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        if (lane + 32 * s < d.n) {
            const float4 *r = w.rec + (size_t)d.idx[s] * 3;
            g.r0[s] = r[0];
            g.r1[s] = r[1];
            g.r2[s] = r[2].x;
        }
    }
}

// Writes one entry to slot k of half h.
template <int S>
__device__ __forceinline__ void put_slot(WarpMem<S> &m, int h, int k, const float4 &r0, const float4 &r1, float r2, float tau,
                                         unsigned pos, unsigned idx) {
    Pair &s = m.half(h)[k >> 1];
    const int i = k & 1;
    float *A = reinterpret_cast<float *>(&s.A) + i, *B = reinterpret_cast<float *>(&s.B) + i, *H = reinterpret_cast<float *>(&s.H) + i;
    A[0] = -r0.x;
    A[2] = -r0.y;
    B[0] = -0.5f * r0.z;
    B[2] = -r0.w;
    H[0] = -0.5f * r1.x;
    H[2] = tau;
    s.c[i] = make_float4(r1.y, r1.z, r1.w, r2);
    s.pos[i] = (int)pos;
    s.idx[i] = idx;
}

// The bounding box, in pixel centres, of the pixels of half h that `live` (one bit per lane) holds.
struct LiveBox {
    float x0, x1, y0, y1;
    bool any;
};
__device__ __forceinline__ LiveBox live_box(const Walk &w, unsigned live, int h) {
    const unsigned m = (live >> (16 * h)) & 0xffffu;
    unsigned col = m | m >> 8;
    col = (col | col >> 4) & 15u;
    LiveBox b;
    b.any = m != 0u;
    b.x0 = w.bx0 + (float)(4 * h + __ffs((int)col) - 1);
    b.x1 = w.bx0 + (float)(4 * h + 31 - __clz((int)col));
    b.y0 = w.by0 + (float)((__ffs((int)m) - 1) >> 2);
    b.y1 = w.by0 + (float)((31 - __clz((int)m)) >> 2);
    return b;
}

// The staged entries into the slots of the halves whose live pixels they can reach (live: one bit per lane for
// the pixels that can still take one of them), in order; n[h] of half h. Where a block is nearly saturated,
// or in the backward nearly not reached yet, most of the entries that its mask lets through only touch pixels
// that are out of the walk: on one 64 x 64 frame of 100,000 Gaussians, where the silhouette's blocks walk lists of
// 59,000 entries, the forward takes 852 us with this cut and 1,372 without. On 16
// frames of 512 x 512 it saves 6 us of 121 forwards and 11 of 152 backwards, on 15 frames of five avatars 12 of 160. A half with
// fewer is filled up, to an even number, with entries that no pixel takes. Returns the slots to walk;
// reach[h]: the lanes whose (last) entry reaches half h.
template <int S>
__device__ __forceinline__ int commit(const Walk &w, const Stage<S> &g, WarpMem<S> &m, unsigned live, int n[2],
                                      unsigned reach[2]) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const LiveBox bl = live_box(w, live, 0), br = live_box(w, live, 1);
    __syncwarp();  // the previous stage's slots are no longer read
    n[0] = n[1] = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        bool left = false, right = false;
        float tau = 0.f;
        if (lane + 32 * s < g.id.n) {
            const Reach e = reach_of(g.r0[s], make_float2(g.r1[s].x, g.r1[s].y));
            float xl, xr;
            tau = alpha_cut(g.r1[s].y);
            const bool all = e.all || !w.masked;  // lists without masks are not cut, but for what reaches no pixel
            reach_rows(e, bl.y0, bl.y1, xl, xr);
            left = bl.any && !e.none && (all || (xr >= bl.x0 && xl <= bl.x1));
            reach_rows(e, br.y0, br.y1, xl, xr);
            right = br.any && !e.none && (all || (xr >= br.x0 && xl <= br.x1));
        }
        const unsigned ml = __ballot_sync(0xffffffffu, left), mr = __ballot_sync(0xffffffffu, right);
        if (left) put_slot(m, 0, n[0] + __popc(ml & lt), g.r0[s], g.r1[s], g.r2[s], tau, g.id.pos[s], g.id.idx[s]);
        if (right) put_slot(m, 1, n[1] + __popc(mr & lt), g.r0[s], g.r1[s], g.r2[s], tau, g.id.pos[s], g.id.idx[s]);
        n[0] += __popc(ml);
        n[1] += __popc(mr);
        reach[0] = ml;
        reach[1] = mr;
    }
    const int top = (max(n[0], n[1]) + 1) & ~1;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int h = 0; h < 2; ++h)
        for (int k = n[h] + lane; k < top; k += 32) put_slot(m, h, k, z, z, 0.f, __int_as_float(0x7f800000), 0u, 0u);
    __syncwarp();
    return top;
}

// A fire-and-forget global float add.
__device__ __forceinline__ void red_add(float *addr, float v) {
    asm volatile("red.global.add.f32 [%0], %1;" :: "l"(addr), "f"(v) : "memory");
}

// Adds 4 floats at a 16-byte aligned address of global memory.
__device__ __forceinline__ void red_add4(float *addr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" :: "l"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// Sums over pixels for 16 slots at a time. The step of slot j leaves one or two numbers per pixel
// (lane) in row j % 16 of a shared-memory matrix; after 16 slots the warp turns round: lane l takes
// slot l % 16 of half l / 16 and adds up that half's 16 pixels (the columns 16 (l / 16) ...) from 16-byte
// loads, one pixel row at a time, two pixels per packed FP32 instruction. Per slot that costs
// the stores and a sixteenth of about 150 instructions, where a shuffle reduction of nine sums
// over the lanes takes about 45 and puts ten dependent shuffles into every step. The rows are
// padded to 36 floats so that the 16-byte loads of eight lanes fall in different banks.
constexpr int kRows = 16;
constexpr int kRowStride = 36;

// The four values of pixel row q of this lane's slot and half, as pairs of neighbouring columns.
__device__ __forceinline__ void row_pairs(const float *rows, int q, float2 v[2]) {
    const int lane = threadIdx.x & 31;
    const float4 a = *reinterpret_cast<const float4 *>(rows + (lane & 15) * kRowStride + (lane & 16) + 4 * q);
    v[0] = make_float2(a.x, a.y);
    v[1] = make_float2(a.z, a.w);
}

// c += sum over the pairs of w times the pixels' values `pix` [32] (pixel row q of this lane's half)
__device__ __forceinline__ void add_dot(float2 &c, const float2 w[2], const float *pix, int q) {
    const float4 a = *reinterpret_cast<const float4 *>(pix + (threadIdx.x & 16) + 4 * q);
    c = __ffma2_rn(w[0], make_float2(a.x, a.y), c);
    c = __ffma2_rn(w[1], make_float2(a.z, a.w), c);
}

// Writes one finished pixel (colour over the background, T, contributor count) and, with a
// target, adds its loss term and returns dL/dpixel in g (also stored to dl_dimg unless that is
// NULL: the fused training-step kernel keeps it in registers).
__device__ __forceinline__ void finish_pixel(const Ctx &c, const FrameInfo &f, int b, int px, int py,
                                             const PixF &p, float *img, float *T_final, int *n_contrib,
                                             const float *target, int loss_kind, float *dl_dimg,
                                             float &loss_acc, float g[3]) {
    const float *bg = c.fparams + (size_t)b * RGBA_FP_STRIDE + 17;
    const long long hw = (long long)f.W * f.H;
    const long long pix = (long long)py * f.W + px;
    float *im = img + f.pix_base * 3 + pix;
    const float o0 = fmaf(p.T, bg[0], p.C0), o1 = fmaf(p.T, bg[1], p.C1), o2 = fmaf(p.T, bg[2], p.C2);
    im[0] = o0;
    im[hw] = o1;
    im[2 * hw] = o2;
    T_final[f.pix_base + pix] = p.T;
    n_contrib[f.pix_base + pix] = p.last;
    g[0] = g[1] = g[2] = 0.0f;
    if (target) {
        const float *tg = target + f.pix_base * 3 + pix;
        const float scale = 1.0f / (3.0f * (float)hw * (float)c.loss_frames);
        const float d0 = o0 - tg[0], d1 = o1 - tg[hw], d2 = o2 - tg[2 * hw];
        if (loss_kind == RGBA_LOSS_L1) {
            loss_acc += (fabsf(d0) + fabsf(d1) + fabsf(d2)) * scale;
            g[0] = d0 > 0.f ? scale : (d0 < 0.f ? -scale : 0.f);
            g[1] = d1 > 0.f ? scale : (d1 < 0.f ? -scale : 0.f);
            g[2] = d2 > 0.f ? scale : (d2 < 0.f ? -scale : 0.f);
        } else {
            loss_acc += 0.5f * (d0 * d0 + d1 * d1 + d2 * d2) * scale;
            g[0] = d0 * scale;
            g[1] = d1 * scale;
            g[2] = d2 * scale;
        }
        if (dl_dimg) {
            float *dl = dl_dimg + f.pix_base * 3 + pix;
            dl[0] = g[0];
            dl[hw] = g[1];
            dl[2 * hw] = g[2];
        }
    }
}

// An empty tile's item: the background, T = 1, no contributors, eight pixels per lane; four
// neighbouring ones at a time where the frame's rows and the arrays allow 16-byte accesses (vec).
template <int TW>
__device__ __forceinline__ void empty_tile(const Ctx &c, long long t, bool vec, float *img, float *T_final, int *n_contrib,
                                           const float *target, int loss_kind, float *dl_dimg, float &loss_acc) {
    constexpr int TH = kTilePix / TW;
    const int lane = threadIdx.x & 31;
    const int b = find_frame(c, t);
    const FrameInfo &f = c.frames[b];
    const int lt = (int)(t - f.tile_base);
    const int ty = lt / f.tiles_x, tx = lt - ty * f.tiles_x;
    if (vec && ((f.W | f.pix_base) & 3) == 0) {
        const float *bg = c.fparams + (size_t)b * RGBA_FP_STRIDE + 17;
        const long long hw = (long long)f.W * f.H;
        const float scale = 1.0f / (3.0f * (float)hw * (float)c.loss_frames);
#pragma unroll
        for (int k = 0; k < kTilePix / 128; ++k) {
            const int p4 = 4 * lane + 128 * k, px = tx * TW + (p4 % TW), py = ty * TH + (p4 / TW);
            if (px >= f.W || py >= f.H) continue;
            const long long pix = (long long)py * f.W + px;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                const long long at = f.pix_base * 3 + ch * hw + pix;
                const float o = fmaf(1.f, bg[ch], 0.f);
                *reinterpret_cast<float4 *>(img + at) = make_float4(o, o, o, o);
                if (target) {
                    const float4 tg = *reinterpret_cast<const float4 *>(target + at);
                    float g[4];
                    const float dd[4] = {o - tg.x, o - tg.y, o - tg.z, o - tg.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const bool l1 = loss_kind == RGBA_LOSS_L1;
                        loss_acc += (l1 ? fabsf(dd[q]) : 0.5f * (dd[q] * dd[q])) * scale;
                        g[q] = l1 ? (dd[q] > 0.f ? scale : (dd[q] < 0.f ? -scale : 0.f)) : dd[q] * scale;
                    }
                    if (dl_dimg) *reinterpret_cast<float4 *>(dl_dimg + at) = make_float4(g[0], g[1], g[2], g[3]);
                }
            }
            *reinterpret_cast<float4 *>(T_final + f.pix_base + pix) = make_float4(1.f, 1.f, 1.f, 1.f);
            *reinterpret_cast<int4 *>(n_contrib + f.pix_base + pix) = make_int4(0, 0, 0, 0);
        }
        return;
    }
#pragma unroll 1
    for (int k = lane; k < kTilePix; k += 32) {
        const int px = tx * TW + (k % TW), py = ty * TH + (k / TW);
        if (px < f.W && py < f.H) {
            const PixF p{(float)px + 0.5f, (float)py + 0.5f, 1.f, 0.f, 0.f, 0.f, 0, true, true};
            float g[3];
            finish_pixel(c, f, b, px, py, p, img, T_final, n_contrib, target, loss_kind, dl_dimg, loss_acc, g);
        }
    }
}

// Compositing statistics of one warp (counting instances only, S = 1): list entries scanned, entries
// that reach the block by their mask, visits that some pixel of the block takes (past the cutoffs;
// warp-uniform), and the (pixel, entry) pairs that blend or take a gradient (this lane's). taken: the
// stage's slots of each half that some pixel took.
struct WalkStats {
    unsigned long long staged, hits, visits;
    unsigned lanes, taken[2];
    // slots j and j + 1 of the stage: whether this lane's pixel takes them
    __device__ __forceinline__ void step(int j, bool a, bool b) {
        const unsigned va = __ballot_sync(0xffffffffu, a), vb = __ballot_sync(0xffffffffu, b);
        taken[0] |= ((va & 0xffffu) ? 1u << j : 0u) | ((vb & 0xffffu) ? 2u << j : 0u);
        taken[1] |= ((va >> 16) ? 1u << j : 0u) | ((vb >> 16) ? 2u << j : 0u);
        lanes += (a ? 1u : 0u) + (b ? 1u : 0u);
    }
    // the stage's end; reach: the lanes whose staged entry went to each half's slots
    __device__ __forceinline__ void stage(const unsigned reach[2]) {
        const int lane = threadIdx.x & 31;
        const unsigned lt = (1u << lane) - 1u;
        bool v = false;
        for (int h = 0; h < 2; ++h) v = v || (((reach[h] >> lane) & 1u) && ((taken[h] >> __popc(reach[h] & lt)) & 1u));
        visits += __popc(__ballot_sync(0xffffffffu, v));
        taken[0] = taken[1] = 0u;
    }
};

// Shared memory of the colour initialisation's sums: the visits' weights and the block's target.
struct __align__(16) AccMem {
    float w[kRows * kRowStride];
    float target[3 * 32];
};

// Adds the weights w and w times the target colour of the entries in slots slot0 ... slot0 + 15 of each half
// (n[h] slots in all) to their records' first four accumulators in acc.
template <int S>
__device__ __forceinline__ void flush_acc(const AccMem &r, const WarpMem<S> &m, int slot0, const int n[2], float *acc) {
    const int lane = threadIdx.x & 31, h = lane >> 4, slot = slot0 + (lane & 15);
    __syncwarp();
    float2 s = make_float2(0.f, 0.f), c0 = s, c1 = s, c2 = s;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float2 v[2];
        row_pairs(r.w, q, v);
        s = __fadd2_rn(s, __fadd2_rn(v[0], v[1]));
        add_dot(c0, v, r.target, q);
        add_dot(c1, v, r.target + 32, q);
        add_dot(c2, v, r.target + 64, q);
    }
    const float t = s.x + s.y;
    if (slot < (h ? n[1] : n[0]) && t > 0.f)  // else no pixel took the entry
        red_add4(acc + (size_t)m.half(h)[slot >> 1].idx[slot & 1] * kG2Floats, t, c0.x + c0.y, c1.x + c1.y, c2.x + c2.y);
    __syncwarp();
}

// The forward walk of one pixel block, until every pixel of the block is done or the list ends.
// ACC: colour-initialisation accumulation into acc (see k_render_fwd).
template <int S, bool ACC, bool STATS>
__device__ __forceinline__ void fwd_walk(const Walk &w, WarpMem<S> &m, PixF &p, AccMem *am, float *acc, WalkStats &st) {
    const int lane = threadIdx.x & 31, h = lane >> 4;
    Feed<S, 1> f;
    Ids<S> d;
    Stage<S> g;
    f.start(w, w.len);
    int scanned = f.fill(w, m);
    load_ids<S>(w, m, f, d);
    scanned += f.fill(w, m);
    load_stage<S>(w, d, g);
    load_ids<S>(w, m, f, d);
    while (g.id.n) {
        if (STATS) st.staged += scanned;
        const unsigned live = __ballot_sync(0xffffffffu, !p.done);
        if (!live) break;
        int n[2];
        unsigned reach[2];
        if (STATS) st.hits += g.id.n;
        const int top = commit<S>(w, g, m, live, n, reach);
        scanned = f.fill(w, m);
        load_stage<S>(w, d, g);
        load_ids<S>(w, m, f, d);
        const Pair *s = m.half(h);
        float4 A = s->A, B = s->B, H = s->H;
        for (int j0 = 0; j0 < top; j0 += kRows) {
            const int j1 = min(top, j0 + kRows);
#pragma unroll 2
            for (int j = j0; j < j1; j += 2, ++s) {
                const float2 power = power_of(p.pxc, p.pyc, A, B, make_float2(H.x, H.y));
                const float tau0 = H.z, tau1 = H.w;
                A = s[1].A;  // the next pair (any value past the last)
                B = s[1].B;
                H = s[1].H;
                const int2 pos = make_int2(s->pos[0], s->pos[1]);
                const float4 ca = s->c[0], cb = s->c[1];
                const float w0 = composite(p, !p.done && !skip(power.x, tau0), power.x, ca, pos.x);
                const float w1 = composite(p, !p.done && !skip(power.y, tau1), power.y, cb, pos.y);
                if (STATS) st.step(j, w0 > 0.f, w1 > 0.f);
                if (ACC) {
                    am->w[(j - j0) * kRowStride + lane] = w0;
                    am->w[(j - j0 + 1) * kRowStride + lane] = w1;
                }
            }
            if (ACC) flush_acc<S>(*am, m, j0, n, acc);
        }
        if (STATS) st.stage(reach);
    }
}

// Backward state of one pixel: its dL/dcolour g, T_final times g . background (TB), the
// transmittance T in front of the current entry and P = g . S, S the colour accumulated behind
// it (only that dot product enters the alpha gradient).
struct PixB {
    float pxc, pyc, T, TB, g0, g1, g2, P;
    int last;
};

__device__ __forceinline__ bool is_finite(float x) { return fabsf(x) < __int_as_float(0x7f800000); }

__device__ __forceinline__ float rcp_ftz(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One list entry for one pixel, in reverse, once the caller has evaluated the entry's power at
// the pixel: live = the pixel blended the entry (its position is within the pixel's contributor
// count and the power passes the cutoff). Gives this pixel's share of the entry's gradient
// sums as two numbers (zeros when not live), g = dL/dpower (alpha = o e^power) and the
// splatting weight w = alpha T, and when live steps T and P back past the entry. The sums over
// the pixels of g (dx, dy, dx^2, dx dy, dy^2, 1) and w dL/dcolour are formed later (flush_rows)
// from these. Branch-free, like the forward step: a lane that is not live keeps its state by
// selects, whatever its exponential gives.
__device__ __forceinline__ void accumulate(PixB &p, bool live, float power, const float4 &Cc, float &dpow,
                                           float &wgt) {
    const float araw = __fmul_rn(Cc.x, exp_ftz(power));
    const float alpha = fminf(kAlphaMax, araw);
    const float oma = 1.0f - alpha;
    const float inv = rcp_ftz(oma);  // 1 - alpha >= 0.01
    const float T = p.T * inv;       // transmittance in front of this Gaussian
    // dL/dalpha = T (g . c - g . S) - T_final / (1 - alpha) g . bg, then S <- alpha c + (1-alpha) S
    const float gc = fmaf(p.g2, Cc.w, fmaf(p.g1, Cc.z, p.g0 * Cc.y));
    const float dalpha = fmaf(T, gc - p.P, -p.TB * inv);
    const float P = fmaf(alpha, gc, oma * p.P);
    wgt = live ? alpha * T : 0.0f;
    p.T = live ? T : p.T;
    p.P = live ? P : p.P;
    // the clamp alpha = 0.99 passes no gradient to the opacity, conic or mean
    dpow = (live && !(araw > kAlphaMax)) ? dalpha * araw : 0.0f;
}

// Shared memory of the backward's gradient sums: per visit and pixel g = dL/dpower and the weight
// w, and the block's dL/dcolour, 0 in place of values that are not finite.
struct __align__(16) GradMem {
    float d[kRows * kRowStride], w[kRows * kRowStride];
    float dl[3 * 32];
};

// Adds the gradient sums of the entries in slots slot0 ... slot0 + 15 of each half (n[h] slots in all):
// the sums over the half's pixels of g (dx, dy, dx^2, dx dy, dy^2, 1), (dx, dy) = pixel centre -
// mean, and of w dL/dcolour, to the entries' 2-D gradient slots in g2, as 16-byte reductions. dy is
// one number per pixel row, so the y moments come from the row sums.
template <int S>
__device__ __forceinline__ void flush_grads(const GradMem &r, const WarpMem<S> &m, const Walk &w, int slot0,
                                            const int n[2], float *g2) {
    const int lane = threadIdx.x & 31, h = lane >> 4;
    const bool mine = slot0 + (lane & 15) < (h ? n[1] : n[0]);
    const int slot = mine ? slot0 + (lane & 15) : slot0;  // none: any other, its sums are not added
    __syncwarp();
    const float *a = reinterpret_cast<const float *>(&m.half(h)[slot >> 1].A) + (slot & 1);
    const float nu = a[0] + (w.bx0 + (float)(4 * h)), nv = a[2] + w.by0;  // first pixel centre - mean
    const float2 dx[2] = {make_float2(nu, nu + 1.0f), make_float2(nu + 2.0f, nu + 3.0f)};
    float t[9];
    float2 c0 = make_float2(0.f, 0.f), c1 = c0, c2 = c0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float dy = nv + (float)q;
        float2 g[2], x[2];
        row_pairs(r.d, q, g);
        x[0] = __fmul2_rn(g[0], dx[0]);
        x[1] = __fmul2_rn(g[1], dx[1]);
        const float2 r0 = __fadd2_rn(g[0], g[1]), r1 = __fadd2_rn(x[0], x[1]);
        const float2 r2 = __ffma2_rn(x[0], dx[0], __fmul2_rn(x[1], dx[1]));
        const float s0 = r0.x + r0.y, s1 = r1.x + r1.y, s2 = r2.x + r2.y, sy = dy * s0;
        t[0] = q ? t[0] + s1 : s1;
        t[1] = q ? t[1] + sy : sy;
        t[2] = q ? t[2] + s2 : s2;
        t[3] = q ? fmaf(dy, s1, t[3]) : dy * s1;
        t[4] = q ? fmaf(dy, sy, t[4]) : dy * sy;
        t[5] = q ? t[5] + s0 : s0;
        row_pairs(r.w, q, g);
        add_dot(c0, g, r.dl, q);
        add_dot(c1, g, r.dl + 32, q);
        add_dot(c2, g, r.dl + 64, q);
    }
    t[6] = c0.x + c0.y;
    t[7] = c1.x + c1.y;
    t[8] = c2.x + c2.y;
    unsigned any = 0u;  // all sums zero: no pixel took the entry
#pragma unroll
    for (int i = 0; i < 9; ++i) any |= __float_as_uint(t[i]);
    if (mine && (any << 1)) {
        float *dst = g2 + (size_t)m.half(h)[slot >> 1].idx[slot & 1] * kG2Floats;
        red_add4(dst, t[0], t[1], t[2], t[3]);
        red_add4(dst + 4, t[4], t[5], t[6], t[7]);
        red_add(dst + 8, t[8]);
    }
    __syncwarp();
}

// The colour gradients of a pixel whose dL/dcolour is infinite or undefined, over list positions [0, top): those values,
// which no weight changes, go to the entries that the pixel blends and to no others. In flush_grads, which takes 0 in
// their place, the zero weights of the other entries staged for the block would make their sums undefined.
__device__ __forceinline__ void odd_colours(const Walk &w, const PixB &p, int top, float *g2) {
#pragma unroll 1
    for (int k = min(p.last, top); k > 0; --k) {
        if (!((w.masks[k - 1] >> w.blk) & 1u)) continue;
        const size_t i = w.list[k - 1];
        const float4 r0 = w.rec[i * 3], r1 = w.rec[i * 3 + 1];
        const float hc = -0.5f * r1.x;
        const float power = power_of(p.pxc, p.pyc, make_float4(-r0.x, -r0.x, -r0.y, -r0.y),
                                     make_float4(-0.5f * r0.z, -0.5f * r0.z, -r0.w, -r0.w), make_float2(hc, hc)).x;
        if (skip(power, alpha_cut(r1.y)) || reach_of(r0, make_float2(r1.x, r1.y)).none) continue;
        float *dst = g2 + i * kG2Floats + 6;
        if (!is_finite(p.g0)) red_add(dst, p.g0);
        if (!is_finite(p.g1)) red_add(dst + 1, p.g1);
        if (!is_finite(p.g2)) red_add(dst + 2, p.g2);
    }
}

// The reverse walk of one pixel block over list positions [0, top), top the block's largest
// contributor count.
template <int S, bool STATS>
__device__ __forceinline__ void bwd_walk(const Walk &w, WarpMem<S> &m, GradMem &gm, PixB &p, float *g2, int last,
                                         WalkStats &st) {
    const int lane = threadIdx.x & 31, h = lane >> 4;
    if (last <= 0) return;
    Feed<S, -1> f;
    Ids<S> d;
    Stage<S> g;
    f.start(w, last);
    int scanned = f.fill(w, m);
    load_ids<S>(w, m, f, d);
    scanned += f.fill(w, m);
    load_stage<S>(w, d, g);
    load_ids<S>(w, m, f, d);
    while (g.id.n) {
        int n[2];
        unsigned reach[2];
        if (STATS) {
            st.staged += scanned;
            st.hits += g.id.n;
        }
        // the pixels that blended any of the stage's entries, or any in front of them: those whose contributor
        // count reaches the stage's last (foremost) entry
        int foremost = 0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int at = g.id.n - 1 - 32 * s;  // its lane, if it is among these 32
            const int v = __shfl_sync(0xffffffffu, (int)g.id.pos[s], at & 31);
            if (at >= 0 && at < 32) foremost = v;
        }
        const unsigned live = __ballot_sync(0xffffffffu, p.last >= foremost);
        const int top = commit<S>(w, g, m, live, n, reach);
        scanned = f.fill(w, m);
        load_stage<S>(w, d, g);
        load_ids<S>(w, m, f, d);
        const Pair *s = m.half(h);
        float4 A = s->A, B = s->B, H = s->H;
        for (int j0 = 0; j0 < top; j0 += kRows) {
            const int j1 = min(top, j0 + kRows);
#pragma unroll 2
            for (int j = j0; j < j1; j += 2, ++s) {
                const float2 power = power_of(p.pxc, p.pyc, A, B, make_float2(H.x, H.y));
                const float tau0 = H.z, tau1 = H.w;
                A = s[1].A;  // the next pair (any value past the last)
                B = s[1].B;
                H = s[1].H;
                const int2 pos = make_int2(s->pos[0], s->pos[1]);
                const float4 ca = s->c[0], cb = s->c[1];
                const bool l0 = pos.x <= p.last && !skip(power.x, tau0), l1 = pos.y <= p.last && !skip(power.y, tau1);
                if (STATS) st.step(j, l0, l1);
                float d0, d1, w0, w1;
                accumulate(p, l0, power.x, ca, d0, w0);
                accumulate(p, l1, power.y, cb, d1, w1);
                gm.d[(j - j0) * kRowStride + lane] = d0;
                gm.d[(j - j0 + 1) * kRowStride + lane] = d1;
                gm.w[(j - j0) * kRowStride + lane] = w0;
                gm.w[(j - j0 + 1) * kRowStride + lane] = w1;
            }
            flush_grads<S>(gm, m, w, j0, n, g2);
        }
        if (STATS) st.stage(reach);
    }
    // hardly ever true, and after the walk, which must not pay for it: tested in every flush, the heaviest blocks took
    // 10 % longer (one 64 x 64 frame of 100,000 Gaussians 603 -> 660 us), tested before the walk, 5 us at 128 x 128
    if (!(is_finite(p.g0) && is_finite(p.g1) && is_finite(p.g2))) odd_colours(w, p, last, g2);
}

// A (tile, pixel block) item: its frame, the block's pixel (one per lane: the block's left 4 x 4 pixels
// in the warp's first half, the right ones in the second, row by row) and the walk over the tile's list.
template <int TW>
__device__ __forceinline__ int block_item(const Ctx &c, unsigned item, int &px, int &py, Walk &w) {
    constexpr int TH = kTilePix / TW, NBX = TW / 8, NB = NBX * (TH / 4);
    static_assert(NB == 8, "one mask bit per block");
    const int lane = threadIdx.x & 31;
    const unsigned wk = item / NB, blk = item - wk * NB;
    const long long t = c.work[wk];
    const int b = find_frame(c, t);
    const FrameInfo &f = c.frames[b];
    const int lt = (int)(t - f.tile_base);
    const int ty = lt / f.tiles_x, tx = lt - ty * f.tiles_x;
    const int bx = tx * TW + (int)(blk % NBX) * 8, by = ty * TH + (int)(blk / NBX) * 4;
    px = bx + ((lane >> 4) << 2) + (lane & 3);
    py = by + ((lane >> 2) & 3);
    w.bx0 = (float)bx + 0.5f;
    w.by0 = (float)by + 0.5f;
    w.blk = blk;
    const unsigned st = c.tile_start[t];
    w.list = c.sorted + st;
    w.masks = c.list_masks(st);
    w.len = (int)(c.tile_start[t + 1] - st);
    w.rec = c.records + (size_t)f.rec_base * 3;
    w.masked = c.masked;
    return b;
}

// Adds a warp's statistics to the counters (dst: staged, hits, visits, pairs), the per-lane
// pair count summed over the warp first.
__device__ __forceinline__ void flush_stats(unsigned long long *dst, WalkStats st) {
    for (int o = 16; o > 0; o >>= 1) st.lanes += __shfl_xor_sync(0xffffffffu, st.lanes, o);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(dst + 0, st.staged);
        atomicAdd(dst + 1, st.hits);
        atomicAdd(dst + 2, st.visits);
        atomicAdd(dst + 3, (unsigned long long)st.lanes);
    }
}

// The loss: warp sums, then one double atomic per CTA.
__device__ __forceinline__ void flush_loss(const Ctx &c, float loss_acc, float *s_red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, o);
    if (lane == 0) s_red[wid] = loss_acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float sum = 0.f;
        for (int i = 0; i < kWarpsPerCta; ++i) sum += s_red[i];
        atomicAdd(&c.cnt->loss, (double)sum);
    }
}

// Items: the pixel blocks of the non-empty tiles (work list order, heaviest tiles first), and one item per
// empty tile, which the warp fills with the background. The empty tiles are spread evenly among the
// blocks: they are bound by memory (44 bytes a pixel with a target) and most of a face-centred frame, so
// they run in the shadow of the compositing instead of after it.
// ACC (colour initialisation, Eq. 3): every blended entry also adds its splatting weight w and
// w times the pixel's colour in acc_target to the record's first four 2-D gradient slots
// (flush_acc: one 16-byte reduction per entry and pixel block).
// STATS (the counting instance): also count the visits that evaluate an entry and the
// (pixel, entry) pairs that blend, into the compositing statistics of the counters.
// Bound by instruction issue (63 to 67 % of the slots), and by the walks of the heaviest blocks: six CTAs per SM
// beat eight (more warps, each slower) except where far more blocks have work than fit. Whole-warp
// entries with a vote per entry, then the half blocks with cut entries: 127 -> 115 us on 16 frames of 512 x 512
// (N = 60,000), 248 -> 182 us with the avatar bound to a mesh, 233 -> 148 us on 15 frames of 256 to 1,024 pixels of
// five avatars, 594 -> 514 us on 64 of eight, 66 -> 37 us on one of 128 x 128, colour initialisation of ten
// frames 107 -> 94 us. Empty tiles after all blocks instead of among the lighter ones: 559 us on the 64, before the cut.
template <int TW, int S, bool ACC, bool STATS = false>
__global__ void __launch_bounds__(32 * kWarpsPerCta, ACC ? 4 : 6)
k_render_fwd(Ctx c, float *__restrict__ img, float *__restrict__ T_final, int *__restrict__ n_contrib,
             const float *__restrict__ target, int loss_kind, float *__restrict__ dl_dimg,
             const float *__restrict__ acc_target) {
    constexpr int TH = kTilePix / TW, NB = (TW / 8) * (TH / 4);
    __shared__ WarpMem<S> s_m[kWarpsPerCta];
    __shared__ AccMem s_acc[ACC ? kWarpsPerCta : 1];
    __shared__ float s_red[kWarpsPerCta];
    pdl_enter();
    if (c.cnt->overflow) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    Walk w;
    AccMem *am = s_acc + (ACC ? wid : 0);
    const unsigned n_work = c.cnt->n_work, n_blocks = n_work * NB;
    const unsigned n_items = n_blocks + ((unsigned)c.T - n_work);
    // the first items, one per resident warp, are the heaviest blocks; from there empty tiles per item,
    // as a 32-bit fraction rounded up: e(i) = i frac / 2^32 of the next i items are empty tiles, and all
    // of them together are exactly the empty tiles
    const unsigned first = min(n_blocks, gridDim.x * kWarpsPerCta), rest = n_items - first;
    const unsigned long long frac = (((unsigned long long)(n_items - n_blocks) << 32) + rest - 1) / max(rest, 1u);
    const bool vec = ((reinterpret_cast<uintptr_t>(img) | reinterpret_cast<uintptr_t>(T_final) |
                       reinterpret_cast<uintptr_t>(n_contrib) | reinterpret_cast<uintptr_t>(target) |
                       reinterpret_cast<uintptr_t>(dl_dimg)) & 15) == 0;
    float loss_acc = 0.0f;
    WalkStats st{0ull, 0ull, 0ull, 0u, {0u, 0u}};  // STATS
    while (true) {
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(&c.cnt->next_fwd, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        unsigned e0 = 0u, e1 = 0u;
        if (item >= first) {
            e0 = (unsigned)(((item - first) * frac) >> 32);
            e1 = (unsigned)(((item - first + 1ull) * frac) >> 32);
        }
        if (e1 != e0) {  // an empty tile: background, T = 1, no contributors
            empty_tile<TW>(c, c.work[n_work + e0], vec, img, T_final, n_contrib, target, loss_kind, dl_dimg, loss_acc);
            continue;
        }
        item -= e0;
        int px, py;
        const int b = block_item<TW>(c, item, px, py, w);
        const FrameInfo &f = c.frames[b];
        PixF p{(float)px + 0.5f, (float)py + 0.5f, 1.f, 0.f, 0.f, 0.f, 0, px < f.W && py < f.H, false};
        p.done = !p.inside;
        if (ACC) {  // the pixel's target colour, read by flush_acc after its first __syncwarp
            const long long hw = (long long)f.W * f.H;
            const float *tg = acc_target + f.pix_base * 3 + (long long)py * f.W + px;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) am->target[32 * ch + lane] = p.inside ? tg[ch * hw] : 0.f;
        }
        fwd_walk<S, ACC, STATS>(w, s_m[wid], p, am, c.grad2d + (size_t)f.rec_base * kG2Floats, st);
        if (p.inside) {
            float g[3];
            finish_pixel(c, f, b, px, py, p, img, T_final, n_contrib, target, loss_kind, dl_dimg, loss_acc, g);
        }
    }
    if (STATS) flush_stats(c.cnt->st_fwd, st);
    // the last warp out puts the work counter back to zero for the next launch
    if (lane == 0 && atomicAdd(&c.cnt->done_fwd, 1u) == gridDim.x * kWarpsPerCta - 1) {
        c.cnt->next_fwd = 0u;
        c.cnt->done_fwd = 0u;
    }
    if (target) flush_loss(c, loss_acc, s_red);
}

// STATS (the counting instance): also count the visits that evaluate an entry and the
// (pixel, entry) pairs that take a gradient, into the compositing statistics of the counters.
// Bound by instruction issue (66 % of the slots, about 65 instructions per step of the two halves) and by the
// walks of the heaviest blocks: four CTAs per SM (128 registers) beat five and six. Whole-warp entries with
// a vote per entry, then the half blocks with cut entries: 16 frames of 512 x 512 of a 60,000-Gaussian avatar, not yet
// fitted, 170 -> 141 us, bound to a mesh 344 -> 240, 64 frames of eight avatars 644 -> 567; one 128 x 128 frame, where
// only 96 warps have work and the length of one warp's walk is what counts, 94 -> 45 to 51 us.
template <int TW, int S, bool STATS = false>
__global__ void __launch_bounds__(32 * kWarpsPerCta, 4)
k_render_bwd(Ctx c, const float *__restrict__ dl_dimg, const float *__restrict__ T_final,
             const int *__restrict__ n_contrib) {
    constexpr int TH = kTilePix / TW, NB = (TW / 8) * (TH / 4);
    __shared__ WarpMem<S> s_m[kWarpsPerCta];
    __shared__ GradMem s_g[kWarpsPerCta];
    pdl_enter();
    if (c.cnt->overflow) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    Walk w;
    GradMem &gm = s_g[wid];
    const unsigned n_items = c.cnt->n_work * NB;
    WalkStats st{0ull, 0ull, 0ull, 0u, {0u, 0u}};  // STATS
    while (true) {
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(&c.cnt->next_bwd, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        int px, py;
        const int b = block_item<TW>(c, item, px, py, w);
        const FrameInfo &f = c.frames[b];
        const float *bgp = c.fparams + (size_t)b * RGBA_FP_STRIDE + 17;
        const long long hw = (long long)f.W * f.H;
        PixB p{(float)px + 0.5f, (float)py + 0.5f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0};
        if (px < f.W && py < f.H) {
            const long long pix = (long long)py * f.W + px;
            const float Tfin = T_final[f.pix_base + pix];
            p.T = Tfin;
            p.last = n_contrib[f.pix_base + pix];
            const float *dl = dl_dimg + f.pix_base * 3 + pix;
            p.g0 = dl[0];
            p.g1 = dl[hw];
            p.g2 = dl[2 * hw];
            p.TB = Tfin * (p.g0 * bgp[0] + p.g1 * bgp[1] + p.g2 * bgp[2]);
        }
        // read by flush_grads, after its first __syncwarp
        gm.dl[lane] = is_finite(p.g0) ? p.g0 : 0.0f;
        gm.dl[32 + lane] = is_finite(p.g1) ? p.g1 : 0.0f;
        gm.dl[64 + lane] = is_finite(p.g2) ? p.g2 : 0.0f;
        int m = p.last;
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        // n_contrib comes from the caller: entries past the list's end do not exist
        const int top = min(m, w.len);
        float *g2 = c.grad2d + (size_t)f.rec_base * kG2Floats;
        bwd_walk<S, STATS>(w, s_m[wid], gm, p, g2, top, st);
    }
    if (STATS) flush_stats(c.cnt->st_bwd, st);
    // the last warp out puts the work counter back to zero for the next launch
    if (lane == 0 && atomicAdd(&c.cnt->done_bwd, 1u) == gridDim.x * kWarpsPerCta - 1) {
        c.cnt->next_bwd = 0u;
        c.cnt->done_bwd = 0u;
    }
}

// Persistent grid: every CTA the SMs can hold at once (occupancy query, cached by the caller
// per kernel instance: all instances of a template share one function type).
template <typename K>
int persistent_grid(K kernel, int sms_hint, int threads, int &cached) {
    if (!cached) {
        int per_sm = 0, dev = 0, sms = sms_hint;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess ||
            per_sm < 1)
            per_sm = 4;
        if (cudaGetDevice(&dev) == cudaSuccess)
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cached = per_sm * sms;
    }
    return cached;
}

template <int TW, int S, bool ACC, bool STATS = false>
cudaError_t fwd_inst(const Ctx &c, int grid, float *img, float *T, int *n, const float *tg, int lk,
                     float *dl, const float *acc_tg, cudaStream_t s) {
    static int cached = 0;
    const int g = persistent_grid(k_render_fwd<TW, S, ACC, STATS>, grid, 32 * kWarpsPerCta, cached);
    return launch_pdl(k_render_fwd<TW, S, ACC, STATS>, dim3(g), dim3(32 * kWarpsPerCta), 0, s, c, img, T, n,
                      tg, lk, dl, acc_tg);
}

// Stages of 64 entries instead of 32: in the forward where the caller asks for staging of 128 or 256, and in both
// directions for batches of at most kFewTiles tiles, whose blocks do not fill the SMs (a larger batch of mostly empty
// tiles may not fill them either, but how many are empty is known on the device only): their time is that of the longest
// walks, which larger stages shorten (fewer waits for records). With 32 and with 64 entries: one
// 64 x 64 frame of 100,000 Gaussians 852 against
// 688 us forwards and 866 against 612 backwards, eight of 128 x 128 272 against 238 and 336 against 270, one of
// 128 x 128 (N = 10,000) 43 against 37 and 55 against 45; where blocks abound the 32 are better (forward of 15 frames of
// five avatars 160 against 170 us, of 16 frames 121 against 125).
constexpr long long kFewTiles = 512;

template <bool ACC>
cudaError_t fwd_dispatch(const Ctx &c, int grid, int sb, float *img, float *T, int *n, const float *tg,
                         int lk, float *dl, const float *acc_tg, bool stats, cudaStream_t s) {
    if (!ACC && stats && c.tw == 16 && sb == 64)
        return fwd_inst<16, 1, false, true>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
    const bool large = sb != 64 || c.T <= kFewTiles;
    if (c.tw == 16)
        return large ? fwd_inst<16, 2, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s)
                     : fwd_inst<16, 1, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
    return large ? fwd_inst<8, 2, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s)
                 : fwd_inst<8, 1, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
}

template <int TW, int S, bool STATS = false>
cudaError_t bwd_inst(const Ctx &c, int grid, const float *dl, const float *T, const int *n,
                     cudaStream_t s) {
    static int cached = 0;
    const int g = persistent_grid(k_render_bwd<TW, S, STATS>, grid, 32 * kWarpsPerCta, cached);
    return launch_pdl(k_render_bwd<TW, S, STATS>, dim3(g), dim3(32 * kWarpsPerCta), 0, s, c, dl, T, n);
}

}  // namespace

cudaError_t launch_render_fwd(const Ctx &c, int grid, int smem_batch, float *img, float *T_final,
                              int *n_contrib, const float *target, int loss_kind,
                              float *dl_dimg, const float *acc_target, bool stats, cudaStream_t s) {
    if (acc_target)
        return fwd_dispatch<true>(c, grid, smem_batch, img, T_final, n_contrib, target, loss_kind, dl_dimg,
                                  acc_target, false, s);
    return fwd_dispatch<false>(c, grid, smem_batch, img, T_final, n_contrib, target, loss_kind, dl_dimg,
                               nullptr, stats, s);
}

// The backward's stages do not grow with smem_batch: its row sums take the shared memory.
cudaError_t launch_render_bwd(const Ctx &c, int grid, int smem_batch, const float *dl_dimg,
                              const float *T_final, const int *n_contrib, bool stats, cudaStream_t s) {
    if (stats && c.tw == 16 && smem_batch == 64) return bwd_inst<16, 1, true>(c, grid, dl_dimg, T_final, n_contrib, s);
    const bool large = c.T <= kFewTiles;
    if (c.tw == 16)
        return large ? bwd_inst<16, 2>(c, grid, dl_dimg, T_final, n_contrib, s)
                     : bwd_inst<16, 1>(c, grid, dl_dimg, T_final, n_contrib, s);
    return large ? bwd_inst<8, 2>(c, grid, dl_dimg, T_final, n_contrib, s)
                 : bwd_inst<8, 1>(c, grid, dl_dimg, T_final, n_contrib, s);
}

}  // namespace rgba
