// Front-to-back alpha compositing ("rasterize", RGBAvatar Sec. 3.2 on the 3DGS renderer) and
// its exact reverse. The binning tile (16x16 or 8x32 pixels) fixes the lists; the compositing
// work is split finer: every warp is an independent persistent worker that takes (tile, pixel
// block) items from one counter, so the few heavy tiles of a face-centred frame spread over
// many warps and no warp ever waits at a CTA barrier. A block is 8 x 4 pixels, one per lane.
//
// Every list entry comes with a byte that says which of the tile's eight blocks its splat can
// reach (made once per (Gaussian, tile) by the scatter). A warp scans its tile's list 64 entries
// at a time, keeps those whose bit for its block is set in a queue of its own, and stages 32 S of
// the queued entries at a time: each lane loads the records of S of them (one step ahead of the
// compositing) and writes them, in the form the pixel loop reads, to the warp's shared-memory
// slots. The warp then visits the slots in list order (in reverse in the backward): it evaluates
// the power at every pixel, skips the entry when no lane passes the cutoff, and otherwise runs
// the pixel step without branches (lanes that do not take part keep their state). The forward
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

// power = -(a dx^2 + c dy^2)/2 - b dx dy = dx ((-a/2) dx + (-b) dy) + (-c/2) dy dy, from a staged
// entry's (u, v, -a/2, -b) and -c/2. Both kernels evaluate through this function and cut with
// skip(), so their decisions agree bit for bit.
__device__ __forceinline__ float power_of(float dx, float dy, const float4 &A, float hc) {
    return __fmaf_rn(dx, __fmaf_rn(A.z, dx, __fmul_rn(A.w, dy)), __fmul_rn(__fmul_rn(hc, dy), dy));
}

// the skip decision: a positive power (never, for a positive definite conic, but kept as the
// definition) or alpha below 1/255 (alpha_cut): most pairs, the far tail of a splat, are rejected
// before the exponential and before the colour is read
__device__ __forceinline__ bool skip(float power, float tau) { return power > 0.0f || power < tau; }

struct PixF {
    float pxc, pyc, T, C0, C1, C2;
    int last;
    bool inside, done;
};

// One list entry for one pixel (forward), once the caller has evaluated the entry's power at
// the pixel: live = the pixel is still compositing and the entry passes the alpha cutoff. A live
// entry that would take T (1 - alpha) below 1e-4 marks the pixel done without blending;
// otherwise it blends. Branch-free, so a warp whose lanes disagree runs it once: a lane that is
// not live keeps its state whatever its exponential gives (alpha is capped at 0.99 and its
// weight is 0). Returns the splatting weight alpha T at the pixel (0 when the entry does not
// blend).
__device__ __forceinline__ float composite(PixF &p, bool live, float power, const float4 &Cc, int pos) {
    const float alpha = fminf(kAlphaMax, __fmul_rn(Cc.x, __expf(power)));
    const float testT = p.T * (1.0f - alpha);
    const bool sat = testT < kTMin;
    p.done = p.done || (live && sat);
    const bool blend = live && !sat;
    const float w = blend ? alpha * p.T : 0.0f;
    p.C0 = fmaf(Cc.y, w, p.C0);
    p.C1 = fmaf(Cc.z, w, p.C1);
    p.C2 = fmaf(Cc.w, w, p.C2);
    p.T = blend ? testT : p.T;
    p.last = blend ? pos : p.last;
    return w;
}

constexpr int kWarpsPerCta = 4;  // independent warps per CTA (they share nothing but the loss sum)

// A warp's shared memory: the queue of entries that reach its block, and the staged slots
// (32 S of them, and one past the end for the loop's look-ahead).
//   a = (u, v, -a/2, -b)   q = (-c/2, tau, list position + 1, Gaussian index)   c = (opacity, r, g, b)
template <int S>
struct WarpMem {
    static constexpr int kQueue = S > 2 ? 256 : 128;  // holds a stage's worth and one scan
    float4 a[32 * S + 1], q[32 * S + 1], c[32 * S];
    uint2 queue[kQueue];  // (list position + 1, Gaussian index)
};

// One compositing warp's view of a (tile, pixel block) item: the tile's list and the block.
struct Walk {
    const unsigned *list;        // the tile's sorted Gaussian indices
    const unsigned char *masks;  // and their block masks
    int len;
    unsigned blk;
    const float4 *rec;  // the frame's render records
    float bx0, by0;     // the block's first pixel centre
};

// The entries of list positions [lo, hi) that reach the block, front to back (DIR = 1) or back to
// front (DIR = -1). scan() appends the hits among the next 64 entries to the queue; the 64 after
// them are in flight meanwhile.
template <int S, int DIR>
struct Feed {
    int lo, hi, at;       // entries not scanned yet: [at, hi) or [lo, at)
    unsigned head, count; // the queue's first element and length
    unsigned idx[2];      // the loaded entries: lane + 32 i past `at`
    bool hit[2];

    __device__ __forceinline__ void load(const Walk &w) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int e = DIR > 0 ? at + lane + 32 * i : at - 1 - lane - 32 * i;
            const bool in = DIR > 0 ? e < hi : e >= lo;
            hit[i] = in && ((w.masks[in ? e : lo] >> w.blk) & 1u);
            idx[i] = in ? w.list[e] : 0u;
        }
    }
    __device__ __forceinline__ void start(const Walk &w, int lo_, int hi_) {
        lo = lo_;
        hi = hi_;
        at = DIR > 0 ? lo : hi;
        head = count = 0u;
        load(w);
    }
    __device__ __forceinline__ bool more() const { return DIR > 0 ? at < hi : at > lo; }
    // until the queue holds a stage's worth (or the list is done); returns the entries scanned
    __device__ __forceinline__ int fill(const Walk &w, WarpMem<S> &m) {
        constexpr unsigned Q = WarpMem<S>::kQueue - 1;
        const int lane = threadIdx.x & 31;
        int scanned = 0;
        while (count < 32u * S && more()) {
            const unsigned b0 = __ballot_sync(0xffffffffu, hit[0]), b1 = __ballot_sync(0xffffffffu, hit[1]);
            const unsigned lt = (1u << lane) - 1u, n0 = __popc(b0), tail = head + count;
            const unsigned pos = DIR > 0 ? at + lane + 1 : at - lane;  // list position + 1
            if (hit[0]) m.queue[(tail + __popc(b0 & lt)) & Q] = make_uint2(pos, idx[0]);
            if (hit[1]) m.queue[(tail + n0 + __popc(b1 & lt)) & Q] = make_uint2(pos + DIR * 32, idx[1]);
            count += n0 + __popc(b1);
            scanned += DIR > 0 ? min(64, hi - at) : min(64, at - lo);
            at += DIR * 64;
            load(w);
        }
        __syncwarp();
        return scanned;
    }
};

// The records of the next 32 S queued entries, on their way to the slots: lane l takes entries
// l, l + 32, ...
template <int S>
struct Stage {
    uint2 e[S];
    float4 r0[S], r1[S];
    float r2[S];
    int n;  // entries
};

template <int S, int DIR>
__device__ __forceinline__ void load_stage(const Walk &w, const WarpMem<S> &m, Feed<S, DIR> &f, Stage<S> &g) {
    const int lane = threadIdx.x & 31;
    g.n = min((int)f.count, 32 * S);
#pragma unroll
    for (int s = 0; s < S; ++s) {
        if (lane + 32 * s < g.n) {
            g.e[s] = m.queue[(f.head + lane + 32 * s) & (WarpMem<S>::kQueue - 1)];
            const float4 *r = w.rec + (size_t)g.e[s].y * 3;
            g.r0[s] = r[0];
            g.r1[s] = r[1];
            g.r2[s] = r[2].x;
        }
    }
    f.head += g.n;
    f.count -= g.n;
}

template <int S>
__device__ __forceinline__ void commit(const Stage<S> &g, WarpMem<S> &m) {
    const int lane = threadIdx.x & 31;
    __syncwarp();  // the previous stage's slots are no longer read
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int k = lane + 32 * s;
        if (k < g.n) {
            m.a[k] = make_float4(g.r0[s].x, g.r0[s].y, -0.5f * g.r0[s].z, -g.r0[s].w);
            m.q[k] = make_float4(-0.5f * g.r1[s].x, alpha_cut(g.r1[s].y), __uint_as_float(g.e[s].x),
                                 __uint_as_float(g.e[s].y));
            m.c[k] = make_float4(g.r1[s].y, g.r1[s].z, g.r1[s].w, g.r2[s]);
        }
    }
    __syncwarp();
}

// A fire-and-forget global float add.
__device__ __forceinline__ void red_add(float *addr, float v) {
    asm volatile("red.global.add.f32 [%0], %1;" :: "l"(addr), "f"(v) : "memory");
}

// Adds 4 floats at a 16-byte aligned address of global memory.
__device__ __forceinline__ void red_add4(float *addr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" :: "l"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// Sums over pixels for 16 slots at a time. The visit of slot j leaves one or two numbers per pixel
// (lane) in row j % 16 of a shared-memory matrix; after 16 slots the warp turns round: lane l takes
// the entry of row l % 16 and the pixel rows 2 (l / 16) and 2 (l / 16) + 1 of the block, and adds up
// its 16 pixels from 16-byte loads, two columns per packed FP32 instruction. Per visit that costs
// the stores and a sixteenth of about 150 instructions, where a shuffle reduction of nine sums
// over the lanes takes about 45 and puts ten dependent shuffles into every visit. The rows are
// padded to 36 floats so that the 16-byte loads of eight lanes fall in different banks.
constexpr int kRows = 16;
constexpr int kRowStride = 36;

// The 16 pixel values of this lane's row and pixel rows, as pairs of neighbouring columns.
__device__ __forceinline__ void row_pairs(const float *rows, int q, float2 v[4]) {
    const int lane = threadIdx.x & 31;
    const float4 *p = reinterpret_cast<const float4 *>(rows + (lane & 15) * kRowStride + 8 * (2 * (lane >> 4) + q));
    const float4 a = p[0], b = p[1];
    v[0] = make_float2(a.x, a.y);
    v[1] = make_float2(a.z, a.w);
    v[2] = make_float2(b.x, b.y);
    v[3] = make_float2(b.z, b.w);
}

// c += sum over the pairs of w times the block's per-pixel values `pix` (pixel row 2 (lane / 16) + q)
__device__ __forceinline__ void add_dot(float2 &c, const float2 w[4], const float *pix, int q) {
    const float4 *p = reinterpret_cast<const float4 *>(pix + 8 * (2 * ((threadIdx.x & 31) >> 4) + q));
    const float4 a = p[0], b = p[1];
    c = __ffma2_rn(w[0], make_float2(a.x, a.y), c);
    c = __ffma2_rn(w[1], make_float2(a.z, a.w), c);
    c = __ffma2_rn(w[2], make_float2(b.x, b.y), c);
    c = __ffma2_rn(w[3], make_float2(b.z, b.w), c);
}

// Adds over both halves of the warp: lanes l and l + 16 hold the two halves of a block's pixels.
template <int N>
__device__ __forceinline__ void add_halves(float t[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] += __shfl_xor_sync(0xffffffffu, t[i], 16);
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

// An empty tile's item: the background, T = 1, no contributors, eight pixels per lane.
template <int TW>
__device__ __forceinline__ void empty_tile(const Ctx &c, long long t, float *img, float *T_final, int *n_contrib,
                                           const float *target, int loss_kind, float *dl_dimg, float &loss_acc) {
    constexpr int TH = kTilePix / TW;
    const int lane = threadIdx.x & 31;
    const int b = find_frame(c, t);
    const FrameInfo &f = c.frames[b];
    const int lt = (int)(t - f.tile_base);
    const int ty = lt / f.tiles_x, tx = lt - ty * f.tiles_x;
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

// Compositing statistics of one warp (counting instances only): list entries scanned, entries
// that reach the block by their mask, visits that evaluated an entry (one with some pixel past the
// cutoffs; warp-uniform), and the (pixel, entry) pairs that blend or take a gradient (this lane's).
struct WalkStats {
    unsigned long long staged, hits, visits;
    unsigned lanes;
};

// Shared memory of the colour initialisation's sums: the visits' weights and the block's target.
struct __align__(16) AccMem {
    float w[kRows * kRowStride];
    float target[3 * 32];
};

// Adds the weights w and w times the target colour of 16 slots' entries (slot0 ...; bit e of
// `visited`: row e holds a visit) to their records' first four accumulators in acc.
template <int S>
__device__ __forceinline__ void flush_acc(const AccMem &r, const WarpMem<S> &m, int slot0, unsigned visited, float *acc) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    float2 s = make_float2(0.f, 0.f), c0 = s, c1 = s, c2 = s;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        float2 v[4];
        row_pairs(r.w, q, v);
        s = __fadd2_rn(s, __fadd2_rn(__fadd2_rn(v[0], v[1]), __fadd2_rn(v[2], v[3])));
        add_dot(c0, v, r.target, q);
        add_dot(c1, v, r.target + 32, q);
        add_dot(c2, v, r.target + 64, q);
    }
    float t[4] = {s.x + s.y, c0.x + c0.y, c1.x + c1.y, c2.x + c2.y};
    add_halves<4>(t);
    if (lane < 16 && ((visited >> lane) & 1u))
        red_add4(acc + (size_t)__float_as_uint(m.q[slot0 + lane].w) * kG2Floats, t[0], t[1], t[2], t[3]);
    __syncwarp();
}

// The forward walk of one pixel block, until every pixel of the block is done or the list ends.
// ACC: colour-initialisation accumulation into acc (see k_render_fwd).
template <int S, bool ACC, bool STATS>
__device__ __forceinline__ void fwd_walk(const Walk &w, WarpMem<S> &m, PixF &p, AccMem *am, float *acc, WalkStats &st) {
    const int lane = threadIdx.x & 31;
    Feed<S, 1> f;
    Stage<S> g;
    f.start(w, 0, w.len);
    int scanned = f.fill(w, m);
    load_stage<S>(w, m, f, g);
    while (g.n) {
        if (STATS) st.staged += scanned;
        if (__all_sync(0xffffffffu, p.done)) break;
        const int n = g.n;
        commit<S>(g, m);
        scanned = f.fill(w, m);
        load_stage<S>(w, m, f, g);
        float4 A = m.a[0], Q = m.q[0];
        for (int j0 = 0; j0 < n; j0 += kRows) {
            unsigned visited = 0u;
            const int j1 = min(n, j0 + kRows);
#pragma unroll 4
            for (int j = j0; j < j1; ++j) {
                const float4 An = m.a[j + 1], Qn = m.q[j + 1];  // the next slot (any value past the last)
                const float dx = __fsub_rn(p.pxc, A.x), dy = __fsub_rn(p.pyc, A.y);
                const float power = power_of(dx, dy, A, Q.x);
                const bool live = !p.done && !skip(power, Q.y);
                if (STATS) ++st.hits;
                if (__any_sync(0xffffffffu, live)) {  // else the colour is not even read
                    const float wgt = composite(p, live, power, m.c[j], (int)__float_as_uint(Q.z));
                    if (STATS) {
                        ++st.visits;
                        st.lanes += wgt > 0.0f ? 1u : 0u;
                    }
                    if (ACC) {
                        am->w[(j - j0) * kRowStride + lane] = wgt;
                        visited |= 1u << (j - j0);
                    }
                }
                A = An;
                Q = Qn;
            }
            if (ACC && visited) flush_acc<S>(*am, m, j0, visited, acc);
        }
    }
}

// Backward state of one pixel: its dL/dcolour g, T_final times g . background (TB), the
// transmittance T in front of the current entry and P = g . S, S the colour accumulated behind
// it (only that dot product enters the alpha gradient).
struct PixB {
    float pxc, pyc, T, TB, g0, g1, g2, P;
    int last;
};

// e^x for the compositing backward, as 2^(x log2 e) on the hardware's base-2 exponential in its
// flush-to-zero form: the general form guards against subnormal results with three more
// instructions, and no weight that counts (alpha >= 1/255) is near that range.
__device__ __forceinline__ float exp_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__fmul_rn(x, 1.44269504088896341f)));
    return y;
}
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
// w, and the block's dL/dcolour.
struct __align__(16) GradMem {
    float d[kRows * kRowStride], w[kRows * kRowStride];
    float dl[3 * 32];
};

// Adds the gradient sums of 16 slots' entries (slot0 ...; bit e of `visited`: row e holds a visit):
// the sums over the block's pixels of g (dx, dy, dx^2, dx dy, dy^2, 1), (dx, dy) = pixel centre -
// mean, and of w dL/dcolour, to the entries' 2-D gradient slots in g2. dy is one number per pixel
// row, so the y moments come from the row sums. Each half of the warp adds half of the nine sums
// as 16-byte reductions: scalar ones of the same sums are nine instead of three per entry.
template <int S>
__device__ __forceinline__ void flush_grads(const GradMem &r, const WarpMem<S> &m, const Walk &w, int slot0,
                                            unsigned visited, float *g2) {
    const int lane = threadIdx.x & 31, e = lane & 15, h = lane >> 4;
    __syncwarp();
    const bool mine = (visited >> e) & 1u;
    const int slot = mine ? slot0 + e : slot0;  // a slot not visited: any other, its sums are not added
    const float2 uv = *reinterpret_cast<const float2 *>(&m.a[slot]);
    float2 dx[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) dx[i] = make_float2(w.bx0 + (float)(2 * i) - uv.x, w.bx0 + (float)(2 * i + 1) - uv.x);
    float t[9];
    float2 c0 = make_float2(0.f, 0.f), c1 = c0, c2 = c0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float dy = w.by0 + (float)(2 * h + q) - uv.y;
        float2 g[4], x[4];
        row_pairs(r.d, q, g);
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = __fmul2_rn(g[i], dx[i]);
        const float2 r0 = __fadd2_rn(__fadd2_rn(g[0], g[1]), __fadd2_rn(g[2], g[3]));
        const float2 r1 = __fadd2_rn(__fadd2_rn(x[0], x[1]), __fadd2_rn(x[2], x[3]));
        const float2 r2 = __fadd2_rn(__ffma2_rn(x[0], dx[0], __fmul2_rn(x[1], dx[1])),
                                     __ffma2_rn(x[2], dx[2], __fmul2_rn(x[3], dx[3])));
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
    add_halves<9>(t);
    if (mine) {
        float *dst = g2 + (size_t)__float_as_uint(m.q[slot].w) * kG2Floats;
        if (h == 0) {
            red_add4(dst, t[0], t[1], t[2], t[3]);
        } else {
            red_add4(dst + 4, t[4], t[5], t[6], t[7]);
            red_add(dst + 8, t[8]);
        }
    }
    __syncwarp();
}

// The reverse walk of one pixel block over list positions [0, top), top the block's largest
// contributor count.
template <int S, bool STATS>
__device__ __forceinline__ void bwd_walk(const Walk &w, WarpMem<S> &m, GradMem &gm, PixB &p, float *g2, int top,
                                         WalkStats &st) {
    const int lane = threadIdx.x & 31;
    if (top <= 0) return;
    Feed<S, -1> f;
    Stage<S> g;
    f.start(w, 0, top);
    int scanned = f.fill(w, m);
    load_stage<S>(w, m, f, g);
    while (g.n) {
        if (STATS) st.staged += scanned;
        const int n = g.n;
        commit<S>(g, m);
        scanned = f.fill(w, m);
        load_stage<S>(w, m, f, g);
        float4 A = m.a[0], Q = m.q[0];
        for (int j0 = 0; j0 < n; j0 += kRows) {
            unsigned visited = 0u;
            const int j1 = min(n, j0 + kRows);
#pragma unroll 2
            for (int j = j0; j < j1; ++j) {
                const float4 An = m.a[j + 1], Qn = m.q[j + 1];  // the next slot (any value past the last)
                const float dx = __fsub_rn(p.pxc, A.x), dy = __fsub_rn(p.pyc, A.y);
                const float power = power_of(dx, dy, A, Q.x);
                const bool live = (int)__float_as_uint(Q.z) <= p.last && !skip(power, Q.y);
                if (STATS) ++st.hits;
                if (__any_sync(0xffffffffu, live)) {  // else the colour is not even read
                    if (STATS) {
                        ++st.visits;
                        st.lanes += live ? 1u : 0u;
                    }
                    float dpow, wgt;
                    accumulate(p, live, power, m.c[j], dpow, wgt);
                    gm.d[(j - j0) * kRowStride + lane] = dpow;
                    gm.w[(j - j0) * kRowStride + lane] = wgt;
                    visited |= 1u << (j - j0);
                }
                A = An;
                Q = Qn;
            }
            if (visited) flush_grads<S>(gm, m, w, j0, visited, g2);
        }
    }
}

// A (tile, pixel block) item: its frame, the block's pixel (one per lane: column lane % 8 of
// row lane / 8 of the 8 x 4 block) and the walk over the tile's list.
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
    px = bx + (lane & 7);
    py = by + (lane >> 3);
    w.bx0 = (float)bx + 0.5f;
    w.by0 = (float)by + 0.5f;
    w.blk = blk;
    const unsigned st = c.tile_start[t];
    w.list = c.sorted + st;
    w.masks = c.list_masks(st);
    w.len = (int)(c.tile_start[t + 1] - st);
    w.rec = c.records + (size_t)f.rec_base * 3;
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

// Items: the pixel blocks of the non-empty tiles (work list order, heaviest tiles first), then
// one item per empty tile, which the warp fills with the background eight pixels per lane.
// ACC (colour initialisation, Eq. 3): every blended entry also adds its splatting weight w and
// w times the pixel's colour in acc_target to the record's first four 2-D gradient slots
// (flush_acc: one 16-byte reduction per entry and pixel block).
// STATS (the counting instance): also count the visits that evaluate an entry and the
// (pixel, entry) pairs that blend, into the compositing statistics of the counters.
// Bound by instruction issue, and by one warp's walk where few blocks have work. Against staging and
// testing every list entry per block: 160 -> 127 us on 16 frames of 512 x 512 (N = 60,000), 123 ->
// 72 us on one of 128 x 128, colour initialisation of ten frames 178 -> 107 us.
template <int TW, int S, bool ACC, bool STATS = false>
__global__ void __launch_bounds__(32 * kWarpsPerCta)
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
    float loss_acc = 0.0f;
    WalkStats st{0ull, 0ull, 0ull, 0u};  // STATS
    while (true) {
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(&c.cnt->next_fwd, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        if (item >= n_blocks) {  // an empty tile: background, T = 1, no contributors
            empty_tile<TW>(c, c.work[n_work + (item - n_blocks)], img, T_final, n_contrib, target, loss_kind,
                           dl_dimg, loss_acc);
            continue;
        }
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
// Bound by instruction issue. 16 frames of 512 x 512 of a 60,000-Gaussian avatar, not yet fitted:
// 301 -> 170 us (222 -> 117 M warp instructions) against staging every list entry per block and
// reducing nine sums by shuffles at every visit; one 128 x 128 frame, where only 80 warps have work
// and the length of one warp's walk is what counts: 182 -> 96 us. Six CTAs per SM (80 registers):
// without the bound the row sums take 128 registers and the occupancy they cost eats the gain
// (307 us).
template <int TW, int S, bool STATS = false>
__global__ void __launch_bounds__(32 * kWarpsPerCta, S == 1 ? 6 : 1)
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
    WalkStats st{0ull, 0ull, 0ull, 0u};  // STATS
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
        gm.dl[lane] = p.g0;  // read by flush_grads, after its first __syncwarp
        gm.dl[32 + lane] = p.g1;
        gm.dl[64 + lane] = p.g2;
        int m = p.last;
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        // n_contrib comes from the caller: entries past the list's end do not exist
        bwd_walk<S, STATS>(w, s_m[wid], gm, p, c.grad2d + (size_t)f.rec_base * kG2Floats, min(m, w.len), st);
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

template <bool ACC>
cudaError_t fwd_dispatch(const Ctx &c, int grid, int sb, float *img, float *T, int *n, const float *tg,
                         int lk, float *dl, const float *acc_tg, bool stats, cudaStream_t s) {
    if (!ACC && stats && c.tw == 16 && sb == 64)
        return fwd_inst<16, 1, false, true>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
    if (c.tw == 16) {
        if (sb == 64) return fwd_inst<16, 1, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
        if (sb == 128) return fwd_inst<16, 2, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
        return fwd_inst<16, 3, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
    }
    if (sb == 64) return fwd_inst<8, 1, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
    if (sb == 128) return fwd_inst<8, 2, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
    return fwd_inst<8, 3, ACC>(c, grid, img, T, n, tg, lk, dl, acc_tg, s);
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

cudaError_t launch_render_bwd(const Ctx &c, int grid, int smem_batch, const float *dl_dimg,
                              const float *T_final, const int *n_contrib, bool stats, cudaStream_t s) {
    if (stats && c.tw == 16 && smem_batch == 64) return bwd_inst<16, 1, true>(c, grid, dl_dimg, T_final, n_contrib, s);
    if (c.tw == 16) {
        if (smem_batch == 64) return bwd_inst<16, 1>(c, grid, dl_dimg, T_final, n_contrib, s);
        if (smem_batch == 128) return bwd_inst<16, 2>(c, grid, dl_dimg, T_final, n_contrib, s);
        return bwd_inst<16, 3>(c, grid, dl_dimg, T_final, n_contrib, s);
    }
    if (smem_batch == 64) return bwd_inst<8, 1>(c, grid, dl_dimg, T_final, n_contrib, s);
    if (smem_batch == 128) return bwd_inst<8, 2>(c, grid, dl_dimg, T_final, n_contrib, s);
    return bwd_inst<8, 3>(c, grid, dl_dimg, T_final, n_contrib, s);
}

}  // namespace rgba
