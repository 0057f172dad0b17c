// Backward through the projection (EWA splatting, activations) and the linear blend (Eq. 1).
//
//   k_gauss_bwd  one CTA per 32 Gaussians of one model, lane = Gaussian, frames 8 or 16 at a time:
//                first, per (frame, Gaussian), the 2-D gradients dL/d(u, v, conic, opacity,
//                colour) from the compositing backward's sums -> dL/dG_b over the 14 channels
//                (chain rule through conic inversion, J W Sigma W^T J^T, R diag(s^2) R^T,
//                quaternion normalisation, exp and sigmoid) into shared memory; then the
//                adjoint of Eq. 1:
//                dG0[ch][i]    += sum_b dG_b[ch][i]
//                ddG[k][a][i]  += sum_b psi_b[k] dG_b[ch_a][i]
//                dpsi_b[k]     partial = sum_{a, i in chunk} dG_k[a][i] dG_b[ch_a][i]
//                the last two as TF32 tensor-core products at FP32 accuracy (three products
//                of split operands).
// Every sum runs in a fixed order (dG0 in registers, the products tile by tile, the warps'
// dpsi sums in warp order), so the results are deterministic; dpsi partials go to a
// [frame][k][chunk] buffer that a second kernel sums.
#include <type_traits>

#include "rgba_internal.cuh"

namespace rgba {
namespace {

constexpr int kBwdThreads = 256;

// The gradient of one (frame, Gaussian) with respect to its 14 blended channels, from the
// compositing backward's sums over the pixels that blend it: S = (S1, S2, S3, S4, S5, S0) of
// g (dx, dy, dx^2, dx dy, dy^2, 1) with g = dL/dpower and (dx, dy) = pixel centre - mean, then
// dL/d(r, g, b). As power = -(a dx^2 + c dy^2) / 2 - b dx dy and alpha = o e^power:
// dL/du = a S1 + b S2, dL/dv = b S1 + c S2, dL/d(a, b, c) = (-S3 / 2, -S4, -S5 / 2) and
// dL/do = S0 / o, with the conic Q = (a, b, c) = Sigma'^-1 recomputed here.
//
// The 2-D covariance is kept as a product of thin factors, Sigma' = U diag(s^2) U^T + 0.3 I with
// U = T R and T = J W (2 x 3), so that no 3 x 3 product is formed on the way back either:
//   G = dL/dSigma' = -Q dL/dQ Q,   dL/ds_m^2 = (U^T G U)_mm,   X = dL/dU = 2 G U diag(s^2),
//   dL/dR = T^T X,   dL/dT = X R^T,   dL/dJ = dL/dT W^T.
// That is about 300 operations where the 3 x 3 covariances and their adjoints took about 900.
// The backward needs no bit-exact replay of the forward decisions (those come from the
// records), only fp32 values to the gradient tolerance, so it uses the hardware's fast
// reciprocal, reciprocal square root and exponential.
//
// v: mean(3), quaternion(4), log-scale(3); V: the frame's parameters; lim: the Jacobian clamp
// bounds 1.3 tan(fov / 2) in x and y. BOUND: Rt [12] = TBN matrix row-major (columns T, B, N), then t
// (the identity and zero for an unbound model of a batch that also has bound ones); the Gaussian
// is mapped from tangent space by x = Rt x_T + t, which makes W the view rotation times Rt. !BOUND:
// no mapping (Rt is not read).
template <bool BOUND>
__device__ __forceinline__ void chain(const float v[10], float op, const float *V, const float *lim,
                                      const float *Rt, const float g2[9], float dG[kNch]) {
    float W[3][3], p[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            W[j][c] = BOUND ? V[4 * j] * Rt[c] + V[4 * j + 1] * Rt[3 + c] + V[4 * j + 2] * Rt[6 + c] : V[4 * j + c];
        p[j] = V[4 * j + 3];
        if (BOUND) p[j] += V[4 * j] * Rt[9] + V[4 * j + 1] * Rt[10] + V[4 * j + 2] * Rt[11];
        p[j] += W[j][0] * v[0] + W[j][1] * v[1] + W[j][2] * v[2];
    }
    float d[3];  // squared scales
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const float s = __expf(v[7 + m]);
        d[m] = s * s;
    }
    const float il = rsqrtf(v[3] * v[3] + v[4] * v[4] + v[5] * v[5] + v[6] * v[6]);
    const float w = v[3] * il, x = v[4] * il, y = v[5] * il, z = v[6] * il;
    const float R[3][3] = {{1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y)},
                           {2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x)},
                           {2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)}};
    const float fx = V[12], fy = V[13], ipz = __frcp_rn(p[2]);
    const float rx0 = p[0] * ipz, ry0 = p[1] * ipz;
    const bool clx = rx0 > lim[0] || rx0 < -lim[0], cly = ry0 > lim[1] || ry0 < -lim[1];
    const float rx = fminf(lim[0], fmaxf(-lim[0], rx0)), ry = fminf(lim[1], fmaxf(-lim[1], ry0));
    const float j00 = fx * ipz, j02 = -j00 * rx, j11 = fy * ipz, j12 = -j11 * ry;  // the entries of J
    float T[2][3], U[2][3], UD[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        T[0][c] = j00 * W[0][c] + j02 * W[2][c];
        T[1][c] = j11 * W[1][c] + j12 * W[2][c];
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            U[r][m] = T[r][0] * R[0][m] + T[r][1] * R[1][m] + T[r][2] * R[2][m];
            UD[r][m] = U[r][m] * d[m];
        }
    const float A = U[0][0] * UD[0][0] + U[0][1] * UD[0][1] + U[0][2] * UD[0][2] + 0.3f;
    const float B = U[0][0] * UD[1][0] + U[0][1] * UD[1][1] + U[0][2] * UD[1][2];
    const float C = U[1][0] * UD[1][0] + U[1][1] * UD[1][1] + U[1][2] * UD[1][2] + 0.3f;
    const float iD = __frcp_rn(A * C - B * B);
    const float ca = C * iD, cb = -B * iD, cc = A * iD;
    const float du = ca * g2[0] + cb * g2[1], dv = cb * g2[0] + cc * g2[1];
    dG[10] = g2[5] * (1.f - op);  // dL/do times the sigmoid's o (1 - o)
    dG[11] = g2[6];
    dG[12] = g2[7];
    dG[13] = g2[8];
    // G = -Q H Q with H = dL/dQ = -(S3, S4, S5) / 2 as a symmetric matrix: the signs cancel
    const float ha = 0.5f * g2[2], hb = 0.5f * g2[3], hc = 0.5f * g2[4];
    const float q00 = ca * ha + cb * hb, q01 = ca * hb + cb * hc, q10 = cb * ha + cc * hb, q11 = cb * hb + cc * hc;
    const float ga = q00 * ca + q01 * cb, gb = q00 * cb + q01 * cc, gc = q10 * cb + q11 * cc;
    float X[2][3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const float h0 = ga * U[0][m] + gb * U[1][m], h1 = gb * U[0][m] + gc * U[1][m];
        const float d2 = 2.f * d[m];
        dG[7 + m] = d2 * (U[0][m] * h0 + U[1][m] * h1);  // dL/ds_m^2 times 2 s_m^2 (s = exp(log-scale))
        X[0][m] = d2 * h0;
        X[1][m] = d2 * h1;
    }
    float dR[3][3], dT[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int m = 0; m < 3; ++m) dR[c][m] = T[0][c] * X[0][m] + T[1][c] * X[1][m];
#pragma unroll
        for (int r = 0; r < 2; ++r) dT[r][c] = X[r][0] * R[c][0] + X[r][1] * R[c][1] + X[r][2] * R[c][2];
    }
    const float dw = 2.f * (z * (dR[1][0] - dR[0][1]) + y * (dR[0][2] - dR[2][0]) + x * (dR[2][1] - dR[1][2]));
    const float dx = 2.f * (y * (dR[0][1] + dR[1][0]) + z * (dR[0][2] + dR[2][0]) + w * (dR[2][1] - dR[1][2]) -
                            2.f * x * (dR[1][1] + dR[2][2]));
    const float dy = 2.f * (x * (dR[0][1] + dR[1][0]) + z * (dR[1][2] + dR[2][1]) + w * (dR[0][2] - dR[2][0]) -
                            2.f * y * (dR[0][0] + dR[2][2]));
    const float dz = 2.f * (x * (dR[0][2] + dR[2][0]) + y * (dR[1][2] + dR[2][1]) + w * (dR[1][0] - dR[0][1]) -
                            2.f * z * (dR[0][0] + dR[1][1]));
    const float dot = w * dw + x * dx + y * dy + z * dz;
    dG[3] = (dw - w * dot) * il;
    dG[4] = (dx - x * dot) * il;
    dG[5] = (dy - y * dot) * il;
    dG[6] = (dz - z * dot) * il;
    // mean: through the projection, and through J (a clamped ratio does not move with p_x or p_y)
    const float dj00 = dT[0][0] * W[0][0] + dT[0][1] * W[0][1] + dT[0][2] * W[0][2];
    const float dj02 = dT[0][0] * W[2][0] + dT[0][1] * W[2][1] + dT[0][2] * W[2][2];
    const float dj11 = dT[1][0] * W[1][0] + dT[1][1] * W[1][1] + dT[1][2] * W[1][2];
    const float dj12 = dT[1][0] * W[2][0] + dT[1][1] * W[2][1] + dT[1][2] * W[2][2];
    const float ax = j00 * ipz, ay = j11 * ipz;  // fx / p_z^2, fy / p_z^2
    const float dp0 = du * j00 - (clx ? 0.f : dj02 * ax);
    const float dp1 = dv * j11 - (cly ? 0.f : dj12 * ay);
    const float dp2 = ax * (dj02 * (clx ? rx : 2.f * rx0) - du * p[0] - dj00) +
                      ay * (dj12 * (cly ? ry : 2.f * ry0) - dv * p[1] - dj11);
#pragma unroll
    for (int c = 0; c < 3; ++c) dG[c] = W[0][c] * dp0 + W[1][c] * dp1 + W[2][c] * dp2;
}

// TBN matrix and barycentric point of Gaussian i in one frame (the same definitions as the
// preprocess, fp32 without its fixed rounding order): out[12] as chain() reads it.
__device__ __forceinline__ bool tbn_fast(const ModelInfo &m, const float *__restrict__ verts, int i, float out[12]) {
    const int f = __ldg(m.face_of + i);
    if ((unsigned)f >= (unsigned)m.n_faces) return false;
    const int i0 = __ldg(m.faces + 3 * f), i1 = __ldg(m.faces + 3 * f + 1), i2 = __ldg(m.faces + 3 * f + 2);
    if ((unsigned)i0 >= (unsigned)m.n_verts || (unsigned)i1 >= (unsigned)m.n_verts ||
        (unsigned)i2 >= (unsigned)m.n_verts)
        return false;
    float a[3], b[3], c[3], e1[3], e2[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a[k] = __ldg(verts + 3 * i0 + k);
        b[k] = __ldg(verts + 3 * i1 + k);
        c[k] = __ldg(verts + 3 * i2 + k);
        e1[k] = b[k] - a[k];
        e2[k] = c[k] - a[k];
    }
    const float *uv = m.face_uv + 6 * f;
    const float du1 = __ldg(uv + 2) - __ldg(uv), dv1 = __ldg(uv + 3) - __ldg(uv + 1);
    const float du2 = __ldg(uv + 4) - __ldg(uv), dv2 = __ldg(uv + 5) - __ldg(uv + 1);
    const float rd = __frcp_rn(du1 * dv2 - dv1 * du2);
    const float n0 = e1[1] * e2[2] - e1[2] * e2[1], n1 = e1[2] * e2[0] - e1[0] * e2[2],
                n2 = e1[0] * e2[1] - e1[1] * e2[0];
    const float il = rsqrtf(n0 * n0 + n1 * n1 + n2 * n2);
    const float nn[3] = {n0 * il, n1 * il, n2 * il};
    const float b0 = __ldg(m.bary + i), b1 = __ldg(m.bary + m.n_pad + i), b2 = __ldg(m.bary + 2 * m.n_pad + i);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        out[3 * k] = (dv2 * e1[k] - dv1 * e2[k]) * rd;
        out[3 * k + 1] = (du1 * e2[k] - du2 * e1[k]) * rd;
        out[3 * k + 2] = nn[k];
        out[9 + k] = b0 * a[k] + b1 * b[k] + b2 * c[k];
    }
    return true;
}

// The backward of one model chunk. One CTA = 32 Gaussians (lane = Gaussian) of one model; the
// frames that render it go FG (8 or 16) at a time. The chunk's blendshape rows are copied to shared
// memory asynchronously at the start. Meanwhile the chain rule per (frame, Gaussian) turns the
// 2-D gradients into dL/dG_b over the 14 channels, straight into shared memory (each item
// reads only its cache and 2-D gradients: the cache carries the opacity and whether the
// Gaussian was kept); then the adjoint of Eq. 1 reduces them over the frames: dG0 by plain
// sums, ddG and the dpsi partials as tensor-core products (below).
// Asynchronous 16-byte copy global -> shared (both addresses 16-byte aligned), completed by
// cp.async.wait_all.
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                 :: "r"(static_cast<unsigned>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}

constexpr int kWarps = kBwdThreads / 32;
// Shared-memory strides in floats: a frame's 14 x 32 blended-channel gradients, and a staged
// blendshape row of 32 Gaussians, each padded by 4 so that the tensor-core fragment loads,
// which step over frames or blendshapes, fall in different banks (stride = 4 mod 32).
constexpr int kDGF = kNch * kBwdChunk + 4;
constexpr int kDgRow = kBwdChunk + 4;

// The adjoint of Eq. 1 is two small dense products per chunk and group of FG frames (ddG: the
// K x FG weights times the FG x (A 32) blended-channel gradients; dpsi: the K x (A 32)
// blendshape rows times the (A 32) x FG gradients), done on the tensor cores as
// m16n8k8 TF32 matrix multiply-accumulates with FP32 accumulators. Each FP32 operand x is split
// into x_hi = tf32(x) and x_lo = tf32(x - x_hi), and a b is accumulated as
// a_lo b_hi + a_hi b_lo + a_hi b_hi (the a_lo b_lo term is below FP32 rounding), which keeps
// the products at FP32 accuracy (the split-operand scheme of Ootomo and Yokota, "Recovering
// single precision accuracy from Tensor Cores", 2022). Fragment layout (m16n8k8, A row-major,
// B column-major), with g = lane / 4 and t = lane % 4: A elements (g, t), (g + 8, t), (g, t + 4), (g + 8, t + 4);
// B elements (t, g), (t + 4, g); C elements (g, 2t), (g, 2t + 1), (g + 8, 2t), (g + 8, 2t + 1).
// Blendshapes are the rows of both products and frames come in eights (the n8 columns of one, a
// k8 step of the other), so a group of up to eight frames costs half of one of sixteen.
__device__ __forceinline__ void split_tf32(float x, unsigned &hi, unsigned &lo) {
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hi) : "f"(x));
    const float r = x - __uint_as_float(hi);
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(lo) : "f"(r));
}

__device__ __forceinline__ void mma_tf32(float d[4], const unsigned a[4], const unsigned b[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// d += a b at FP32 accuracy from split operands (small terms first)
__device__ __forceinline__ void mma_3xtf32(float d[4], const unsigned ah[4], const unsigned al[4],
                                           const unsigned bh[2], const unsigned bl[2]) {
    mma_tf32(d, al, bh);
    mma_tf32(d, ah, bl);
    mma_tf32(d, ah, bh);
}

// ADAM: the fused Adam update of rgba_step_adam_async; every model is rendered by at most FG
// frames, so the reductions below are complete after one group. Their results are parked in
// shared memory (G0's in s_g0, the blendshapes' in the slots of the staged rows, whose values
// are read again from memory) and the CTA then streams the update over the chunk's rows; the
// gradient arrays are not written.
// The plain instance's stand-in for FusedAdam: the same members, one model, never read.
struct NoAdam {
    FusedAdamModel m[1];
    float b1, b2, eps, ibc1, ibc2;
    const int *step_dev;
};
template <bool ADAM>
using AdamArg = typename std::conditional<ADAM, FusedAdam, NoAdam>::type;

// BOUND: some model of the batch has a tangent-space binding (the chain rule then maps through
// each bound Gaussian's TBN frame); otherwise that mapping is compiled out.
// FG: frames per group, 8 where every model of the batch is rendered by at most eight, else 16.
// Bound by the latency of its phases (loads, chain rule, two products, stores) at few warps per SM,
// so the shared memory and registers are held to three CTAs per SM where that needs no spills to
// speak of: not for the fused update and the tangent-space mapping with 16 frames, which keep two
// (the mapping: 135 us with two, 147 with three). Measured against 3 x 3 covariances, frames always
// in sixteens and two CTAs per SM: 64 frames of eight avatars of 30,000 to 100,000 Gaussians
// 666 -> 406 us, ten frames of 60,000 (K = 20) 92 -> 74, 16 frames of 60,000 (K = 32) 113 -> 100,
// the same bound to a mesh 145 -> 129. Eights everywhere: 16 frames 143 us, as the blendshape
// gradients are then read back and added to.
template <bool ADAM, bool BOUND, int FG>
__global__ void __launch_bounds__(kBwdThreads, (ADAM || BOUND) && FG == 16 ? 2 : 3)
k_gauss_bwd(Ctx c, int max_k, int max_ka, AdamArg<ADAM> fa) {
    extern __shared__ float smem[];
    float *s_dG = smem;                                   // [FG][kDGF]: [14][32] per frame
    float *s_psi = s_dG + FG * kDGF;                      // [FG][max_k]
    float *s_dgc = s_psi + FG * max_k;                    // [k][A][kDgRow]: the chunk's blendshapes
    __shared__ __align__(16) float s_g0[ADAM ? kNch * kBwdChunk : 1];  // ADAM: the G0 gradients
    __shared__ long long s_rec[FG];
    __shared__ float s_lim[FG][2];
    __shared__ const float *s_verts[FG];
    pdl_enter();
    __shared__ float s_fp[FG][RGBA_FP_STRIDE];
    __shared__ int s_ch[kNch];               // the model's blended channels, by slot
    // dpsi: each warp's sums, [32 blendshapes][FG], in s_dG's place when that is free by then
    const bool alias = !ADAM && max_k <= 32;
    float *s_red = alias ? s_dG : s_dgc + max_ka * kDgRow;
    const ModelInfo &m = c.models[blockIdx.y];
    const int chunk = blockIdx.x;
    const int i0 = chunk * kBwdChunk;
    if (i0 >= m.n_pad || m.nb == 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = i0 + lane;
    const bool in_pad = i < m.n_pad; // row slot (padding slots receive zeros)
    const int K = m.k, A = m.A;
    float ibc1 = 0.f, ibc2 = 0.f;
    if (ADAM) {
        ibc1 = fa.step_dev ? adam_ibc(fa.step_dev, fa.b1) : fa.ibc1;
        ibc2 = fa.step_dev ? adam_ibc(fa.step_dev, fa.b2) : fa.ibc2;
    }
    const FusedAdamModel &am = fa.m[ADAM ? blockIdx.y : 0];
    {  // the chunk's blendshape rows travel to shared memory while the chain rule runs
        const int per_row = min(kBwdChunk, m.n_pad - i0) >> 2;  // n_pad, i0 multiples of 4
        auto copy = [&](int rr, int q) {
            cp_async16(s_dgc + rr * kDgRow + 4 * q, m.dg + (size_t)rr * m.n_pad + i0 + 4 * q);
        };
        if (per_row == kBwdChunk / 4) {  // a full chunk: thread t copies quad t % 8 of every 32nd row
            for (int rr = threadIdx.x / (kBwdChunk / 4); rr < K * A; rr += kBwdThreads / (kBwdChunk / 4))
                copy(rr, threadIdx.x % (kBwdChunk / 4));
        } else {
            for (int e = threadIdx.x; e < K * A * per_row; e += kBwdThreads) copy(e / per_row, e % per_row);
        }
    }
    if (threadIdx.x < A) s_ch[threadIdx.x] = m.chans[threadIdx.x];
    for (int g0 = 0; g0 < m.nb; g0 += FG) {
        const int ng = min(FG, m.nb - g0);
        if (threadIdx.x < ng) {
            const int b = c.mframes[m.frame_off + g0 + threadIdx.x];
            const FrameInfo &f = c.frames[b];
            s_rec[threadIdx.x] = f.rec_base;
            const float *fp = c.fparams + (size_t)b * RGBA_FP_STRIDE;
            s_lim[threadIdx.x][0] = 1.3f * __fdividef(0.5f * f.W, fp[12]);
            s_lim[threadIdx.x][1] = 1.3f * __fdividef(0.5f * f.H, fp[13]);
            s_verts[threadIdx.x] = f.verts;
        }
        for (int e = threadIdx.x; e < ng * RGBA_FP_STRIDE; e += kBwdThreads) {
            const int fl = e / RGBA_FP_STRIDE, q = e - fl * RGBA_FP_STRIDE;
            s_fp[fl][q] = c.fparams[(size_t)c.mframes[m.frame_off + g0 + fl] * RGBA_FP_STRIDE + q];
        }
        for (int e = threadIdx.x; e < FG * max_k; e += kBwdThreads) {
            const int fl = e / max_k, kk = e % max_k;
            s_psi[e] = (fl < ng && kk < K) ? c.psi[(size_t)c.mframes[m.frame_off + g0 + fl] * c.k_stride + kk] : 0.f;
        }
        __syncthreads();
        // dL/dG_b per (frame, Gaussian) of the chunk (zero for culled Gaussians and for frames
        // past the group's end, which the loops below run over too); a warp takes 32
        // consecutive Gaussians of one frame
        {
            constexpr int kItems = FG * kBwdChunk / kBwdThreads;
            float4 c0[kItems], c1[kItems], c2[kItems], ga[kItems], gb[kItems], gc[kItems];
            bool live[kItems];
#pragma unroll
            for (int u = 0; u < kItems; ++u) {  // every load of both items in flight at once
                const int e = threadIdx.x + u * kBwdThreads;
                const int fl = e / kBwdChunk, gi = i0 + (e & (kBwdChunk - 1));
                live[u] = fl < ng && gi < m.n;
                const long long r = live[u] ? s_rec[fl] + gi : 0;
                c0[u] = c1[u] = c2[u] = ga[u] = gb[u] = gc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (live[u]) {
                    c0[u] = c.cache[r * 3 + 0];
                    c1[u] = c.cache[r * 3 + 1];
                    c2[u] = c.cache[r * 3 + 2];  // (log-scale z, -, opacity, kept)
                    const float4 *gp = reinterpret_cast<const float4 *>(c.grad2d + r * kG2Floats);
                    ga[u] = gp[0];
                    gb[u] = gp[1];
                    gc[u] = gp[2];
                }
            }
#pragma unroll 1
            for (int u = 0; u < kItems; ++u) {
                const int e = threadIdx.x + u * kBwdThreads;
                const int fl = e / kBwdChunk, li = e & (kBwdChunk - 1);
                float dG[kNch];
#pragma unroll
                for (int q = 0; q < kNch; ++q) dG[q] = 0.f;
                if (live[0] && c2[0].w != 0.f) {  // item u sits in slot 0 (a rolled loop keeps the code small)
                    const float v[10] = {c0[0].x, c0[0].y, c0[0].z, c0[0].w, c1[0].x, c1[0].y, c1[0].z, c1[0].w, c2[0].x, c2[0].y};
                    const float g2[9] = {ga[0].x, ga[0].y, ga[0].z, ga[0].w, gb[0].x, gb[0].y, gb[0].z, gb[0].w, gc[0].x};
                    if (BOUND) {
                        float Rt[12] = {1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f};
                        if (m.n_faces == 0 || tbn_fast(m, s_verts[fl], i0 + li, Rt))
                            chain<true>(v, c2[0].z, s_fp[fl], s_lim[fl], Rt, g2, dG);
                    } else {
                        chain<false>(v, c2[0].z, s_fp[fl], s_lim[fl], nullptr, g2, dG);
                    }
                }
#pragma unroll
                for (int q = 0; q < kNch; ++q) s_dG[fl * kDGF + q * kBwdChunk + li] = dG[q];
                if (c.grad_blended && fl < ng && i0 + li < m.n_pad) {  // rgba_render_bwd's optional output
                    float *o = c.grad_blended + s_rec[fl] * kNch + i0 + li;
#pragma unroll
                    for (int q = 0; q < kNch; ++q) o[(size_t)q * m.n_pad] = dG[q];
                }
#pragma unroll
                for (int w = 0; w + 1 < kItems; ++w) {
                    c0[w] = c0[w + 1];
                    c1[w] = c1[w + 1];
                    c2[w] = c2[w + 1];
                    ga[w] = ga[w + 1];
                    gb[w] = gb[w + 1];
                    gc[w] = gc[w + 1];
                    live[w] = live[w + 1];
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // dG0[ch][i] = sum_b dG_b[ch][i]
        if ((ADAM ? am.p0 != nullptr : m.gg0 != nullptr) && in_pad) {
            for (int ch = warp; ch < kNch; ch += kWarps) {
                float a = 0.f;
                for (int fl = 0; fl < ng; ++fl) a += s_dG[fl * kDGF + ch * kBwdChunk + lane];
                const size_t o = (size_t)ch * m.n_pad + i;
                if (ADAM) {  // parked for the update below, exactly as the separate update reads it
                    s_g0[ch * kBwdChunk + lane] = 0.f + a;
                } else {
                    m.gg0[o] = (g0 == 0 ? 0.f : m.gg0[o]) + a;
                }
            }
        }
        const int grp = lane >> 2, tig = lane & 3;
        // dpsi_b[k] partial = sum over a, i of dG_k[a][i] dG_b[ch_a][i]: D (k x frames) =
        // A (k x columns) B (columns x frames), a column being (channel slot a, Gaussian i) and
        // 8 columns one k-step; the warps split the k-steps, their sums meet in s_red
        auto weight_grads = [&]() {
            if (!c.grad_psi) return;
            const int KS = A * (kBwdChunk / 8);
            for (int kb = 0; kb < K; kb += 32) {
                float acc[2][FG / 8][4];
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int n = 0; n < FG / 8; ++n) acc[j][n][0] = acc[j][n][1] = acc[j][n][2] = acc[j][n][3] = 0.f;
                for (int ks = warp; ks < KS; ks += kWarps) {
                    const int sa = ks / (kBwdChunk / 8), ib = (ks % (kBwdChunk / 8)) * 8;
                    const float *dg = s_dG + s_ch[sa] * kBwdChunk + ib + tig + grp * kDGF;
                    unsigned bh[FG / 8][2], bl[FG / 8][2];
#pragma unroll
                    for (int n = 0; n < FG / 8; ++n) {
                        split_tf32(dg[n * 8 * kDGF], bh[n][0], bl[n][0]);
                        split_tf32(dg[n * 8 * kDGF + 4], bh[n][1], bl[n][1]);
                    }
                    // padding columns hold whatever the caller left there: zero them
                    const bool v0 = i0 + ib + tig < m.n, v1 = i0 + ib + tig + 4 < m.n;
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int k0 = kb + j * 16 + grp, k1 = k0 + 8;
                        const float *as = s_dgc + (k0 * A + sa) * kDgRow + ib + tig, *bs = as + 8 * A * kDgRow;
                        unsigned ah[4], al[4];
                        split_tf32(k0 < K && v0 ? as[0] : 0.f, ah[0], al[0]);
                        split_tf32(k1 < K && v0 ? bs[0] : 0.f, ah[1], al[1]);
                        split_tf32(k0 < K && v1 ? as[4] : 0.f, ah[2], al[2]);
                        split_tf32(k1 < K && v1 ? bs[4] : 0.f, ah[3], al[3]);
#pragma unroll
                        for (int n = 0; n < FG / 8; ++n) mma_3xtf32(acc[j][n], ah, al, bh[n], bl[n]);
                    }
                }
                if (alias) __syncthreads();  // the sums take the place of s_dG, which nobody reads any more
#pragma unroll
                for (int j = 0; j < 2; ++j)  // this warp's sums, then the warps' in a fixed order
#pragma unroll
                    for (int n = 0; n < FG / 8; ++n) {
                        float *r = s_red + warp * (32 * FG) + (j * 16 + grp) * FG + n * 8 + 2 * tig;
                        *reinterpret_cast<float2 *>(r) = make_float2(acc[j][n][0], acc[j][n][1]);
                        *reinterpret_cast<float2 *>(r + 8 * FG) = make_float2(acc[j][n][2], acc[j][n][3]);
                    }
                __syncthreads();
                for (int e = threadIdx.x; e < 32 * FG; e += kBwdThreads) {
                    const int kk = kb + e / FG, fl = e % FG;
                    float t = 0.f;
#pragma unroll
                    for (int w = 0; w < kWarps; ++w) t += s_red[w * (32 * FG) + e];
                    if (fl < ng && kk < K)
                        c.dpsi_part[m.dpsi_off + ((long long)(g0 + fl) * K + kk) * m.n_chunks + chunk] = t;
                }
                __syncthreads();
            }
        };
        // ddG[k][a][i] = sum_b psi_b[k] dG_b[ch_a][i]: D (k x columns) = A (k x frames)
        // B (frames x columns), a k-step per 8 frames; the warps split the 8-column tiles and a
        // tile's split gradients serve 32 blendshapes
        auto basis_grads = [&]() {
            if (!ADAM && m.gdg == nullptr) return;
            const int NT = A * (kBwdChunk / 8);
            for (int kb = 0; kb < K; kb += 32) {
                unsigned ah[2][FG / 8][4], al[2][FG / 8][4];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int k0 = kb + j * 16 + grp, k1 = k0 + 8;
#pragma unroll
                    for (int q = 0; q < FG / 8; ++q) {
                        const int f0 = q * 8 + tig, f1 = f0 + 4;
                        split_tf32(k0 < K ? s_psi[f0 * max_k + k0] : 0.f, ah[j][q][0], al[j][q][0]);
                        split_tf32(k1 < K ? s_psi[f0 * max_k + k1] : 0.f, ah[j][q][1], al[j][q][1]);
                        split_tf32(k0 < K ? s_psi[f1 * max_k + k0] : 0.f, ah[j][q][2], al[j][q][2]);
                        split_tf32(k1 < K ? s_psi[f1 * max_k + k1] : 0.f, ah[j][q][3], al[j][q][3]);
                    }
                }
                for (int nt = warp; nt < NT; nt += kWarps) {
                    const int sa = nt / (kBwdChunk / 8), ib = (nt % (kBwdChunk / 8)) * 8;
                    const float *dg = s_dG + s_ch[sa] * kBwdChunk + ib + grp;
                    unsigned bh[FG / 8][2], bl[FG / 8][2];
#pragma unroll
                    for (int q = 0; q < FG / 8; ++q) {
                        split_tf32(dg[(q * 8 + tig) * kDGF], bh[q][0], bl[q][0]);
                        split_tf32(dg[(q * 8 + tig + 4) * kDGF], bh[q][1], bl[q][1]);
                    }
                    const int i = ib + 2 * tig;  // columns i, i + 1 of the rows k0 and k1
                    float *o0 = ADAM ? nullptr : m.gdg + (size_t)((kb + grp) * A + sa) * m.n_pad + i0 + i;
                    const size_t step = (size_t)8 * A * m.n_pad;  // eight blendshapes on
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int q = 0; q < FG / 8; ++q) mma_3xtf32(d, ah[j][q], al[j][q], bh[q], bl[q]);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int kk = kb + j * 16 + 8 * h + grp;
                            if (kk >= K) continue;
                            if (ADAM) {  // s_dgc is no longer read (dpsi is done): its slots park the gradients
                                float *o = s_dgc + (kk * A + sa) * kDgRow + i;
                                o[0] = 0.f + d[2 * h];
                                o[1] = 0.f + d[2 * h + 1];
                            } else if (i0 + i < m.n_pad) {  // n_pad - i0 is a multiple of 4: i + 1 too
                                float2 *o = reinterpret_cast<float2 *>(o0 + (2 * j + h) * step);
                                const float2 old = g0 == 0 ? make_float2(0.f, 0.f) : *o;
                                *o = make_float2(old.x + d[2 * h], old.y + d[2 * h + 1]);
                            }
                        }
                    }
                }
            }
        };
        if (ADAM) {  // the blendshape gradients are parked in the rows that the weight gradients read
            weight_grads();
            basis_grads();
        } else {
            basis_grads();
            weight_grads();
        }
        __syncthreads();
    }
    if (ADAM) {
        // the update, streamed over the chunk's rows (G0 rows, then blendshape rows) by the whole
        // CTA, float4 by float4, with the loads of several float4s in flight per thread
        const int cols4 = min(kBwdChunk, m.n_pad - i0) >> 2;
        const int rows0 = am.p0 ? kNch : 0, rowsd = am.pd ? K * A : 0;
        const int total = (rows0 + rowsd) * cols4;
        constexpr int kU = 4;
        for (int e0 = threadIdx.x; e0 < total; e0 += kU * kBwdThreads) {
            float4 pp[kU], mm[kU], vv[kU];
            int rows[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {  // every load first
                const int e = e0 + u * kBwdThreads;
                rows[u] = e < total ? e / cols4 : -1;
                if (rows[u] >= 0) {
                    const int row = rows[u], c4 = e - row * cols4;
                    const bool base = row < rows0;
                    const size_t off = (size_t)(base ? row : row - rows0) * m.n_pad + i0 + 4 * c4;
                    pp[u] = *reinterpret_cast<const float4 *>((base ? am.p0 : am.pd) + off);
                    mm[u] = *reinterpret_cast<const float4 *>((base ? am.m0 : am.md) + off);
                    vv[u] = *reinterpret_cast<const float4 *>((base ? am.v0 : am.vd) + off);
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (rows[u] < 0) continue;
                const int e = e0 + u * kBwdThreads, row = rows[u], c4 = e - row * cols4;
                const bool base = row < rows0;
                const int rr = base ? row : row - rows0;
                const size_t off = (size_t)rr * m.n_pad + i0 + 4 * c4;
                const float4 g = *reinterpret_cast<const float4 *>((base ? s_g0 + rr * kBwdChunk : s_dgc + rr * kDgRow) + 4 * c4);
                const float lr = base ? am.lr0[rr] : am.lrd[rr % A];
                float p4[4] = {pp[u].x, pp[u].y, pp[u].z, pp[u].w}, m4[4] = {mm[u].x, mm[u].y, mm[u].z, mm[u].w},
                      v4[4] = {vv[u].x, vv[u].y, vv[u].z, vv[u].w};
                const float g4[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) adam_update(p4[q], g4[q], m4[q], v4[q], lr, fa.b1, fa.b2, fa.eps, ibc1, ibc2);
                *reinterpret_cast<float4 *>((base ? am.p0 : am.pd) + off) = make_float4(p4[0], p4[1], p4[2], p4[3]);
                *reinterpret_cast<float4 *>((base ? am.m0 : am.md) + off) = make_float4(m4[0], m4[1], m4[2], m4[3]);
                *reinterpret_cast<float4 *>((base ? am.v0 : am.vd) + off) = make_float4(v4[0], v4[1], v4[2], v4[3]);
            }
        }
    }
}

// dpsi[b][k] = sum over chunks of the partials; zero for k >= the model's k.
constexpr int kDpsiThreads = 256;

// One CTA per (blendshape k, frame b): the CTA's threads stride over the chunk partials, then
// a warp-shuffle and shared-memory sum.
__global__ void __launch_bounds__(kDpsiThreads) k_dpsi_reduce(Ctx c) {
    __shared__ float s_w[kDpsiThreads / 32];
    pdl_enter();
    const int kk = blockIdx.x, b = blockIdx.y;
    const FrameInfo &f = c.frames[b];
    const ModelInfo &m = c.models[f.model];
    float s = 0.f;
    if (kk < m.k) {
        // position of frame b in its model's frame list
        int j = 0;
        for (int q = 0; q < m.nb; ++q)
            if (c.mframes[m.frame_off + q] == b) j = q;
        const float *p = c.dpsi_part + m.dpsi_off + ((long long)j * m.k + kk) * m.n_chunks;
        for (int q = threadIdx.x; q < m.n_chunks; q += kDpsiThreads) s += p[q];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < kDpsiThreads / 32; ++w) t += s_w[w];
        c.grad_psi[(size_t)b * c.k_stride + kk] = t;
    }
}

}  // namespace

namespace {
template <bool ADAM, bool BOUND, int FG>
cudaError_t gauss_bwd_inst(const Ctx &c, int max_chunks, int max_k, int max_ka, const AdamArg<ADAM> &fa,
                           cudaStream_t s) {
    auto bytes = [](int k, int ka) {
        const int red = ADAM || k > 32 ? kWarps * 32 * FG : 0;  // as in the kernel
        return (FG * kDGF + FG * k + ka * kDgRow + red) * (int)sizeof(float);
    };
    // set once, at the largest size any batch can ask for, so no attribute call happens while
    // a stream is being captured
    static int attr_device = -1;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (attr_device != dev) {
        e = cudaFuncSetAttribute(k_gauss_bwd<ADAM, BOUND, FG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 bytes(RGBA_MAX_K, RGBA_MAX_K * 13));
        if (e != cudaSuccess) return e;
        attr_device = dev;
    }
    dim3 g2(max_chunks, c.M);
    return launch_pdl(k_gauss_bwd<ADAM, BOUND, FG>, g2, dim3(kBwdThreads), (size_t)bytes(max_k, max_ka), s, c, max_k,
                      max_ka, fa);
}

template <bool ADAM, bool BOUND>
cudaError_t gauss_bwd_frames(const Ctx &c, int max_chunks, int max_nb, int max_k, int max_ka, const AdamArg<ADAM> &fa,
                             cudaStream_t s) {
    return max_nb <= 8 ? gauss_bwd_inst<ADAM, BOUND, 8>(c, max_chunks, max_k, max_ka, fa, s)
                       : gauss_bwd_inst<ADAM, BOUND, 16>(c, max_chunks, max_k, max_ka, fa, s);
}
}  // namespace

cudaError_t launch_gauss_bwd(const Ctx &c, int max_chunks, int max_nb, int max_k, int max_ka, const FusedAdam *fa,
                             bool any_bound, cudaStream_t s) {
    if (c.M == 0 || max_chunks == 0) return cudaSuccess;
    if (fa)
        return any_bound ? gauss_bwd_frames<true, true>(c, max_chunks, max_nb, max_k, max_ka, *fa, s)
                         : gauss_bwd_frames<true, false>(c, max_chunks, max_nb, max_k, max_ka, *fa, s);
    const NoAdam none{};
    return any_bound ? gauss_bwd_frames<false, true>(c, max_chunks, max_nb, max_k, max_ka, none, s)
                     : gauss_bwd_frames<false, false>(c, max_chunks, max_nb, max_k, max_ka, none, s);
}

cudaError_t launch_dpsi_reduce(const Ctx &c, int max_k, cudaStream_t s) {
    (void)max_k;
    if (!c.grad_psi || c.B == 0 || c.k_stride == 0) return cudaSuccess;
    return launch_pdl(k_dpsi_reduce, dim3(c.k_stride, c.B), dim3(kDpsiThreads), 0, s, c);
}

}  // namespace rgba
