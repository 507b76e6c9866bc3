// loss_ssim.cu -- fused gradient of the weighted L1 + SSIM loss on
// channel-last renders with an 8-bit RGBA reference (VkSplat Sec. 4.5).
//
//   L = (1 - lam) mean|x - y| + lam (1 - mean SSIM),
// SSIM per channel with an 11x11 Gaussian window (sigma 1.5), zero padding,
// C1 = 0.01^2, C2 = 0.03^2, means over 3 x all pixels of all views.
//
// With the window moments mu_x, mu_y, E[x^2], E[y^2], E[xy] at q,
//   dSSIM_sum / dx_p = (w * A)(p) + 2 x_p (w * B)(p) + y_p (w * Cc)(p),
// A = dSSIM/dmu_x, B = dSSIM/dE[x^2], Cc = dSSIM/dE[xy] at each q (the window
// is symmetric).  A CTA takes one or two tiles of a view and colour channel: x and y
// are staged with a 10-pixel halo, separable 11-tap passes give the five moments at
// the positions whose windows reach the tile, then A, B, Cc there, and two more
// separable passes give the gradient at the tile's pixels -- one kernel, no
// intermediate image in global memory, no layout conversion.
//
// The moments are taken about a per-tile shift (x and y at the tile's centre
// pixel): variances and the covariance are shift-invariant, and with values
// near the local mean E[x^2] - mu_x^2 no longer cancels in FP32 on flat
// image regions.  Zero padding becomes padding with -shift.
//
// Issue- and FP32-bound (68% of issue slots, 2.8 IPC).  Every pass is register-blocked
// along its window: a thread reads the 11 + n - 1 values of n neighbouring outputs once
// instead of 11 values an output.  Moments and partials are packed pairs (FFMA2).  The
// three channels of a tile are neighbouring CTAs, so that small images fill the chip and
// the channels' accesses to one pixel meet in L2.  All staging loads of a thread are in
// flight together (four rows at a time took a third longer).  Against one output a
// thread in 16x16 tiles of all channels, four 1080p views and 403x301:
//  - SsimWide, 32x31 tiles: 1.43 -> 0.56 ms, 33 -> 15 us; about 400 FP32 operations a
//    pixel and channel with the halos.  The height 31 gives each pass just under 256
//    tasks, one per thread (51 rows x 5 groups, 42 columns x 6, 41 rows x 6, 32 x 8).
//  - SsimExact, 16x16 tiles, two to a CTA: 1.43 -> 0.94 ms, 33 -> 22 us; half as many
//    operations again in the halos, and divisions instead of one reciprocal (0.08 ms),
//    for the bits of 16x16 tiles.  The tile's shift enters every rounding, so another
//    tiling differs by 6e-7 of the gradient.  That is the kernel's own error, but the
//    projection backward of needle-shaped Gaussians multiplies it by a thousand, beyond
//    what two runs of an FP32 optimisation may differ by; with BF16 moments their stored
//    rounding (4e-3) hides it.  Hence the rule: BF16 moments take SsimWide.
#include "raster_blocks.cuh"

namespace gs {

constexpr int kSsR = 5;                    // window radius
// The two forms of the kernel: tile, tiles side by side per CTA, outputs per thread of
// the four passes (kN1 to kN4), threads, CTAs per SM, threads per staged row; then the
// shared-memory pitches.
struct SsimWide {
    static constexpr int kW = 32, kH = 31, kP = 1, kN1 = 9, kN2 = 7, kN3 = 6, kN4 = 4;
    static constexpr int kThreads = 256, kCtas = 3, kRow = 64;
    static constexpr int kPx = 55, kPm = 43, kPa = 47, kPh = 33;
    static constexpr bool kExact = false;
};
struct SsimExact {
    static constexpr int kW = 16, kH = 16, kP = 2, kN1 = 9, kN2 = 7, kN3 = 4, kN4 = 3;
    static constexpr int kThreads = 224, kCtas = 4, kRow = 56;
    static constexpr int kPx = 53, kPm = 27, kPa = 27, kPh = 17;
    static constexpr bool kExact = true;
};
template <typename F>
struct SsimGeo {
    static constexpr int kQw = F::kW + 2 * kSsR, kQh = F::kH + 2 * kSsR;     // positions whose window reaches a tile
    static constexpr int kXw = F::kP * F::kW + 4 * kSsR, kXh = F::kH + 4 * kSsR;   // staged pixels
    static constexpr int kG1 = (kQw + F::kN1 - 1) / F::kN1, kG2 = (kQh + F::kN2 - 1) / F::kN2;
    static constexpr int kG3 = (F::kW + F::kN3 - 1) / F::kN3, kG4 = (F::kH + F::kN4 - 1) / F::kN4;
    static_assert(F::kP * kXh * kG1 <= F::kThreads && F::kP * kQw * kG2 <= F::kThreads &&
                      F::kP * kQh * kG3 <= F::kThreads && F::kP * F::kW * kG4 <= F::kThreads,
                  "one task per thread in every pass");
    static constexpr int kOver = kG2 * F::kN2 + 2 * kSsR - kXh;   // rows read past the end
    static_assert(F::kPx >= F::kP * F::kW - F::kW + kG1 * F::kN1 + 2 * kSsR && kOver >= 0, "what the last groups read");
    // Pitches odd in the unit read across rows (no bank conflicts).  The outputs past
    // the edge that a last group computes and drops read what follows in shared memory.
    struct Smem {
        union {
            float2 xy[kXh][F::kPx];                // (x, y)
            struct {
                float2 ab[F::kP][kQh][F::kPa];     // (A, B)
                float c[F::kP][kQh][F::kPa];       // Cc
            } abc;
        };
        union {
            struct {
                float4 m03[F::kP][kXh][F::kPm];    // (mu_x, mu_y, E[x^2], E[y^2]) of the rows
                float m4[F::kP][kXh][F::kPm];      // E[xy]
                float past[kOver * F::kPm + 1];
            } h;
            struct {
                float2 ab[F::kP][kQh][F::kPh];
                float c[F::kP][kQh][F::kPh];
            } habc;
        };
    };
};
constexpr float kSsC1 = 0.01f * 0.01f;

// Window tap k (0..10): exp(-(k - 5)^2 / (2 * 1.5^2)) normalised to unit sum,
// evaluated in FP64 and rounded to FP32; with unrolled tap loops these become
// immediate operands of the FMAs.
__host__ __device__ constexpr float ssim_w(int k)
{
    return (k == 0 || k == 10) ? 0.0010283801f
         : (k == 1 || k == 9)  ? 0.0075987582f
         : (k == 2 || k == 8)  ? 0.036000773f
         : (k == 3 || k == 7)  ? 0.10936069f
         : (k == 4 || k == 6)  ? 0.21300554f
                               : 0.26601171f;
}
constexpr float kSsC2 = 0.03f * 0.03f;

template <typename F>
__host__ __device__ __forceinline__ int64_t ssim_tiles(const ViewDesc& vd)
{
    return (int64_t)((vd.W + F::kP * F::kW - 1) / (F::kP * F::kW)) * ((vd.H + F::kH - 1) / F::kH);
}

template <typename F>
__device__ __forceinline__ int ssim_view_of_tile(const Views& V, int64_t t, int64_t& first)
{
    int64_t base = 0;
    for (int v = 0; v < V.n; v++) {
        const int64_t nt = ssim_tiles<F>(V.v[v]);
        if (t < base + nt || v == V.n - 1) {
            first = base;
            return v;
        }
        base += nt;
    }
    first = 0;
    return 0;
}

__device__ __forceinline__ float target_code(uchar4 t, int c)
{
    return (float)(c == 0 ? t.x : (c == 1 ? t.y : t.z));
}

__device__ __forceinline__ float target_channel(uchar4 t, int c)
{
    return target_code(t, c) * (1.0f / 255.0f);
}

// Alpha masking (MASK): the loss is taken on the render and the reference
// both multiplied by the reference's alpha m = A / 255, so masked-out pixels
// add nothing; the gradient with respect to the render carries the factor m.
template <bool MASK>
__device__ __forceinline__ float pix_mask(uchar4 t)
{
    return MASK ? (float)t.w * (1.0f / 255.0f) : 1.0f;
}

template <bool MASK, typename F>
__global__ void __launch_bounds__(F::kThreads, F::kCtas)
    k_loss_l1_ssim(Views V, const float* __restrict__ image, const uchar4* __restrict__ target, float lam, float inv_n,
                   float* __restrict__ dl, float* __restrict__ part, WsHeader* __restrict__ hdr)
{
    if (!after_previous()) return;
    using G = SsimGeo<F>;
    constexpr int kSsP = F::kP, kSsThreads = F::kThreads;
    constexpr int kQw = G::kQw, kQh = G::kQh, kXw = G::kXw, kXh = G::kXh;
    constexpr int kN1 = F::kN1, kN2 = F::kN2, kN3 = F::kN3, kN4 = F::kN4;
    constexpr int kG1 = G::kG1, kG2 = G::kG2, kG3 = G::kG3, kG4 = G::kG4;
    constexpr int kPm = F::kPm, kPh = F::kPh;
    extern __shared__ __align__(16) unsigned char ssim_smem[];
    typename G::Smem& sm = *reinterpret_cast<typename G::Smem*>(ssim_smem);
    __shared__ float red[2][kSsThreads / 32];
    __shared__ float2 shift[kSsP];
    __shared__ bool is_last;

    const int tid = threadIdx.x;
    int64_t first;
    const int c = (int)(blockIdx.x % 3u);        // colour channel
    const int64_t tile = blockIdx.x / 3u;
    const int v = ssim_view_of_tile<F>(V, tile, first);
    const ViewDesc& vd = V.v[v];
    const int lt = (int)(tile - first);
    const int TX = (vd.W + kSsP * F::kW - 1) / (kSsP * F::kW);
    const int ox = (lt % TX) * (kSsP * F::kW), oy = (lt / TX) * F::kH;
    float l1 = 0.f, ss = 0.f;

    // The tiles' shifts, their centre pixels, and the staged pixels: all loads of a
    // thread are in flight together (one memory round trip a tile).  A CTA of one tile
    // subtracts its shift here, otherwise the first pass does.
    // (a non-finite centre pixel shifts by nothing: it reaches only its own windows)
    const int sp = kSsP == 1 ? 0 : min(tid, kSsP - 1);
    const int64_t cpix = vd.pix_base + (int64_t)min(oy + F::kH / 2, vd.H - 1) * vd.W +
                         min(ox + F::kW * sp + F::kW / 2, vd.W - 1);
    const uchar4 tc = target[cpix];
    const float ic = image[3 * cpix + c];
    float2 own;      // the shift; its y a code where the target's scale enters unrounded
    constexpr float kYs = MASK || !F::kExact ? 1.0f : 1.0f / 255.0f;
    {
        // F::kRow threads a row, so that no index is divided
        constexpr int RS = kSsThreads / F::kRow, NR = (kXh + RS - 1) / RS;
        static_assert(kSsThreads % F::kRow == 0 && kXw <= F::kRow, "whole rows");
        const int col = tid % F::kRow, r0 = tid / F::kRow, x = ox - 2 * kSsR + col;
        const bool xin = col < kXw && x >= 0 && x < vd.W;
        const int64_t pix0 = vd.pix_base + (int64_t)(oy - 2 * kSsR + r0) * vd.W + x;
        float xi[NR];
        uchar4 ti[NR];
#pragma unroll
        for (int k = 0; k < NR; k++) {
            const int r = r0 + RS * k, y = oy - 2 * kSsR + r;
            xi[k] = 0.f;
            ti[k] = make_uchar4(0, 0, 0, 0);
            if (xin && r < kXh && y >= 0 && y < vd.H) {
                const int64_t pix = pix0 + (int64_t)(RS * k) * vd.W;
                xi[k] = image[3 * pix + c];
                ti[k] = target[pix];
            }
        }
        const float mc = pix_mask<MASK>(tc);
        own.x = isfinite(ic * mc) ? ic * mc : 0.f;
        own.y = MASK || !F::kExact ? target_channel(tc, c) * mc : target_code(tc, c);
        if (kSsP > 1 && tid < kSsP) shift[tid] = own;
#pragma unroll
        for (int k = 0; k < NR; k++) {
            const int r = r0 + RS * k;
            const float m = pix_mask<MASK>(ti[k]);
            if (col < kXw && r < kXh)
                sm.xy[r][col] = kSsP > 1 ? make_float2(xi[k] * m, target_channel(ti[k], c) * m)
                                         : make_float2(xi[k] * m - own.x, target_channel(ti[k], c) * m - own.y);
        }
    }
    __syncthreads();
    // horizontal pass: 5 moments at the staged rows and the windows' columns of each tile
    if (tid < kSsP * kXh * kG1) {
        const int p = kSsP == 1 ? 0 : tid / (kXh * kG1), i = kSsP == 1 ? tid : tid % (kXh * kG1);
        const int r = i % kXh, q0 = (i / kXh) * kN1;
        const float2 s2 = kSsP == 1 ? own : shift[p], sh = f2(-s2.x, -s2.y), sf = f2(1.f, kYs);
        const float2* row = sm.xy[r] + F::kW * p + q0;
        float2 m01[kN1], m23[kN1];
        float m4[kN1];
#pragma unroll
        for (int o = 0; o < kN1; o++) {
            m01[o] = m23[o] = make_float2(0.f, 0.f);
            m4[o] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < kN1 + 2 * kSsR; j++) {
            const float2 xy = kSsP == 1 ? row[j] : fma2(sh, sf, row[j]);
            const float2 sq = mul2(xy, xy);
            const float pr = xy.x * xy.y;
#pragma unroll
            for (int o = 0; o < kN1; o++) {
                if (j - o < 0 || j - o > 2 * kSsR) continue;
                const float w = ssim_w(j - o);
                m01[o] = fma2(f2(w, w), xy, m01[o]);
                m23[o] = fma2(f2(w, w), sq, m23[o]);
                m4[o] = fmaf(w, pr, m4[o]);
            }
        }
#pragma unroll
        for (int o = 0; o < kN1; o++) {
            if (q0 + o >= kQw) break;
            sm.h.m03[p][r][q0 + o] = make_float4(m01[o].x, m01[o].y, m23[o].x, m23[o].y);
            sm.h.m4[p][r][q0 + o] = m4[o];
        }
    }
    __syncthreads();
    // vertical pass, SSIM and its partials at the windows' positions
    if (tid < kSsP * kQw * kG2) {
        const int p = kSsP == 1 ? 0 : tid / (kQw * kG2), i = kSsP == 1 ? tid : tid % (kQw * kG2);
        const int qc = i % kQw, r0 = (i / kQw) * kN2;
        const float2 sh = kSsP == 1 ? own : shift[p];
        const float4* h03 = &sm.h.m03[p][r0][qc];
        const float* h4 = &sm.h.m4[p][r0][qc];
        float2 m01[kN2], m23[kN2];
        float m4[kN2];
#pragma unroll
        for (int o = 0; o < kN2; o++) {
            m01[o] = m23[o] = make_float2(0.f, 0.f);
            m4[o] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < kN2 + 2 * kSsR; j++) {
            const float4 a = h03[j * kPm];
            const float e = h4[j * kPm];
#pragma unroll
            for (int o = 0; o < kN2; o++) {
                if (j - o < 0 || j - o > 2 * kSsR) continue;
                const float w = ssim_w(j - o);
                m01[o] = fma2(f2(w, w), f2(a.x, a.y), m01[o]);
                m23[o] = fma2(f2(w, w), f2(a.z, a.w), m23[o]);
                m4[o] = fmaf(w, e, m4[o]);
            }
        }
        const int x = ox + F::kW * p - kSsR + qc;
#pragma unroll
        for (int o = 0; o < kN2; o++) {
            const int qr = r0 + o, y = oy - kSsR + qr;
            if (qr >= kQh) break;
            float A = 0.f, B = 0.f, Cc = 0.f;
            if (x >= 0 && y >= 0 && x < vd.W && y < vd.H) {
                const float m[5] = {m01[o].x, m01[o].y, m23[o].x, m23[o].y, m4[o]};
                const float mx = m[0] + sh.x, my = fmaf(sh.y, kYs, m[1]);
                const float vx = m[2] - m[0] * m[0], vy = m[3] - m[1] * m[1], cxy = m[4] - m[0] * m[1];
                const float a1 = 2.f * mx * my + kSsC1, a2 = 2.f * cxy + kSsC2;
                const float b1 = mx * mx + my * my + kSsC1, b2 = vx + vy + kSsC2;
                float s;
                if constexpr (F::kExact) {
                    const float ib = 1.0f / (b1 * b2);
                    s = a1 * a2 * ib;
                    A = 2.f * my * (a2 - a1) * ib - 2.f * mx * s / b1 + 2.f * mx * s / b2;
                    B = -s / b2;
                    Cc = 2.f * a1 * ib;
                } else {
                    // one hardware reciprocal (an ulp): 1 / b1 = b2 ib, 1 / b2 = b1 ib
                    const float ib = __fdividef(1.0f, b1 * b2), ib2 = b1 * ib;
                    s = a1 * a2 * ib;
                    A = 2.f * (my * (a2 - a1) * ib + mx * s * (ib2 - b2 * ib));
                    B = -s * ib2;
                    Cc = 2.f * a1 * ib;
                }
                if (qr >= kSsR && qr < kSsR + F::kH && qc >= kSsR && qc < kSsR + F::kW) ss += s;
            }
            sm.abc.ab[p][qr][qc] = make_float2(A, B);
            sm.abc.c[p][qr][qc] = Cc;
        }
    }
    __syncthreads();
    // the tiles' own pixels, requested before the last two passes need them
    const int p4 = kSsP == 1 ? 0 : tid / (F::kW * kG4), pc = tid % F::kW, pr0 = (tid % (F::kW * kG4)) / F::kW * kN4;
    const int px = ox + F::kW * p4 + pc;
    float ox4[kN4];
    uchar4 ot4[kN4];
#pragma unroll
    for (int o = 0; o < kN4; o++) {
        const int py = oy + pr0 + o;
        ox4[o] = 0.f;
        ot4[o] = make_uchar4(0, 0, 0, 0);
        if (p4 < kSsP && pr0 + o < F::kH && px < vd.W && py < vd.H) {
            const int64_t ppix = vd.pix_base + (int64_t)py * vd.W + px;
            ox4[o] = image[3 * ppix + c];
            ot4[o] = target[ppix];
        }
    }
    // horizontal pass of A, B, Cc at the tiles' columns
    if (tid < kSsP * kQh * kG3) {
        const int p = kSsP == 1 ? 0 : tid / (kQh * kG3), i = kSsP == 1 ? tid : tid % (kQh * kG3);
        const int r = i % kQh, q0 = (i / kQh) * kN3;
        const float2* rab = &sm.abc.ab[p][r][q0];
        const float* rc = &sm.abc.c[p][r][q0];
        float2 ab[kN3];
        float d[kN3];
#pragma unroll
        for (int o = 0; o < kN3; o++) {
            ab[o] = make_float2(0.f, 0.f);
            d[o] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < kN3 + 2 * kSsR; j++) {
            const float2 a = rab[j];
            const float e = rc[j];
#pragma unroll
            for (int o = 0; o < kN3; o++) {
                if (j - o < 0 || j - o > 2 * kSsR) continue;
                const float w = ssim_w(j - o);
                ab[o] = fma2(f2(w, w), a, ab[o]);
                d[o] = fmaf(w, e, d[o]);
            }
        }
#pragma unroll
        for (int o = 0; o < kN3; o++)
            if (q0 + o < F::kW) {
                sm.habc.ab[p][r][q0 + o] = ab[o];
                sm.habc.c[p][r][q0 + o] = d[o];
            }
    }
    __syncthreads();
    // vertical pass at the tiles' pixels; combine with the L1 term
    if (p4 < kSsP) {
        const float2* cab = &sm.habc.ab[p4][pr0][pc];
        const float* cc = &sm.habc.c[p4][pr0][pc];
        float2 ab[kN4];
        float d[kN4];
#pragma unroll
        for (int o = 0; o < kN4; o++) {
            ab[o] = make_float2(0.f, 0.f);
            d[o] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < kN4 + 2 * kSsR; j++) {
            const float2 a = cab[j * kPh];
            const float e = cc[j * kPh];
#pragma unroll
            for (int o = 0; o < kN4; o++) {
                if (j - o < 0 || j - o > 2 * kSsR) continue;
                const float w = ssim_w(j - o);
                ab[o] = fma2(f2(w, w), a, ab[o]);
                d[o] = fmaf(w, e, d[o]);
            }
        }
#pragma unroll
        for (int o = 0; o < kN4; o++) {
            const int py = oy + pr0 + o;
            if (pr0 + o >= F::kH || px >= vd.W || py >= vd.H) continue;
            const int64_t ppix = vd.pix_base + (int64_t)py * vd.W + px;
            const float m = pix_mask<MASK>(ot4[o]);
            const float x = ox4[o] * m, y = target_channel(ot4[o], c) * m;
            const float df = x - y;
            const float dS = ab[o].x + 2.f * x * ab[o].y + y * d[o];
            const float sg = df > 0.f ? 1.f : (df < 0.f ? -1.f : 0.f);
            dl[3 * ppix + c] = MASK ? m * (((1.f - lam) * sg - lam * dS) * inv_n) : ((1.f - lam) * sg - lam * dS) * inv_n;
            l1 += fabsf(df);
        }
    }
    // per-CTA partial sums (L1, SSIM), then the last CTA adds them in order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        l1 += __shfl_down_sync(0xffffffffu, l1, o);
        ss += __shfl_down_sync(0xffffffffu, ss, o);
    }
    if ((tid & 31) == 0) { red[0][tid >> 5] = l1; red[1][tid >> 5] = ss; }
    __syncthreads();
    if (tid == 0) {
        float a = 0.f, b = 0.f;
        for (int i = 0; i < kSsThreads / 32; i++) { a += red[0][i]; b += red[1][i]; }
        part[2 * blockIdx.x] = a;
        part[2 * blockIdx.x + 1] = b;
        __threadfence();
        is_last = atomicAdd(&hdr->loss_counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (is_last) {
        __threadfence();
        float a = 0.f, b = 0.f;
        for (unsigned i = tid; i < gridDim.x; i += kSsThreads) {
            a += ((volatile float*)part)[2 * i];
            b += ((volatile float*)part)[2 * i + 1];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
        __syncthreads();
        if ((tid & 31) == 0) { red[0][tid >> 5] = a; red[1][tid >> 5] = b; }
        __syncthreads();
        if (tid == 0) {
            float ta = 0.f, tb = 0.f;
            for (int i = 0; i < kSsThreads / 32; i++) { ta += red[0][i]; tb += red[1][i]; }
            hdr->loss = (1.f - lam) * ta * inv_n + lam * (1.f - tb * inv_n);
            hdr->loss_counter = 0;
        }
    }
}

template <typename F>
static int64_t ssim_ctas(const Views& V)
{
    int64_t t = 0;
    for (int v = 0; v < V.n; v++) t += ssim_tiles<F>(V.v[v]);
    return 3 * t;
}

int64_t ssim_blocks(const Views& V) { return std::max(ssim_ctas<SsimWide>(V), ssim_ctas<SsimExact>(V)); }

void launch_loss_l1_ssim(const Plan& P, const WsPtrs& w, const float* image, const void* target_rgba8, float lam,
                         bool alpha_mask, float* dl, cudaStream_t st)
{
    const float inv_n = 1.0f / (float)(3 * P.views.pixels);
    const uchar4* t = static_cast<const uchar4*>(target_rgba8);
#define GS_SSIM(MASK, F)                                                                                            \
    do {                                                                                                            \
        constexpr int smem = (int)sizeof(SsimGeo<F>::Smem);                                                         \
        cudaFuncSetAttribute(k_loss_l1_ssim<MASK, F>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);           \
        launch_after(k_loss_l1_ssim<MASK, F>, (unsigned)ssim_ctas<F>(P.views), F::kThreads, smem, st, P.views,      \
                     image, t, lam, inv_n, dl, w.loss_part, w.hdr);                                                 \
    } while (0)
    const bool wide = P.mom_bf16;      // see the top of the file
    if (alpha_mask && wide) GS_SSIM(true, SsimWide);
    else if (wide) GS_SSIM(false, SsimWide);
    else if (alpha_mask) GS_SSIM(true, SsimExact);
    else GS_SSIM(false, SsimExact);
#undef GS_SSIM
}

}  // namespace gs
