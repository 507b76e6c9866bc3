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
// is symmetric).  A CTA takes two 16x16 tiles of a view and colour channel: x and y
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
// Issue- and FP32-bound (70% of issue slots).  Every pass is register-blocked along its window: a thread
// reads the 11 + n - 1 values of n neighbouring outputs once instead of 11 values an
// output.  Moments and partials are packed pairs (FFMA2).  The three channels of a tile
// are neighbouring CTAs, so that small images fill the chip and the channels' accesses
// to one pixel meet in L2.  All staging loads of a thread are in flight together (four
// rows at a time took a third longer).  Against one output a thread in 16x16 tiles of
// all channels, four 1080p views and 403x301: 1.43 -> 0.94 ms, 33 -> 22 us; about 600
// FP32 operations a pixel and channel with the halos.
//
// 16x16 tiles, because a window then lies at most 18 pixels from its shift.  Tiles of
// 32x31 run in 0.56 ms (400 operations), but their windows lie up to 26 pixels from it:
// where the image steps in between, E[x^2] - mu_x^2 cancels more.  RMS error of the
// gradient against 64 bits over its RMS, 480x384: noise 1.4e-7 and flat 1.1e-6 in both;
// checkerboards of 16, 31, 48 and 96 pixels 1.7e-6, 7.0e-6, 2.0e-6 and 2.0e-6 here and
// 1.9e-5, 1.3e-5, 1.3e-5 and 4.1e-6 there.
#include "raster_blocks.cuh"

namespace gs {

constexpr int kSsR = 5;                    // window radius
// Tile, tiles side by side per CTA, outputs per thread of the four passes, threads, CTAs
// per SM, threads per staged row; then the shared-memory pitches.
constexpr int kSsW = 16, kSsH = 16, kSsP = 2, kN1 = 9, kN2 = 7, kN3 = 4, kN4 = 3;
constexpr int kSsThreads = 224, kSsCtas = 4, kSsRow = 56;
constexpr int kPx = 53, kPm = 27, kPa = 27, kPh = 17;
constexpr int kQw = kSsW + 2 * kSsR, kQh = kSsH + 2 * kSsR;             // positions whose window reaches a tile
constexpr int kXw = kSsP * kSsW + 4 * kSsR, kXh = kSsH + 4 * kSsR;      // staged pixels
constexpr int kG1 = (kQw + kN1 - 1) / kN1, kG2 = (kQh + kN2 - 1) / kN2;
constexpr int kG3 = (kSsW + kN3 - 1) / kN3, kG4 = (kSsH + kN4 - 1) / kN4;
static_assert(kSsP * kXh * kG1 <= kSsThreads && kSsP * kQw * kG2 <= kSsThreads && kSsP * kQh * kG3 <= kSsThreads &&
                  kSsP * kSsW * kG4 <= kSsThreads,
              "one task per thread in every pass");
constexpr int kOver = kG2 * kN2 + 2 * kSsR - kXh;      // rows read past the end
static_assert(kPx >= kSsP * kSsW - kSsW + kG1 * kN1 + 2 * kSsR && kOver >= 0, "what the last groups read");
// Pitches odd in the unit read across rows (no bank conflicts).  The outputs past
// the edge that a last group computes and drops read what follows in shared memory.
struct SsimSmem {
    union {
        float2 xy[kXh][kPx];                // (x, y)
        struct {
            float2 ab[kSsP][kQh][kPa];      // (A, B)
            float c[kSsP][kQh][kPa];        // Cc
        } abc;
    };
    union {
        struct {
            float4 m03[kSsP][kXh][kPm];     // (mu_x, mu_y, E[x^2], E[y^2]) of the rows
            float m4[kSsP][kXh][kPm];       // E[xy]
            float past[kOver * kPm + 1];
        } h;
        struct {
            float2 ab[kSsP][kQh][kPh];
            float c[kSsP][kQh][kPh];
        } habc;
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

__host__ __device__ __forceinline__ int64_t ssim_tiles(const ViewDesc& vd)
{
    return (int64_t)((vd.W + kSsP * kSsW - 1) / (kSsP * kSsW)) * ((vd.H + kSsH - 1) / kSsH);
}

__device__ __forceinline__ int ssim_view_of_tile(const Views& V, int64_t t, int64_t& first)
{
    int64_t base = 0;
    for (int v = 0; v < V.n; v++) {
        const int64_t nt = ssim_tiles(V.v[v]);
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

template <bool MASK>
__global__ void __launch_bounds__(kSsThreads, kSsCtas)
    k_loss_l1_ssim(Views V, const float* __restrict__ image, const uchar4* __restrict__ target, float lam, float inv_n,
                   float* __restrict__ dl, float* __restrict__ part, WsHeader* __restrict__ hdr)
{
    if (!after_previous()) return;
    extern __shared__ __align__(16) unsigned char ssim_smem[];
    SsimSmem& sm = *reinterpret_cast<SsimSmem*>(ssim_smem);
    __shared__ float red[2][kSsThreads / 32];
    __shared__ float2 shift[kSsP];
    __shared__ bool is_last;

    const int tid = threadIdx.x;
    int64_t first;
    const int c = (int)(blockIdx.x % 3u);        // colour channel
    const int64_t tile = blockIdx.x / 3u;
    const int v = ssim_view_of_tile(V, tile, first);
    const ViewDesc& vd = V.v[v];
    const int lt = (int)(tile - first);
    const int TX = (vd.W + kSsP * kSsW - 1) / (kSsP * kSsW);
    const int ox = (lt % TX) * (kSsP * kSsW), oy = (lt / TX) * kSsH;
    float l1 = 0.f, ss = 0.f;

    // The tiles' shifts, their centre pixels, and the staged pixels: all loads of a
    // thread are in flight together (one memory round trip a tile).  The first pass
    // subtracts the shifts.
    // (a non-finite centre pixel shifts by nothing: it reaches only its own windows)
    const int sp = min(tid, kSsP - 1);
    const int64_t cpix = vd.pix_base + (int64_t)min(oy + kSsH / 2, vd.H - 1) * vd.W +
                         min(ox + kSsW * sp + kSsW / 2, vd.W - 1);
    const uchar4 tc = target[cpix];
    const float ic = image[3 * cpix + c];
    // (the shift's y is a code where the target's scale enters unrounded)
    constexpr float kYs = MASK ? 1.0f : 1.0f / 255.0f;
    {
        // kSsRow threads a row, so that no index is divided
        constexpr int RS = kSsThreads / kSsRow, NR = (kXh + RS - 1) / RS;
        static_assert(kSsThreads % kSsRow == 0 && kXw <= kSsRow, "whole rows");
        const int col = tid % kSsRow, r0 = tid / kSsRow, x = ox - 2 * kSsR + col;
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
        if (tid < kSsP)
            shift[tid] = make_float2(isfinite(ic * mc) ? ic * mc : 0.f,
                                     MASK ? target_channel(tc, c) * mc : target_code(tc, c));
#pragma unroll
        for (int k = 0; k < NR; k++) {
            const int r = r0 + RS * k;
            const float m = pix_mask<MASK>(ti[k]);
            if (col < kXw && r < kXh) sm.xy[r][col] = make_float2(xi[k] * m, target_channel(ti[k], c) * m);
        }
    }
    __syncthreads();
    // horizontal pass: 5 moments at the staged rows and the windows' columns of each tile
    if (tid < kSsP * kXh * kG1) {
        const int p = tid / (kXh * kG1), i = tid % (kXh * kG1);
        const int r = i % kXh, q0 = (i / kXh) * kN1;
        const float2 s2 = shift[p], sh = f2(-s2.x, -s2.y), sf = f2(1.f, kYs);
        const float2* row = sm.xy[r] + kSsW * p + q0;
        float2 m01[kN1], m23[kN1];
        float m4[kN1];
#pragma unroll
        for (int o = 0; o < kN1; o++) {
            m01[o] = m23[o] = make_float2(0.f, 0.f);
            m4[o] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < kN1 + 2 * kSsR; j++) {
            const float2 xy = fma2(sh, sf, row[j]);
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
        const int p = tid / (kQw * kG2), i = tid % (kQw * kG2);
        const int qc = i % kQw, r0 = (i / kQw) * kN2;
        const float2 sh = shift[p];
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
        const int x = ox + kSsW * p - kSsR + qc;
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
                const float ib = 1.0f / (b1 * b2);
                const float s = a1 * a2 * ib;
                A = 2.f * my * (a2 - a1) * ib - 2.f * mx * s / b1 + 2.f * mx * s / b2;
                B = -s / b2;
                Cc = 2.f * a1 * ib;
                if (qr >= kSsR && qr < kSsR + kSsH && qc >= kSsR && qc < kSsR + kSsW) ss += s;
            }
            sm.abc.ab[p][qr][qc] = make_float2(A, B);
            sm.abc.c[p][qr][qc] = Cc;
        }
    }
    __syncthreads();
    // the tiles' own pixels, requested before the last two passes need them
    const int p4 = tid / (kSsW * kG4), pc = tid % kSsW, pr0 = (tid % (kSsW * kG4)) / kSsW * kN4;
    const int px = ox + kSsW * p4 + pc;
    float ox4[kN4];
    uchar4 ot4[kN4];
#pragma unroll
    for (int o = 0; o < kN4; o++) {
        const int py = oy + pr0 + o;
        ox4[o] = 0.f;
        ot4[o] = make_uchar4(0, 0, 0, 0);
        if (p4 < kSsP && pr0 + o < kSsH && px < vd.W && py < vd.H) {
            const int64_t ppix = vd.pix_base + (int64_t)py * vd.W + px;
            ox4[o] = image[3 * ppix + c];
            ot4[o] = target[ppix];
        }
    }
    // horizontal pass of A, B, Cc at the tiles' columns
    if (tid < kSsP * kQh * kG3) {
        const int p = tid / (kQh * kG3), i = tid % (kQh * kG3);
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
            if (q0 + o < kSsW) {
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
            if (pr0 + o >= kSsH || px >= vd.W || py >= vd.H) continue;
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

int64_t ssim_blocks(const Views& V)
{
    int64_t t = 0;
    for (int v = 0; v < V.n; v++) t += ssim_tiles(V.v[v]);
    return 3 * t;
}

void launch_loss_l1_ssim(const Plan& P, const WsPtrs& w, const float* image, const void* target_rgba8, float lam,
                         bool alpha_mask, float* dl, cudaStream_t st)
{
    const float inv_n = 1.0f / (float)(3 * P.views.pixels);
    const uchar4* t = static_cast<const uchar4*>(target_rgba8);
#define GS_SSIM(MASK)                                                                                               \
    do {                                                                                                            \
        constexpr int smem = (int)sizeof(SsimSmem);                                                                 \
        cudaFuncSetAttribute(k_loss_l1_ssim<MASK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);              \
        launch_after(k_loss_l1_ssim<MASK>, (unsigned)ssim_blocks(P.views), kSsThreads, smem, st, P.views, image, t, \
                     lam, inv_n, dl, w.loss_part, w.hdr);                                                           \
    } while (0)
    if (alpha_mask) GS_SSIM(true);
    else GS_SSIM(false);
#undef GS_SSIM
}

}  // namespace gs
