// raster_blocks.cuh -- what the raster forward and the pixel-parallel raster
// backward share: 4x4-pixel blocks walked by 8-lane groups, two pixels per
// lane held as packed FP32 pairs.
//
// A Gaussian's footprint in a tile is small (about 20 blended pixels an entry
// at 3M Gaussians, 1080p), so a warp that walks one entry over its 8x4 or 8x8
// pixels leaves most lanes idle.  Here each warp covers 8x8 pixels as four
// 4x4 blocks; the 8 lanes of a block walk the block's own entry list, so one
// warp instruction serves four (entry, block) visits.  Counted over 300 tiles
// of the 3M, 4x1080p scene, per list entry: 2.45 warp visits for 8x4 blocks,
// 1.68 for 8x8, and 0.91 warp iterations here (3.0 block visits / 4, and the
// longest of a warp's four lists counts).
#pragma once

#include "gs_internal.cuh"

namespace gs {

// ---- packed FP32 pairs: each half is one correctly rounded operation, the
// same bits as the scalar form, at half the issue slots.  Written with the
// explicit rounding, which keeps a product and a sum from being fused.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

#define GS_PACKED2(name, op)                                                                                   \
    __device__ __forceinline__ float2 name(float2 a, float2 b)                                                 \
    {                                                                                                          \
        unsigned long long d;                                                                                  \
        asm(op ".rn.f32x2 %0, %1, %2;"                                                                         \
            : "=l"(d)                                                                                          \
            : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b))); \
        return *reinterpret_cast<float2*>(&d);                                                                 \
    }
GS_PACKED2(mul2, "mul")
GS_PACKED2(add2, "add")
GS_PACKED2(sub2, "sub")
#undef GS_PACKED2

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// ---- geometry of the blocks of a TW x TH tile
template <int TW, int TH>
struct TileBlocks {
    static constexpr int kThreads = TW * TH / 2;        // two pixels per lane
    static constexpr int kWarps = kThreads / 32;
    static constexpr int kCols = TW / 4, kRows = TH / 4;
    static constexpr int kBlocks = kCols * kRows;
    static constexpr int kWarpsPerRow = TW / 8;
    // first pixel of this lane (its second one is two rows below), tile-relative
    __device__ static __forceinline__ int px(int w, int lane)
    {
        return (w % kWarpsPerRow) * 8 + ((lane >> 3) & 1) * 4 + (lane & 3);
    }
    __device__ static __forceinline__ int py(int w, int lane)
    {
        return (w / kWarpsPerRow) * 8 + (lane >> 4) * 4 + ((lane >> 2) & 1);
    }
};

// Conservative mask of the tile's BW x 4 blocks (BW = 4 or 8) that an entry can
// contribute to; warp w's four blocks are the bits 4w .. 4w + 3 (lane group
// g = bit 4w + g): 4x4 blocks in quads of 8x8 pixels, 8x4 blocks row by row.
// (x, y): the mean relative to the centre of the tile's first pixel.  A pair needs
// d^2 <= r^2 = min(9, 2 ln(255 o)); for each row of blocks the ellipse's extreme x over
// the row's band gives the first and last block: with h(dy) = sqrt(r^2/a - det dy^2 / a^2) the ellipse spans
// x - (b/a) dy -/+ h(dy), extreme at dy = -/+ ys (the offset of the leftmost /
// rightmost point) clamped to the band.  Against the box of the ellipse this
// drops 17% of the (entry, block) visits at the size above and costs about
// 100 instructions an entry on one lane.
// r^2 is widened by 0.2% + 1e-3, and by 4e-6 of the condition number
// kappa = a c / det, which bounds the rounding of det here and of the raster's own
// exponent (terms up to kappa d^2 cancel to d^2); past kappa = 1e5 every block
// is taken.
template <int TW, int TH, int BW>
__device__ __forceinline__ uint32_t block_mask(float x, float y, float a, float b, float c, float op)
{
    constexpr int NC = TW / BW, NR = TH / 4, NB = NC * NR;
    constexpr uint32_t kAll = NB == 32 ? 0xffffffffu : (1u << (NB & 31)) - 1u;
    if (!(op * 255.0f > 1.0f)) return 0u;      // alpha never reaches 1/255
    const float ac = a * c, det = ac - b * b;
    if (!(det > 0.0f)) return kAll;
    const float idet = __fdividef(1.0f, det);
    const float kappa = ac * idet;
    if (!(kappa < 1e5f)) return kAll;
    const float r2 = fmaf(fminf(9.0f, 2.0f * __logf(op * 255.0f)), fmaf(4e-6f, kappa, 1.002f), 1e-3f);
    const float s = r2 * idet;
    const float ex = sqrt_approx(s * c), ey = sqrt_approx(s * a);
    const float mg = fmaf(1e-5f, ex + ey + fabsf(x) + fabsf(y), 0.02f);
    const float ia = __fdividef(1.0f, a);
    const float k = -b * ia, u = r2 * ia * 1.00001f, w = det * ia * ia;
    const float ys = -b * __fdividef(ex, c);
    const float ylo = -ey - mg, yhi = ey + mg;
    uint32_t mask = 0;
#pragma unroll
    for (int by = 0; by < NR; by++) {
        const float lo = fmaxf((float)(4 * by) - y, ylo), hi = fminf((float)(4 * by + 3) - y, yhi);
        const float dR = fminf(fmaxf(ys, lo), hi), dL = fminf(fmaxf(-ys, lo), hi);
        const float hR = sqrt_approx(fmaxf(0.0f, fmaf(-w * dR, dR, u)));
        const float hL = sqrt_approx(fmaxf(0.0f, fmaf(-w * dL, dL, u)));
        const float xr = x + fmaf(k, dR, hR) + mg, xl = x + fmaf(k, dL, -hL) - mg;
        const int b0 = max(0, __float2int_ru((xl - (float)(BW - 1)) * (1.0f / BW)));
        const int b1 = min(NC - 1, __float2int_rd(xr * (1.0f / BW)));
        if (lo <= hi && b0 <= b1) {
            const uint32_t row = (2u << b1) - (1u << b0);
            if (BW == 8) {
                mask |= row << (by * NC);
            } else {
                // quads: columns 2, 3 belong to the next warp
                const uint32_t spread = NC == 4 ? (row & 3u) | ((row & 12u) << 2) : row;
                mask |= spread << ((by >> 1) * 2 * NC + (by & 1) * 2);
            }
        }
    }
    return mask;
}

// A record copied to shared memory without passing registers (three 16-byte
// asynchronous copies); the bounds-checked build copies a zero record (no
// block takes it) for an index outside the records.
__device__ __forceinline__ void rec_copy_async(float4* dst, const ProjRec* __restrict__ rec, uint32_t pid,
                                               int64_t pairs, uint32_t* status)
{
    (void)pairs;
    (void)status;
    if (!GS_DCHECK((int64_t)pid < pairs, status)) {
        dst[0] = dst[1] = dst[2] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const float4* src = reinterpret_cast<const float4*>(rec + pid);
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
#pragma unroll
    for (int i = 0; i < 3; i++)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16u * i), "l"(src + i) : "memory");
}

__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

}  // namespace gs
