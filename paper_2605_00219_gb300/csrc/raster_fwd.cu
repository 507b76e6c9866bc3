// raster_fwd.cu -- front-to-back alpha compositing per tile (VkSplat Sec. 2
// pipeline, Table 2 "Rasterization Fwd"), and the L1 loss gradient
// (Sec. 4.5, L1 term).
//
// One CTA per tile, two pixels per thread, each warp 8x8 pixels as four 4x4
// blocks (raster_blocks.cuh).  The tile's sorted list is staged through shared
// memory one chunk at a time (coalesced reads of the sorted pair indices, then
// asynchronous 48-byte record copies); with each entry the loader stores a
// mask of the blocks it can contribute to.  Each warp turns the masks of its
// four blocks into four lists of entry offsets (ballots), padded with a
// stand-in entry to the longest, and walks them together: the 8 lanes of a
// block read their own list.  Transmittance is a compensated FP32 pair
// (TwoProduct with FMA, the low part carried alongside), so the product over
// hundreds of factors keeps close to full FP32 accuracy.
#include "raster_blocks.cuh"

namespace gs {

// Issue-bound (79% of issue slots at the headline size; ALU pipe 65%).  Per
// warp iteration (four visits) about 66 instructions, of which the transmittance
// update is packed (FMUL2 / FFMA2, both pixels of a lane); about 0.38 ms of
// the 1.38 ms at 3M Gaussians, 4x1080p, is outside the walk (staging 0.29,
// block lists 0.06, masks 0.02).  One warp over 8x4 pixels with one pixel per
// lane took 2.07 ms.  9 blocks per SM at 56 registers: 1.38 ms, 8 at 64 registers
// 1.42, 10 at 48 registers 1.49; the walk unrolled by 2 at 9 blocks 1.65.
template <int TW, int TH>
__global__ void __launch_bounds__(TileBlocks<TW, TH>::kThreads, TW * TH == 256 ? 9 : TW * TH == 512 ? 4 : 16)
k_raster_fwd(Views V, const uint32_t* __restrict__ order, const uint2* __restrict__ ranges,
             const uint32_t* __restrict__ pid_sorted, const ProjRec* __restrict__ rec, const float* __restrict__ bg,
             float* __restrict__ image, float* __restrict__ tfinal, uint32_t* __restrict__ nlast,
             WsHeader* __restrict__ hdr, uint32_t cap)
{
    if (!after_previous()) return;
    using TB = TileBlocks<TW, TH>;
    constexpr int NT = TB::kThreads, NW = TB::kWarps, CH = TW == 8 ? 64 : 128;   // CH: list entries per staged chunk
    constexpr int IPT = (CH + NT - 1) / NT;      // staged entries per thread
    // entry CH of each buffer is a stand-in that no pixel blends (opacity 0),
    // for the lanes of a block whose list is shorter than its warp's longest
    // staged entry: (mean x, y (tile-relative), exponent A, B), (exponent C,
    // opacity, red, green), (blue, -, -, -)
    __shared__ float4 sE[2][CH + 1][3];
    __shared__ uint32_t sM[2][CH];
    __shared__ float4 sraw[CH][3];     // records in flight
    __shared__ uint16_t slist[4 * NW][CH + 2];   // byte offsets of a block's entries
    __shared__ unsigned long long sblend[NW];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, grp = lane >> 3;
    const int64_t gt = order[blockIdx.x];   // longest lists first
    const int v = view_of_tile(V, gt);
    const ViewDesc& vd = V.v[v];
    const int lt = (int)(gt - vd.tile_base);
    const int ox = (lt % vd.TX) * TW, oy = (lt / vd.TX) * TH;
    const int px = ox + TB::px(w, lane), py = oy + TB::py(w, lane);   // and (px, py + 2)
    const bool in0 = px < vd.W && py < vd.H, in1 = px < vd.W && py + 2 < vd.H;
    // pixel centres relative to the tile's first pixel (the staged means are too)
    const float fx = (float)(px - ox) + 0.5f, fy0 = (float)(py - oy) + 0.5f, fy1 = (float)(py + 2 - oy) + 0.5f;
    const uint2 r = range_at(ranges, gt, cap, &hdr->status);
    if (tid < 6) sE[tid / 3][CH][tid % 3] = make_float4(0.f, 0.f, 0.f, 0.f);

    // transmittance T = Th - nTl: the low part is carried negated, so that
    // both it and the rounding of each product come from one FMA
    const float2 one = f2(1.0f, 1.0f);
    float2 Th = one, nTl = f2(0.0f, 0.0f);
    float C0[2] = {0.f, 0.f}, C1[2] = {0.f, 0.f}, C2[2] = {0.f, 0.f};
    // the exponent cutoff of a pixel; NaN once it is done (no pair passes)
    const float kDone = __int_as_float(0x7fffffff);
    float thr0 = in0 ? kPow2Min : kDone, thr1 = in1 ? kPow2Min : kDone;
    uint32_t last0 = 0, last1 = 0, nbl = 0;

    auto stage = [&](int buf, int i) {
        const float4 qa = sraw[i][0], qb = sraw[i][1], qc = sraw[i][2];
        sE[buf][i][0] = pair_coefs(tile_mean(qa.x, qc.z, ox), tile_mean(qa.y, qc.w, oy), qa.z, qa.w, qb.x);
        sE[buf][i][1] = make_float4(pair_c2(qb.x), qb.y, qb.z, qb.w);
        sE[buf][i][2].x = qc.x;
        sM[buf][i] = block_mask<TW, TH, 4>(qa.x - ((float)ox + 0.5f), qa.y - ((float)oy + 0.5f), qa.z, qa.w, qb.x, qb.y);
    };
    // chunk 0 is staged directly; afterwards the records of chunk i + 1 are
    // copied to shared memory while chunk i is composited (the pair indices
    // one chunk further ahead) and turned into staged entries at its end
    uint32_t pid_next[IPT];
#pragma unroll
    for (int u = 0; u < IPT; u++) {
        const uint32_t i = tid + u * NT;
        pid_next[u] = 0u;
        if (i < CH && r.x + i < r.y) rec_copy_async(sraw[i], rec, pid_sorted[r.x + i], V.pairs, &hdr->status);
        if (i < CH && r.x + CH + i < r.y) pid_next[u] = pid_sorted[r.x + CH + i];
    }
    copy_async_wait();
#pragma unroll
    for (int u = 0; u < IPT; u++) {
        const uint32_t i = tid + u * NT;
        if (i < CH && r.x + i < r.y) stage(0, i);
    }
    int cur = 0;
    for (uint32_t base = r.x; base < r.y; base += CH, cur ^= 1) {
        const bool done = isnan(thr0) && isnan(thr1);
        if (__syncthreads_count(done) == NT) break;
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const uint32_t i = tid + u * NT;
            if (i < CH && base + CH + i < r.y) rec_copy_async(sraw[i], rec, pid_next[u], V.pairs, &hdr->status);
            if (i < CH && base + 2 * CH + i < r.y) pid_next[u] = pid_sorted[base + 2 * CH + i];
        }
        const char* __restrict__ cE = reinterpret_cast<const char*>(sE[cur]);
        const int cnt = (int)min((uint32_t)CH, r.y - base);
        // the four blocks' entry lists, in list order (a finished block's
        // stays empty)
        const uint32_t dn = __ballot_sync(0xffffffffu, done);
        uint32_t live = 0;
        int n4[4];
#pragma unroll
        for (int g = 0; g < 4; g++) {
            live |= ((dn >> (8 * g)) & 0xffu) == 0xffu ? 0u : 1u << g;
            n4[g] = 0;
        }
        for (int c0 = 0; c0 < cnt; c0 += 32) {
            const uint32_t m = c0 + lane < cnt ? (sM[cur][c0 + lane] >> (4 * w)) & live : 0u;
#pragma unroll
            for (int g = 0; g < 4; g++) {
                const uint32_t bal = __ballot_sync(0xffffffffu, m & (1u << g));
                if (m & (1u << g)) slist[4 * w + g][n4[g] + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(48 * (c0 + lane));
                n4[g] += __popc(bal);
            }
        }
        const int n = grp == 0 ? n4[0] : grp == 1 ? n4[1] : grp == 2 ? n4[2] : n4[3];
        int nmax = max(max(n4[0], n4[1]), max(n4[2], n4[3]));
        uint16_t* lp = slist[4 * w + grp];
        for (int i = n + (lane & 7); i <= nmax; i += 8) lp[i] = (uint16_t)(48 * CH);
        __syncwarp();
        uint32_t lo0 = ~0u, lo1 = ~0u;       // the pixels' last blended entries of this chunk
        uint32_t off = lp[0];
#pragma unroll 1
        for (int i = 0; i < nmax; i++) {
            const float4* __restrict__ e = reinterpret_cast<const float4*>(cE + off);
            const float4 a = e[0];
            const float4 b = e[1];
            const float blue = e[2].x;
            const uint32_t offc = off;
            off = lp[i + 1];
            const float dx = pix_offset(fx, a.x);
            const float dy0 = pix_offset(fy0, a.y), dy1 = pix_offset(fy1, a.y);
            const PowX px2 = pair_power2_x(dx, a.z, a.w);
            const float p0 = pair_power2_y(px2, dy0, b.x), p1 = pair_power2_y(px2, dy1, b.x);
            // one test a pixel for both skips; a pixel that skips takes
            // alpha = 0, which leaves its transmittance as it is
            const float ar0 = __fmul_rn(b.y, ex2_approx(p0)), ar1 = __fmul_rn(b.y, ex2_approx(p1));
            bool h0 = p0 >= thr0 && ar0 >= kAlphaMin, h1 = p1 >= thr1 && ar1 >= kAlphaMin;
            float2 al = f2(h0 ? fminf(kAlphaMax, ar0) : 0.f, h1 ? fminf(kAlphaMax, ar1) : 0.f);
            // compensated T (1 - alpha): om + om_err = 1 - alpha exactly
            // (ne = -om_err), pr the rounded product, the low part
            // Th om_err + Tl om + (Th om - pr) carried without renormalising
            const float2 om = sub2(one, al), nom = sub2(al, one);
            const float2 ne = add2(al, sub2(om, one));
            float2 pr = mul2(Th, om);
            float2 nlo = fma2(Th, ne, fma2(nTl, om, fma2(Th, nom, pr)));
            const float2 sum = sub2(pr, nlo);
            if (__any_sync(0xffffffffu, fminf(sum.x, sum.y) < kTMin)) {
                // a pixel stops before this pair (once per pixel)
                const bool s0 = sum.x < kTMin, s1 = sum.y < kTMin;
                if (s0) { pr.x = Th.x; nlo.x = nTl.x; al.x = 0.f; h0 = false; thr0 = kDone; }
                if (s1) { pr.y = Th.y; nlo.y = nTl.y; al.y = 0.f; h1 = false; thr1 = kDone; }
                if (__all_sync(0xffffffffu, isnan(thr0) && isnan(thr1))) nmax = 0;   // the warp is finished
            }
            const float2 wgt = mul2(al, Th);
            if (h0) {
                C0[0] = fmaf(b.z, wgt.x, C0[0]);
                C1[0] = fmaf(b.w, wgt.x, C1[0]);
                C2[0] = fmaf(blue, wgt.x, C2[0]);
                lo0 = offc;
                nbl++;
            }
            if (h1) {
                C0[1] = fmaf(b.z, wgt.y, C0[1]);
                C1[1] = fmaf(b.w, wgt.y, C1[1]);
                C2[1] = fmaf(blue, wgt.y, C2[1]);
                lo1 = offc;
                nbl++;
            }
            Th = pr;
            nTl = nlo;
        }
        if (lo0 != ~0u) last0 = base - r.x + lo0 / 48u + 1u;
        if (lo1 != ~0u) last1 = base - r.x + lo1 / 48u + 1u;
        copy_async_wait();
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const uint32_t i = tid + u * NT;
            if (i < CH && base + CH + i < r.y) stage(cur ^ 1, i);
        }
    }
    if (gt == 0 && tid < 3) hdr->bg[tid] = bg ? bg[tid] : 0.f;
    const float2 T = sub2(Th, nTl);
    float b0 = 0.f, b1 = 0.f, b2 = 0.f;
    if (bg) { b0 = bg[0]; b1 = bg[1]; b2 = bg[2]; }
#pragma unroll
    for (int k = 0; k < 2; k++) {
        if (k ? in1 : in0) {
            const int64_t pix = vd.pix_base + (int64_t)(py + 2 * k) * vd.W + px;
            const float Tk = k ? T.y : T.x;
            image[3 * pix + 0] = fmaf(Tk, b0, C0[k]);
            image[3 * pix + 1] = fmaf(Tk, b1, C1[k]);
            image[3 * pix + 2] = fmaf(Tk, b2, C2[k]);
            tfinal[pix] = Tk;
            nlast[pix] = k ? last1 : last0;
        }
    }
    // blended pair count: warp reduce, one atomic per CTA
    const unsigned long long c = __reduce_add_sync(0xffffffffu, nbl & 0xffffu) +
                                 ((unsigned long long)__reduce_add_sync(0xffffffffu, nbl >> 16) << 16);
    if (lane == 0) sblend[w] = c;
    __syncthreads();
    if (tid == 0) {
        unsigned long long s = 0;
        for (int i = 0; i < NW; i++) s += sblend[i];
        if (s) atomicAdd(&hdr->blended, s);
    }
}

void launch_raster_fwd(const Plan& P, const WsPtrs& w, const float* bg, float* image, cudaStream_t st)
{
    const Views& V = P.views;
    const unsigned grid = (unsigned)V.tiles;
#define GS_RF(TW, TH) launch_after(k_raster_fwd<TW, TH>, grid, TileBlocks<TW, TH>::kThreads, 0, st,                           \
        V, w.tile_order, w.ranges, w.pid_sorted, w.rec, bg, image, w.tfinal, w.nlast, w.hdr, (uint32_t)P.cap)
    if (V.tw == 8) GS_RF(8, 8);
    else if (V.th == 16) GS_RF(16, 16);
    else GS_RF(16, 32);
#undef GS_RF
}

// ---------------------------------------------------------------------------
// L1 loss and gradient
// ---------------------------------------------------------------------------

constexpr int kLossThreads = 256;
constexpr int kLossItems = 8;

__device__ __forceinline__ float l1_sign(float d, float inv_n) { return d > 0.f ? inv_n : (d < 0.f ? -inv_n : 0.f); }

// VEC: the three arrays are 16-byte aligned; each thread takes kLossItems / 2
// float4 (a block 2 x kLossThreads x kLossItems values), the ragged end
// value by value.
template <bool VEC>
__global__ void __launch_bounds__(kLossThreads) k_loss_l1(const float* __restrict__ image,
                                                          const float* __restrict__ target, float* __restrict__ dl,
                                                          int64_t n, float inv_n, float* __restrict__ part,
                                                          WsHeader* __restrict__ hdr)
{
    if (!after_previous()) return;
    __shared__ float ws[kLossThreads / 32];
    __shared__ bool is_last;
    float s = 0.f;
    if (VEC) {
        const int64_t base4 = (int64_t)blockIdx.x * kLossThreads * (kLossItems / 2);
#pragma unroll
        for (int i = 0; i < kLossItems / 2; i++) {
            const int64_t i4 = base4 + i * kLossThreads + threadIdx.x, e = 4 * i4;
            if (e + 3 < n) {
                const float4 a = reinterpret_cast<const float4*>(image)[i4];
                const float4 b = reinterpret_cast<const float4*>(target)[i4];
                const float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
                reinterpret_cast<float4*>(dl)[i4] =
                    make_float4(l1_sign(d0, inv_n), l1_sign(d1, inv_n), l1_sign(d2, inv_n), l1_sign(d3, inv_n));
                s += (fabsf(d0) + fabsf(d1)) + (fabsf(d2) + fabsf(d3));
            } else {
                for (int64_t k = e; k < n && k < e + 4; k++) {
                    const float d = image[k] - target[k];
                    dl[k] = l1_sign(d, inv_n);
                    s += fabsf(d);
                }
            }
        }
    } else {
        const int64_t base = (int64_t)blockIdx.x * kLossThreads * kLossItems;
#pragma unroll
        for (int i = 0; i < kLossItems; i++) {
            const int64_t idx = base + i * kLossThreads + threadIdx.x;
            if (idx < n) {
                const float d = image[idx] - target[idx];
                dl[idx] = l1_sign(d, inv_n);
                s += fabsf(d);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int i = 0; i < kLossThreads / 32; i++) t += ws[i];
        part[blockIdx.x] = t;
        __threadfence();
        const uint32_t done = atomicAdd(&hdr->loss_counter, 1u);
        is_last = done == gridDim.x - 1;
    }
    __syncthreads();
    if (is_last) {
        // the last CTA sums the partials: thread t takes indices t, t + 256,
        // ... (Kahan-compensated), then a fixed-order tree -- deterministic
        __threadfence();
        float t = 0.f, comp = 0.f;
        for (unsigned i = threadIdx.x; i < gridDim.x; i += kLossThreads) {
            const float y = ((volatile float*)part)[i] - comp;
            const float u = t + y;
            comp = (u - t) - y;
            t = u;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            float tt = 0.f;
            for (int i = 0; i < kLossThreads / 32; i++) tt += ws[i];
            hdr->loss = tt * inv_n;
            hdr->loss_counter = 0;
        }
    }
}

void launch_loss_l1(const Plan& P, const WsPtrs& w, const float* image, const float* target, float* dl,
                    cudaStream_t st)
{
    const int64_t n = 3 * P.views.pixels;
    const bool vec = ((reinterpret_cast<uintptr_t>(image) | reinterpret_cast<uintptr_t>(target) |
                       reinterpret_cast<uintptr_t>(dl)) & 15u) == 0;
    const int64_t per_block = (int64_t)kLossThreads * kLossItems * (vec ? 2 : 1);
    const int64_t blocks = (n + per_block - 1) / per_block;
    if (vec)
        launch_after(k_loss_l1<true>, (unsigned)blocks, kLossThreads, 0, st, image, target, dl, n, 1.0f / (float)n,
                     w.loss_part, w.hdr);
    else
        launch_after(k_loss_l1<false>, (unsigned)blocks, kLossThreads, 0, st, image, target, dl, n, 1.0f / (float)n,
                     w.loss_part, w.hdr);
}

}  // namespace gs
