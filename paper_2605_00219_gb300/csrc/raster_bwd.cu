// raster_bwd.cu -- rasterization backward parallel over Gaussians (VkSplat
// Sec. 4.2, first implementation; Fig. 2), with no pixel-level atomics.
//
// One CTA (4 warps) per tile.  The tile's list (up to the largest n_last of
// its pixels) is processed in batches of S Gaussians, S chosen per tile by
// the paper's rule S = roundup32(sqrt(N P)) capped at 128 (N = list length,
// P = pixels), or fixed by the tuning.  For each batch:
//
//  Phase A (pixels across threads): transmittance is recomputed front to
//    back from the running per-pixel state -- T as a compensated FP32 pair,
//    the blended colour prefix with Neumaier compensation -- and the state
//    (T, S) at the end of every 32-Gaussian sub-batch is kept in shared
//    memory, where S = C_image - prefix is the colour still to come.
//  Phase B (Gaussians across threads): warp k takes sub-batch k, lane l its
//    l-th Gaussian.  The lanes form a wavefront over the pixels: at step s
//    lane l handles pixel s - (31 - l), receives (T, S) from lane l + 1 by
//    warp shuffle, walks back over its own Gaussian (T_before = T / (1 - a),
//    S += c a T_before) and hands the state on.  Each lane accumulates its
//    Gaussian's nine gradients in registers; when S < 128 the warps split the
//    pixels instead and the partial sums are added in a fixed order.
//
// Output: one gradient record per intersection, at its emission slot, so
// the projection backward reads each Gaussian's records contiguously.  The
// result is deterministic (no atomics, fixed summation order).
#include <type_traits>

#include "raster_blocks.cuh"

namespace gs {

struct BwdSmem {
    float4* runA;   // [P] (T hi, T lo, prefix r, prefix g)
    float4* runB;   // [P] (prefix b, comp r, comp g, comp b)
    float4* pimg;   // [P] (C r, g, b, -)
    float4* pdl;    // [P] (dL/dC r, g, b, n_last bits)
    float4* st;     // [4][P] state (T, S r, S g, S b) after each sub-batch
    float4* gA;     // [128] (mx, my relative to the tile's first pixel, ca, cb)
    float4* gB;     // [128] (cc, o, r, g)
    float* gC;      // [128] blue
    uint32_t* ge;   // [128] emission slot
    float* red;     // [128][9] partial gradients
    int* misc;
};

__host__ __device__ constexpr size_t bwd_smem_bytes(int P)
{
    return (size_t)16 * P * 4 + (size_t)16 * 4 * P + 128 * (16 + 16 + 4 + 4) + 128 * 9 * 4 + 16;
}

__device__ __forceinline__ void neumaier_add(float& s, float& c, float x)
{
    const float t = s + x;
    c += fabsf(s) >= fabsf(x) ? (s - t) + x : (x - t) + s;
    s = t;
}

template <int P>
__global__ void __launch_bounds__(kBwdThreads) k_raster_bwd(Views V, const uint32_t* __restrict__ order,
                                                            const uint2* __restrict__ ranges,
                                                            const uint32_t* __restrict__ vals_sorted,
                                                            const uint32_t* __restrict__ pid_sorted,
                                                            const ProjRec* __restrict__ rec,
                                                            const float* __restrict__ image,
                                                            const float* __restrict__ dl,
                                                            const uint32_t* __restrict__ nlast,
                                                            GradRec* __restrict__ gradrec, int fixed_S)
{
    if (!after_previous()) return;
    extern __shared__ float4 smem4[];
    BwdSmem sm;
    sm.runA = smem4;
    sm.runB = sm.runA + P;
    sm.pimg = sm.runB + P;
    sm.pdl = sm.pimg + P;
    sm.st = sm.pdl + P;
    sm.gA = sm.st + 4 * P;
    sm.gB = sm.gA + 128;
    sm.gC = reinterpret_cast<float*>(sm.gB + 128);
    sm.ge = reinterpret_cast<uint32_t*>(sm.gC + 128);
    sm.red = reinterpret_cast<float*>(sm.ge + 128);
    sm.misc = reinterpret_cast<int*>(sm.red + 128 * 9);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t gt = order[blockIdx.x];   // longest lists first
    const int v = view_of_tile(V, gt);
    const ViewDesc& vd = V.v[v];
    const int lt = (int)(gt - vd.tile_base);
    const int tw = V.tw;
    const int ox = (lt % vd.TX) * tw, oy = (lt / vd.TX) * V.th;
    const uint2 r = ranges[gt];
    const uint32_t start = r.x, ntile = r.y - r.x;

    if (tid == 0) sm.misc[0] = 0;
    __syncthreads();
    // per-pixel inputs
    int my_max = 0;
    for (int pi = tid; pi < P; pi += kBwdThreads) {
        const int px = ox + pi % tw, py = oy + pi / tw;
        float4 im = make_float4(0.f, 0.f, 0.f, 0.f), d = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t nl = 0;
        if (px < vd.W && py < vd.H) {
            const int64_t pix = vd.pix_base + (int64_t)py * vd.W + px;
            im = make_float4(image[3 * pix], image[3 * pix + 1], image[3 * pix + 2], 0.f);
            d = make_float4(dl[3 * pix], dl[3 * pix + 1], dl[3 * pix + 2], 0.f);
            nl = nlast[pix];
        }
        d.w = __uint_as_float(nl);
        sm.pimg[pi] = im;
        sm.pdl[pi] = d;
        sm.runA[pi] = make_float4(1.f, 0.f, 0.f, 0.f);
        sm.runB[pi] = make_float4(0.f, 0.f, 0.f, 0.f);
        my_max = max(my_max, (int)nl);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) my_max = max(my_max, __shfl_xor_sync(0xffffffffu, my_max, o));
    if (lane == 0) atomicMax(&sm.misc[0], my_max);
    __syncthreads();
    const uint32_t L = min(ntile, (uint32_t)sm.misc[0]);

    int S = fixed_S;
    if (S <= 0) {
        const float x = sqrtf((float)L * (float)P);
        S = ((int)ceilf(x) + 31) & ~31;
    }
    S = min(max(S, 32), 128);
    const int nsub = S / 32;
    const int ngroups = (nsub == 3) ? 1 : 4 / nsub;
    const int glen = P / ngroups;

    for (uint32_t bb = 0; bb < L; bb += S) {
        const int cnt = (int)min((uint32_t)S, L - bb);
        if (tid < cnt) {
            const uint32_t k = start + bb + tid;
            const ProjRec q = rec[pid_sorted[k]];
            sm.gA[tid] = make_float4(tile_mean(q.a.x, q.c.z, ox), tile_mean(q.a.y, q.c.w, oy), q.a.z, q.a.w);
            sm.gB[tid] = q.b;
            sm.gC[tid] = q.c.x;
            sm.ge[tid] = vals_sorted[k];
        }
        __syncthreads();

        // ---------------- Phase A: pixel-parallel forward recompute ----------------
        const int nsub_used = (cnt + 31) >> 5;
        for (int pi = tid; pi < P; pi += kBwdThreads) {
            float4 ra = sm.runA[pi], rb = sm.runB[pi];
            float Th = ra.x, Tl = ra.y;
            float ps0 = ra.z, ps1 = ra.w, ps2 = rb.x, pc0 = rb.y, pc1 = rb.z, pc2 = rb.w;
            const float4 d = sm.pdl[pi];
            const float4 im = sm.pimg[pi];
            const uint32_t nl = __float_as_uint(d.w);
            // pixel centre relative to the tile's first pixel (the staged means are too)
            const float fx = (float)(pi % tw) + 0.5f, fy = (float)(pi / tw) + 0.5f;
            for (int k = 0; k < nsub_used; k++) {
                const int j1 = min(cnt, 32 * k + 32);
                for (int j = 32 * k; j < j1; j++) {
                    if (bb + j >= nl) break;
                    const float4 a = sm.gA[j];
                    const float4 b = sm.gB[j];
                    const float dx = pix_offset(fx, a.x), dy = pix_offset(fy, a.y);
                    const float4 pc = pair_coefs(a.x, a.y, a.z, a.w, b.x);
                    const float p2 = pair_power2(dx, dy, pc.z, pc.w, pair_c2(b.x));
                    if (p2 < kPow2Min) continue;
                    const float G = ex2_approx(p2);
                    const float araw = __fmul_rn(b.y, G);
                    if (araw < kAlphaMin) continue;
                    const float alpha = fminf(kAlphaMax, araw);
                    const float wgt = alpha * Th;
                    neumaier_add(ps0, pc0, b.z * wgt);
                    neumaier_add(ps1, pc1, b.w * wgt);
                    neumaier_add(ps2, pc2, sm.gC[j] * wgt);
                    const float om = __fsub_rn(1.0f, alpha);
                    const float om_err = __fsub_rn(-alpha, __fsub_rn(om, 1.0f));
                    const float pr = __fmul_rn(Th, om);
                    const float pe = __fmaf_rn(Th, om, -pr);
                    const float lo = __fmaf_rn(Th, om_err, __fmaf_rn(Tl, om, pe));
                    const float hi = __fadd_rn(pr, lo);
                    Tl = __fsub_rn(lo, __fsub_rn(hi, pr));
                    Th = hi;
                }
                sm.st[k * P + pi] =
                    make_float4(Th + Tl, (im.x - ps0) - pc0, (im.y - ps1) - pc1, (im.z - ps2) - pc2);
            }
            sm.runA[pi] = make_float4(Th, Tl, ps0, ps1);
            sm.runB[pi] = make_float4(ps2, pc0, pc1, pc2);
        }
        __syncthreads();

        // ---------------- Phase B: Gaussian-parallel wavefront ----------------
        const int sub = warp % nsub;
        const int pg = warp / nsub;
        const bool warp_on = (nsub != 3 || warp < 3) && sub < nsub_used;
        const int j = sub * 32 + lane;
        const bool act = warp_on && j < cnt;
        float g_mx = 0.f, g_my = 0.f, g_ca = 0.f, g_cb = 0.f, g_cc = 0.f, g_o = 0.f, g_r = 0.f, g_g = 0.f,
              g_b = 0.f;
        if (warp_on) {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            float cbl = 0.f;
            if (act) { a = sm.gA[j]; b = sm.gB[j]; cbl = sm.gC[j]; }
            const uint32_t myidx = bb + j;
            const int p0 = pg * glen;
            float T = 1.f, S0 = 0.f, S1 = 0.f, S2 = 0.f;
            const int nsteps = glen + 31;
            for (int s = 0; s < nsteps; s++) {
                float Ti = __shfl_down_sync(0xffffffffu, T, 1);
                float Si0 = __shfl_down_sync(0xffffffffu, S0, 1);
                float Si1 = __shfl_down_sync(0xffffffffu, S1, 1);
                float Si2 = __shfl_down_sync(0xffffffffu, S2, 1);
                if (lane == 31 && s < glen) {
                    const float4 q = sm.st[sub * P + p0 + s];
                    Ti = q.x; Si0 = q.y; Si1 = q.z; Si2 = q.w;
                }
                const int pl = s - (31 - lane);
                if (act && pl >= 0 && pl < glen) {
                    const int pi = p0 + pl;
                    const float4 d = sm.pdl[pi];
                    if (myidx < __float_as_uint(d.w)) {
                        const float dx = pix_offset((float)(pi % tw) + 0.5f, a.x);
                        const float dy = pix_offset((float)(pi / tw) + 0.5f, a.y);
                        const float4 pc = pair_coefs(a.x, a.y, a.z, a.w, b.x);
                        const float p2 = pair_power2(dx, dy, pc.z, pc.w, pair_c2(b.x));
                        if (p2 >= kPow2Min) {
                            const float G = ex2_approx(p2);
                            const float araw = __fmul_rn(b.y, G);
                            const float alpha = fminf(kAlphaMax, araw);
                            if (araw >= kAlphaMin) {
                                const float om = 1.0f - alpha;
                                const float rom = 1.0f / om;
                                const float Tb = Ti * rom;
                                const float wgt = alpha * Tb;
                                g_r = fmaf(wgt, d.x, g_r);
                                g_g = fmaf(wgt, d.y, g_g);
                                g_b = fmaf(wgt, d.z, g_b);
                                float da = d.x * (b.z * Tb - Si0 * rom);
                                da = fmaf(d.y, b.w * Tb - Si1 * rom, da);
                                da = fmaf(d.z, cbl * Tb - Si2 * rom, da);
                                Si0 = fmaf(b.z, wgt, Si0);
                                Si1 = fmaf(b.w, wgt, Si1);
                                Si2 = fmaf(cbl, wgt, Si2);
                                Ti = Tb;
                                if (araw <= kAlphaMax) {
                                    g_o = fmaf(da, G, g_o);
                                    const float dp = da * araw;
                                    g_ca = fmaf(-0.5f * dx * dx, dp, g_ca);
                                    g_cb = fmaf(-dx * dy, dp, g_cb);
                                    g_cc = fmaf(-0.5f * dy * dy, dp, g_cc);
                                    g_mx = fmaf(fmaf(a.z, dx, a.w * dy), dp, g_mx);
                                    g_my = fmaf(fmaf(a.w, dx, b.x * dy), dp, g_my);
                                }
                            }
                        }
                    }
                }
                T = Ti; S0 = Si0; S1 = Si1; S2 = Si2;
            }
        }
        if (ngroups == 1) {
            if (act) {
                GradRec o;
                o.a = make_float4(g_mx, g_my, g_ca, g_cb);
                o.b = make_float4(g_cc, g_o, g_r, g_g);
                o.c = make_float4(g_b, 0.f, 0.f, 0.f);
                gradrec[sm.ge[j]] = o;
            }
        } else {
            if (act) {
                float* rr = sm.red + (pg * S + j) * 9;
                rr[0] = g_mx; rr[1] = g_my; rr[2] = g_ca; rr[3] = g_cb; rr[4] = g_cc;
                rr[5] = g_o; rr[6] = g_r; rr[7] = g_g; rr[8] = g_b;
            }
            __syncthreads();
            if (tid < cnt) {
                float acc[9];
#pragma unroll
                for (int i = 0; i < 9; i++) acc[i] = 0.f;
                for (int q = 0; q < ngroups; q++) {
                    const float* rr = sm.red + (q * S + tid) * 9;
#pragma unroll
                    for (int i = 0; i < 9; i++) acc[i] += rr[i];
                }
                GradRec o;
                o.a = make_float4(acc[0], acc[1], acc[2], acc[3]);
                o.b = make_float4(acc[4], acc[5], acc[6], acc[7]);
                o.c = make_float4(acc[8], 0.f, 0.f, 0.f);
                gradrec[sm.ge[tid]] = o;
            }
        }
        __syncthreads();
    }
    // entries past every pixel's last blended pair receive zero gradients
    for (uint32_t k = start + L + tid; k < r.y; k += kBwdThreads) {
        GradRec o;
        o.a = o.b = o.c = make_float4(0.f, 0.f, 0.f, 0.f);
        gradrec[vals_sorted[k]] = o;
    }
}

// ===========================================================================
// The same backward with one pixel's sums per lane replaced by groups of 8 or 16
// lanes that walk 8x4- or 8x8-pixel blocks, two or four pixels per lane.
// ===========================================================================

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Sums nine values over the GL = 8 or 16 lanes of a group in halving steps, in
// the order of bfly9: (16 lanes: rows y, y + 1 first), then columns c, c + 4, then
// c, c + 2 and c, c + 1.  Afterwards lane s of the group holds sum
// group_sum_index<GL>(s) in `p` (-1: none); with 8 lanes, lane 0 also sum 2 in `q`.
template <int GL>
__device__ __forceinline__ void group_sums(const float* v, int lane, float& p, float& q)
{
    auto sx = [](float x, int o) { return __shfl_xor_sync(0xffffffffu, x, o); };
    constexpr int A = GL / 2, B = GL / 4, C = GL / 8;
    const bool ha = lane & A, hb = lane & B, hc = lane & C;
    const float2 k01 = add2(f2(ha ? v[5] : v[0], ha ? v[6] : v[1]), f2(sx(ha ? v[0] : v[5], A), sx(ha ? v[1] : v[6], A)));
    const float2 k23 = add2(f2(ha ? v[7] : v[2], ha ? v[8] : v[3]), f2(sx(ha ? v[2] : v[7], A), sx(ha ? v[3] : v[8], A)));
    const float k4 = v[4] + sx(v[4], A);
    const float2 m01 = add2(f2(hb ? k23.y : k01.x, hb ? k4 : k01.y), f2(sx(hb ? k01.x : k23.y, B), sx(hb ? k01.y : k4, B)));
    const float m2 = k23.x + sx(k23.x, B);
    p = (hc ? m01.y : m01.x) + sx(hc ? m01.x : m01.y, C);
    q = m2 + sx(m2, C);
    if (GL == 8) {
        if ((lane & 7) == 7) p = q;
    } else {
        const bool hd = lane & 1;
        p = (hd ? q : p) + sx(hd ? p : q, 1);
    }
}

template <int GL>
__device__ __forceinline__ int group_sum_index(int lane)
{
    const bool ha = lane & (GL / 2), hb = lane & (GL / 4), hc = lane & (GL / 8);
    if (GL == 16 && (lane & 1)) return hb || hc ? -1 : ha ? 7 : 2;
    if (hb && hc) return ha ? (GL == 8 ? 7 : -1) : 4;      // sum 4 is in both halves
    const int k = hb ? 3 : hc ? 1 : 0;
    return ha ? 5 + k : k;
}

// Walk of 8 x BH-pixel blocks of a TW x TH tile, GL lanes to a block (8 BH / GL
// pixels each).  Every (entry, block) visit sums its nine values over the block's lanes
// into a shared-memory slot of its own; an entry's slots are consecutive (a prefix
// sum over the batch of how many blocks each entry's mask holds), and after the
// batch one thread per entry adds them in block order.  A batch with more visits
// than slots is walked in passes.  The sums take the order of k_raster_bwd_px at one
// pixel per thread (rows y, y + 2; y, y + 1; columns c, c + 4; ...; blocks in
// order), so the records are the same bits: for needle-shaped Gaussians the
// projection backward amplifies a last-ulp change of a record up to 1e4-fold.
// BH = 8 takes the order of two pixels per thread (rows y, y + 4 one after the other,
// then y, y + 2; ...) for that choice's FP32 records.
//
// Issue-bound (73% of issue slots at 20 warps per SM; ALU 55%, FMA 34%, LSU 28%;
// 3M Gaussians, one 1080p view).  k_raster_bwd_px spends a warp visit per entry and
// 8x4 block (2.45 an entry) with a quarter of the lanes blending; here a warp
// iteration serves four (GL = 8: 0.68 an entry) or two (GL = 16: 1.16) visits, and
// the packed operations both pixels of a pair.  The walk without clamps and guards
// (no entry of the batch near alpha 0.99, no value so large that a product may
// overflow) saves 26 of about 215 instructions: 2.80 -> 2.66 ms.
//   GL = 8 (64 entries a batch, 10 blocks of 64 threads per SM): 1.17 -> 0.69 ms
//     (3M, one 1080p view, FP32), 4.67 -> 2.66 ms (four views), 0.174 -> 0.100 ms
//     (200k, 720p).  9 / 11 blocks per SM 2.72 / 2.72 ms.
//   GL = 16 (128 entries a batch, 128 threads): 27.1 -> 20.7 us (2,000 Gaussians,
//     128x128), 209 -> 183 us (400k, 640x360); 64 entries a batch 23.4 / 214 us.
//     GL = 8 takes 29.0 / 242 us there: too few blocks to hide one block's chain.
//   BH = 8, GL = 16 (64 entries a batch): against two pixels per thread of a warp per
//     8x8 block 0.96 -> 0.83 ms (3M, one 1080p view), 0.140 -> 0.113 (200k, 720p),
//     38.8 -> 36.7 us (2,000, 128x128); slower where few tiles are long (the launcher
//     has the line and the figures).
// Colours and loss gradients up to this size have finite products and sums, which the
// walk without guards multiplies by zero for the pixels that do not blend an entry.
constexpr float kTame = 1e15f;

template <int TW, int TH, int GL, int BH>
struct BwdBlocks {
    static constexpr int kCols = TW / 8, kBlocks = kCols * (TH / BH);
    static constexpr int kThreads = GL * kBlocks;
    static constexpr int kGroups = 32 / GL;                   // blocks per warp
    static constexpr int kPix = 8 * BH / GL;                  // pixels per lane
    static constexpr int kBatch = kPix == 4 ? 64 : 128;       // list entries per staged batch
    static constexpr int kSlots = BH == 8 ? 160 : GL == 8 ? 224 : 384;   // (entry, block) sums of one pass over a batch
    static constexpr int kBlocksPerSM = (kPix == 4 ? 10 : 5) * 256 / (TW * TH);
};

template <int TW, int TH, int GL, int BH>
__global__ void __launch_bounds__(BwdBlocks<TW, TH, GL, BH>::kThreads, BwdBlocks<TW, TH, GL, BH>::kBlocksPerSM)
k_raster_bwd_blocks(Views V, const uint32_t* __restrict__ order, const uint2* __restrict__ ranges,
                    const uint32_t* __restrict__ vals_sorted, const uint32_t* __restrict__ pid_sorted,
                    const ProjRec* __restrict__ rec, const float* __restrict__ tfinal, const float* __restrict__ bg,
                    const float* __restrict__ dl, const uint32_t* __restrict__ nlast, GradRec* __restrict__ gradrec,
                    uint32_t* __restrict__ status, uint32_t cap)
{
    if (!after_previous()) return;
    using B = BwdBlocks<TW, TH, GL, BH>;
    constexpr int NT = B::kThreads, NC = B::kCols, NB = B::kBlocks, BB = B::kBatch, S = B::kSlots;
    constexpr int NG = B::kGroups;
    constexpr int H = B::kPix / 2;               // packed pixel pairs per lane
    constexpr int IPT = (BB + NT - 1) / NT;      // staged entries per thread
    constexpr int kEnt = 48;                     // bytes of a staged entry
    static_assert(BB % 32 == 0 && NB <= S && 36 * (S + NB) < 65536 && kEnt * BB < 65536, "offsets fit 16 bits");
    // staged entry: (mean x, y (tile-relative), exponent A, B), (exponent C,
    // opacity, blue, blue), (red, red, green, green) -- the colours as pairs for
    // the packed operations; entry BB: a stand-in that no pixel blends
    __shared__ float4 sE[2][BB + 1][3];
    __shared__ float sQ[2][3][BB];           // conic a, b, c
    __shared__ uint32_t sM[2][BB], sBase[2][BB], sSlot[2][BB];
    // slots of each run of 32 entries; bit 31: an entry's alpha may reach the
    // 0.99 clamp, or a colour or gradient is beyond kTame
    __shared__ uint32_t sTot[2][BB / 32];
    __shared__ uint32_t slist[NB][BB + 2];   // entry's byte offset | slot's byte offset << 16
    __shared__ float part[S + NB][9];        // the last NB slots take the stand-in's sums
    __shared__ int smax[NB];

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, grp = lane / GL, blk = NG * w + grp;
    const int64_t gt = order[blockIdx.x];   // longest lists first
    const int v = view_of_tile(V, gt);
    const ViewDesc& vd = V.v[v];
    const int lt = (int)(gt - vd.tile_base);
    const int ox = (lt % vd.TX) * TW, oy = (lt / vd.TX) * TH;
    // this lane's column and first row; its pixels are the block's four rows
    // (8 lanes) or rows y, y + 2, ... (16 lanes)
    const int px = ox + (blk % NC) * 8 + (lane & 7);
    const int py = oy + (blk / NC) * BH + (GL == 8 ? 0 : (lane >> 3) & 1);
    constexpr int RS = GL == 8 ? 1 : 2;          // row step between the lane's pixels
    const uint2 r = range_at(ranges, gt, cap, status);
    const float fx = (float)(px - ox) + 0.5f, fy = (float)(py - oy) + 0.5f;
    if (tid < 6) sE[tid / 3][BB][tid % 3] = make_float4(0.f, 0.f, 0.f, 0.f);

    // The lane's pixels as packed pairs: rows (0, 1) and (2, 3), or (y, y + 2).
    // Per pixel:
    // last blended entry, compensated T after it, dL/dC, and nU = -sum_c dL/dC_c S_c
    // with S_c the colour still to come behind an entry (from T_final bg_c):
    // dL/dalpha = T dL/dC . col + nU / (1 - alpha)
    const float2 one = f2(1.0f, 1.0f), zero = f2(0.f, 0.f);
    // 1.0 the compiler cannot see through: x * one1 + y keeps the rounded x (a
    // packed product and sum would be fused)
    const float one1f = __uint_as_float(0x3f800000u | (cap >> 31));
    const float2 one1 = f2(one1f, one1f);
    float2 Th[H], Tl[H], nU[H], d0[H], d1[H], d2[H];
    int nl[2 * H];
    // a pixel of the tile has a dL/dC, or the background a colour, beyond kTame
    bool odd = bg && !(fabsf(bg[0]) <= kTame && fabsf(bg[1]) <= kTame && fabsf(bg[2]) <= kTame);
    {
        float t[2 * H], e0[2 * H], e1[2 * H], e2[2 * H], u[2 * H];
#pragma unroll
        for (int k = 0; k < 2 * H; k++) {
            t[k] = 1.0f; e0[k] = 0.f; e1[k] = 0.f; e2[k] = 0.f; u[k] = 0.f; nl[k] = 0;
            if (px < vd.W && py + RS * k < vd.H) {
                const int64_t pix = vd.pix_base + (int64_t)(py + RS * k) * vd.W + px;
                nl[k] = (int)nlast[pix];
                t[k] = tfinal[pix];
                e0[k] = dl[3 * pix]; e1[k] = dl[3 * pix + 1]; e2[k] = dl[3 * pix + 2];
                odd |= !(fabsf(e0[k]) <= kTame && fabsf(e1[k]) <= kTame && fabsf(e2[k]) <= kTame);
                if (bg) u[k] = t[k] * fmaf(e0[k], bg[0], fmaf(e1[k], bg[1], e2[k] * bg[2]));
            }
        }
#pragma unroll
        for (int h = 0; h < H; h++) {
            Th[h] = f2(t[2 * h], t[2 * h + 1]);
            Tl[h] = zero;
            nU[h] = f2(-u[2 * h], -u[2 * h + 1]);
            d0[h] = f2(e0[2 * h], e0[2 * h + 1]);
            d1[h] = f2(e1[2 * h], e1[2 * h + 1]);
            d2[h] = f2(e2[2 * h], e2[2 * h + 1]);
        }
        int mx = max(nl[0], nl[1]);
        if (H == 2) mx = max(mx, max(nl[2 * H - 2], nl[2 * H - 1]));
#pragma unroll
        for (int o = GL / 2; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane % GL == 0) smax[blk] = mx;
    }
    odd = __syncthreads_or(odd);
    int L = 0;
#pragma unroll
    for (int i = 0; i < NB; i++) L = max(L, smax[i]);
    L = min(L, (int)(r.y - r.x));

    // Batches from the back, double-buffered: the records of the batch below
    // are copied into the other buffer while this batch is walked, and turned
    // into staged entries in place by the thread that copied them before the
    // barrier that ends the walk.  An entry's mask keeps the blocks it can
    // contribute to and one of whose pixels blended at or past it; its slots
    // follow those of the entries behind it.
    uint32_t pid_next[IPT], e_next[IPT];
    auto fetch = [&](int b, int buf) {     // records of batch b (pid_next), indices of the one below
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const int i = tid + u * NT;
            if (i < BB && b + i < L) {
                rec_copy_async(sE[buf][i], rec, pid_next[u], V.pairs, status);
                e_next[u] = vals_sorted[r.x + b + i];
            }
            if (i < BB && b >= BB) pid_next[u] = pid_sorted[r.x + b - BB + i];
        }
    };
    auto stage = [&](int b, int buf) {
        copy_async_wait();
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const int i = tid + u * NT;
            if (i < BB) {            // whole warps
                uint32_t m = 0;
                bool flag = false;
                if (b + i < L) {
                    const float4 qa = sE[buf][i][0], qb = sE[buf][i][1], qc = sE[buf][i][2];
                    sE[buf][i][0] = pair_coefs(tile_mean(qa.x, qc.z, ox), tile_mean(qa.y, qc.w, oy), qa.z, qa.w, qb.x);
                    sE[buf][i][1] = make_float4(pair_c2(qb.x), qb.y, qc.x, qc.x);
                    sE[buf][i][2] = make_float4(qb.z, qb.z, qb.w, qb.w);
                    // o <= 0.98 and a conic conditioned well enough that the
                    // exponent stays below 1e-6: o 2^p < 0.99 at every pixel
                    const float ac = qa.z * qb.x;
                    flag = odd || !(qb.y <= 0.98f) || !(ac < 1e4f * (ac - qa.w * qa.w)) ||
                           !(fabsf(qb.z) <= kTame && fabsf(qb.w) <= kTame && fabsf(qc.x) <= kTame);
                    sQ[buf][0][i] = qa.z;
                    sQ[buf][1][i] = qa.w;
                    sQ[buf][2][i] = qb.x;
                    sSlot[buf][i] = e_next[u];
#pragma unroll
                    for (int k = 0; k < NB; k++) m |= b + i < smax[k] ? 1u << k : 0u;
                    uint32_t q = block_mask<TW, TH, 8>(qa.x - ((float)ox + 0.5f), qa.y - ((float)oy + 0.5f), qa.z, qa.w,
                                                       qb.x, qb.y);
                    if constexpr (BH == 8) {     // two rows of 8x4 blocks are one
                        q |= q >> NC;
                        uint32_t f = 0;
#pragma unroll
                        for (int y = 0; y < TH / 8; y++) f |= (q >> (2 * NC * y) & ((1u << NC) - 1u)) << (NC * y);
                        q = f;
                    }
                    m &= q;
                }
                sM[buf][i] = m;
                const uint32_t c = __popc(m);
                uint32_t x = c;             // inclusive sum over this and the higher lanes
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_down_sync(0xffffffffu, x, o);
                    if (lane + o < 32) x += y;
                }
                sBase[buf][i] = x - c;
                flag = __any_sync(0xffffffffu, flag);
                if (lane == 0) sTot[buf][i >> 5] = x | (flag ? 0x80000000u : 0u);
            }
        }
    };
    int bb = ((L + BB - 1) / BB - 1) * BB;
    if (bb >= 0) {
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const int i = tid + u * NT;
            pid_next[u] = i < BB && bb + i < L ? pid_sorted[r.x + bb + i] : 0u;
        }
        fetch(bb, 0);
        stage(bb, 0);
        if (bb > 0) fetch(bb - BB, 1);
    }
    __syncthreads();
    const int vi = group_sum_index<GL>(lane);
    char* const pbase = reinterpret_cast<char*>(part) + 4 * vi;
    for (int cur = 0; bb >= 0; cur ^= 1) {
        const int cnt = min(BB, L - bb);
        uint32_t total = 0, flags = 0;
#pragma unroll
        for (int c = 0; c < BB / 32; c++) {
            total += sTot[cur][c] & 0x7fffffffu;
            flags |= sTot[cur][c] >> 31;
        }
        // last blended entries relative to the batch, as staged byte offsets
        int nb[2 * H];
#pragma unroll
        for (int k = 0; k < 2 * H; k++) nb[k] = kEnt * max(-1, min(nl[k] - bb, BB));
        const char* __restrict__ cE = reinterpret_cast<const char*>(sE[cur]);
        // passes of at most S slots (nearly always one)
        for (uint32_t first = 0;;) {
            uint32_t next = total;
            int ng[NG];
#pragma unroll
            for (int g = 0; g < NG; g++) ng[g] = 0;
            uint32_t above = 0;      // slots of the higher 32-entry runs
            if (total - first > (uint32_t)S) next = first;
#pragma unroll
            for (int c = BB / 32 - 1; c >= 0; c--) {
                const int i = 32 * c + lane;
                const uint32_t m0 = sM[cur][i], base = above + sBase[cur][i], end = base + __popc(m0);
                const bool in = base >= first && end <= first + S;
                const uint32_t m = in ? m0 : 0u;
                if (in) next = max(next, end);
                above += sTot[cur][c] & 0x7fffffffu;
                const uint32_t q = m >> (NG * w);
                const uint32_t s0 = base - first + __popc(m & ((1u << (NG * w)) - 1u));
#pragma unroll
                for (int g = 0; g < NG; g++) {
                    const uint32_t bal = __ballot_sync(0xffffffffu, q & (1u << g));
                    if (q & (1u << g))
                        slist[NG * w + g][ng[g] + __popc(bal & (0xfffffffeu << lane))] =
                            (uint32_t)(kEnt * i) | (36u * (s0 + __popc(q & ((1u << g) - 1u)))) << 16;
                    ng[g] += __popc(bal);
                }
            }
            if (total - first > (uint32_t)S) next = __reduce_max_sync(0xffffffffu, next);
            int n = ng[0], nmax = ng[0];
#pragma unroll
            for (int g = 1; g < NG; g++) {
                n = grp == g ? ng[g] : n;
                nmax = max(nmax, ng[g]);
            }
            uint32_t* lp = slist[blk];
            for (int i = n + lane % GL; i <= nmax; i += GL) lp[i] = (uint32_t)(kEnt * BB) | (36u * (S + blk)) << 16;
            __syncwarp();
            // (without a flag alpha needs no clamp and every product is finite)
            auto walk = [&](auto careful_t) {
            constexpr bool careful = decltype(careful_t)::value;
            uint32_t ent = lp[0];
#pragma unroll 1
            for (int i = 0; i < nmax; i++) {
                const uint32_t off = ent & 0xffffu, so = ent >> 16;
                ent = lp[i + 1];
                const float4* __restrict__ e = reinterpret_cast<const float4*>(cE + off);
                const float4 a = e[0];
                const float4 b = e[1];
                const float4 rg = e[2];
                const float dx = pix_offset(fx, a.x);
                const PowX px2 = pair_power2_x(dx, a.z, a.w);   // shared by the lane's pixels
                const float2 dx2 = f2(dx, dx);
                float2 g9[9];         // sums over the lane's pairs
#pragma unroll
                for (int h = 0; h < H; h++) {
                    const float2 dy = f2(pix_offset(fy + (float)(RS * 2 * h), a.y),
                                         pix_offset(fy + (float)(RS * (2 * h + 1)), a.y));
                    const float p0 = pair_power2_y(px2, dy.x, b.x), p1 = pair_power2_y(px2, dy.y, b.x);
                    float2 G = f2(ex2_approx(p0), ex2_approx(p1));
                    float2 as = f2(__fmul_rn(b.y, G.x), __fmul_rn(b.y, G.y));
                    const bool h0 = (int)off < nb[2 * h] && p0 >= kPow2Min && as.x >= kAlphaMin;
                    const bool h1 = (int)off < nb[2 * h + 1] && p1 >= kPow2Min && as.y >= kAlphaMin;
                    // a pixel that does not blend takes alpha = 0: T and U stay, its
                    // sums are zero (selected, so that nothing non-finite gets in)
                    G = f2(h0 ? G.x : 0.f, h1 ? G.y : 0.f);
                    as = f2(h0 ? as.x : 0.f, h1 ? as.y : 0.f);
                    float2 al = as;
                    if constexpr (careful) al = f2(fminf(kAlphaMax, as.x), fminf(kAlphaMax, as.y));
                    // compensated T before this entry (div_one_minus on both pixels;
                    // nom = -(1 - alpha), ne = -om_err)
                    const float2 nom = sub2(al, one);
                    const float2 ne = sub2(al, add2(nom, one));
                    const float2 rc = f2(rcp_approx(-nom.x), rcp_approx(-nom.y));
                    const float2 q = mul2(Th[h], rc);
                    Tl[h] = mul2(fma2(q, ne, add2(fma2(q, nom, Th[h]), Tl[h])), rc);
                    Th[h] = q;
                    const float2 wgt = mul2(al, q);
                    const float2 dcol =
                        fma2(d0[h], f2(rg.x, rg.y), fma2(d1[h], f2(rg.z, rg.w), mul2(d2[h], f2(b.z, b.w))));
                    float2 da = fma2(q, dcol, mul2(nU[h], rc));
                    if (h0) nU[h].x = fmaf(-wgt.x, dcol.x, nU[h].x);
                    if (h1) nU[h].y = fmaf(-wgt.y, dcol.y, nU[h].y);
                    float2 t6 = mul2(wgt, d0[h]), t7 = mul2(wgt, d1[h]), t8 = mul2(wgt, d2[h]);
                    if constexpr (careful) {
                        // no gradient where the 0.99 clamp holds
                        da = f2(h0 && as.x <= kAlphaMax ? da.x : 0.f, h1 && as.y <= kAlphaMax ? da.y : 0.f);
                        t6 = f2(h0 ? t6.x : 0.f, h1 ? t6.y : 0.f);
                        t7 = f2(h0 ? t7.x : 0.f, h1 ? t7.y : 0.f);
                        t8 = f2(h0 ? t8.x : 0.f, h1 ? t8.y : 0.f);
                    }
                    // moments of dp = dL/dpower; the conic and the constant factors
                    // are applied per entry
                    const float2 dp = mul2(da, as);
                    if constexpr (BH == 8) {
                        // the sums of two lanes of k_raster_bwd_px, a pixel after the other
                        const float2 y = mul2(dy, dp);
                        if (h == 0) {
                            g9[0] = dp;
                            g9[1] = y;
                            g9[4] = mul2(dy, y);
                            g9[5] = mul2(da, G);
                            g9[6] = t6;
                            g9[7] = t7;
                            g9[8] = t8;
                        } else {
                            g9[0] = fma2(dp, one1, g9[0]);
                            g9[1] = fma2(y, one1, g9[1]);
                            g9[4] = fma2(dy, y, g9[4]);
                            g9[5] = fma2(da, G, g9[5]);
                            float2 s6 = fma2(wgt, d0[h], g9[6]), s7 = fma2(wgt, d1[h], g9[7]),
                                   s8 = fma2(wgt, d2[h], g9[8]);
                            if constexpr (careful) {
                                s6 = f2(h0 ? s6.x : g9[6].x, h1 ? s6.y : g9[6].y);
                                s7 = f2(h0 ? s7.x : g9[7].x, h1 ? s7.y : g9[7].y);
                                s8 = f2(h0 ? s8.x : g9[8].x, h1 ? s8.y : g9[8].y);
                            }
                            g9[6] = s6;
                            g9[7] = s7;
                            g9[8] = s8;
                            g9[0] = mul2(g9[0], dx2);
                            g9[2] = mul2(dx2, g9[0]);
                            g9[3] = mul2(dx2, g9[1]);
                        }
                        continue;
                    }
                    float2 t[9];
                    t[0] = mul2(dp, dx2);
                    t[1] = mul2(dy, dp);
                    t[2] = mul2(dx2, t[0]);
                    t[3] = mul2(dx2, t[1]);
                    t[4] = mul2(dy, t[1]);
                    t[5] = mul2(da, G);
                    t[6] = t6;
                    t[7] = t7;
                    t[8] = t8;
#pragma unroll
                    for (int k = 0; k < 9; k++) g9[k] = h ? fma2(t[k], one1, g9[k]) : t[k];
                }
                float g[9];
#pragma unroll
                for (int k = 0; k < 9; k++) g[k] = __fadd_rn(g9[k].x, g9[k].y);
                float p, q2;
                group_sums<GL>(g, lane, p, q2);
                if (GL == 8 || vi >= 0) *reinterpret_cast<float*>(pbase + so) = p;
                if (GL == 8 && (lane & 7) == 0) *reinterpret_cast<float*>(pbase + so + 8) = q2;
            }
            };
            if (flags) walk(std::true_type{});
            else walk(std::false_type{});
            const bool more = next < total;
            if (!more && bb > 0) stage(bb - BB, cur ^ 1);
            __syncthreads();
            // one thread per entry adds its slots in block order and writes the
            // record: slots 0-4 hold sums of dp (dx, dy, dx^2, dx dy, dy^2):
            // dL/dmean = conic (sum dx dp, sum dy dp) and dL/dconic =
            // -(sum dx^2 dp / 2, sum dx dy dp, sum dy^2 dp / 2)
#pragma unroll
            for (int u = 0; u < IPT; u++) {
                const int j = tid + u * NT;
                if (j < cnt) {
                    uint32_t base = sBase[cur][j];
                    for (int c = (j >> 5) + 1; c < BB / 32; c++) base += sTot[cur][c] & 0x7fffffffu;
                    const uint32_t nsl = __popc(sM[cur][j]);
                    if (base >= first && base + nsl <= first + S) {
                        float sm[9];
#pragma unroll
                        for (int c = 0; c < 9; c++) sm[c] = 0.f;
                        for (uint32_t k = base - first; k < base - first + nsl; k++)
#pragma unroll
                            for (int c = 0; c < 9; c++) sm[c] += part[k][c];
                        const float ca = sQ[cur][0][j], cb = sQ[cur][1][j], cc = sQ[cur][2][j];
                        const uint32_t e = sSlot[cur][j];
                        if (GS_DCHECK(e < cap, status)) {
                            float4* o = reinterpret_cast<float4*>(gradrec + e);
                            o[0] = make_float4(fmaf(ca, sm[0], cb * sm[1]), fmaf(cb, sm[0], cc * sm[1]),
                                               -0.5f * sm[2], -sm[3]);
                            o[1] = make_float4(-0.5f * sm[4], sm[5], sm[6], sm[7]);
                            reinterpret_cast<float*>(o + 2)[0] = sm[8];
                        }
                    }
                }
            }
            first = next;
            if (!more) break;
            __syncthreads();
        }
        bb -= BB;
        if (bb > 0) fetch(bb - BB, cur);   // this batch's entries are not read any more
        __syncthreads();
    }
    // entries past every pixel's last blended pair receive zero gradients
    for (uint32_t k = r.x + (uint32_t)L + tid; k < r.y; k += NT) {
        GradRec o;
        o.a = o.b = o.c = make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t e = vals_sorted[k];
        if (GS_DCHECK(e < cap, status)) gradrec[e] = o;
    }
}

void launch_raster_bwd_px(const Plan& P, const WsPtrs& w, const float* bg, const float* dl, cudaStream_t st);

void launch_raster_bwd(const Plan& P, const WsPtrs& w, const float* image, const float* dl, cudaStream_t st)
{
    if (P.tuning.bwd_impl == 0 || P.tuning.bwd_impl == 2) {
        const float* bg = reinterpret_cast<const float*>(reinterpret_cast<const char*>(w.hdr) + offsetof(WsHeader, bg));
        if (P.tuning.bwd_impl == 0) launch_raster_bwd_px(P, w, bg, dl, st);
        else launch_raster_bwd2(P, w, bg, dl, st);
        return;
    }
    const Views& V = P.views;
    const int np = V.tw * V.th;
    const unsigned grid = (unsigned)V.tiles;
    const int fixed = P.tuning.bwd_batch;
#define GS_RB(NP)                                                                                           \
    do {                                                                                                    \
        const size_t sb = bwd_smem_bytes(NP);                                                               \
        static bool attr_set = false;                                                                       \
        if (!attr_set) {                                                                                    \
            cudaFuncSetAttribute(k_raster_bwd<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sb);   \
            attr_set = true;                                                                                \
        }                                                                                                   \
        launch_after(k_raster_bwd<NP>, grid, kBwdThreads, sb, st, V, w.tile_order, w.ranges, w.vals_sorted, \
                     w.pid_sorted, w.rec, image, dl, w.nlast, w.gradrec, fixed);                            \
    } while (0)
    if (np == 64) GS_RB(64);
    else if (np == 256) GS_RB(256);
    else GS_RB(512);
#undef GS_RB
}

}  // namespace gs

// ===========================================================================
// Second implementation: pixels across threads, per-Gaussian gradients
// reduced across each warp's pixels by shuffles (no atomics).
//
// One CTA per tile, one, two or four pixels per thread, each warp an 8x4, 8x8 or
// 8x16 pixel block (so a small Gaussian touches few warps).  This form runs for 8x8
// tiles, for four pixels per thread and where a few long lists are the launch's time;
// the others walk blocks by lane groups (k_raster_bwd_blocks).  Every pixel walks its own
// list prefix back to front from its last blended entry: T before an entry is recovered
// by a compensated division of T after it by (1 - alpha) (div_one_minus:
// hardware reciprocal, exact remainder, carried low part), and the colour
// still to come S grows from T_final * bg without cancellation; only its
// projection U = dL/dC . S is carried, since dL/dalpha needs no more.  The
// list is staged BB entries at a time with a mask of the warp blocks each
// entry's 3-sigma box touches; a warp visits only its entries, and for an
// entry that
// at least one of its pixels blended it sums nine values over its 32 pixels
// with a halving butterfly (12 shuffles; afterwards nine lanes each hold one
// fully reduced value) into its own shared-memory slot: the opacity and
// colour gradients and the moments dx dp, dy dp, dx^2 dp, dx dy dp, dy^2 dp
// of dp = dL/dpower, from which the mean and conic gradients follow per
// entry (the mean gradient is the conic times the first two).  After each
// batch the warps' slots are added in warp order and written to each entry's
// emission slot, so the result does not depend on scheduling.
// ===========================================================================

namespace gs {

// Halving-butterfly reduction of nine per-lane values over a warp: returns
// the lane's share of the result; `vi` (from bfly_index) says which of the
// nine sums it is (-1: none).
__device__ __forceinline__ float bfly9(const float* v, int lane)
{
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4, h1 = lane & 2;
    float k[5];
#pragma unroll
    for (int i = 0; i < 5; i++) {
        const float lo = v[i], hi = i < 4 ? v[5 + i] : 0.f;
        k[i] = (h4 ? hi : lo) + __shfl_xor_sync(0xffffffffu, h4 ? lo : hi, 16);
    }
    float m[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const float lo = k[i], hi = i < 2 ? k[3 + i] : 0.f;
        m[i] = (h3 ? hi : lo) + __shfl_xor_sync(0xffffffffu, h3 ? lo : hi, 8);
    }
    float nn[2];
#pragma unroll
    for (int i = 0; i < 2; i++) {
        const float lo = m[i], hi = i < 1 ? m[2 + i] : 0.f;
        nn[i] = (h2 ? hi : lo) + __shfl_xor_sync(0xffffffffu, h2 ? lo : hi, 4);
    }
    float p = (h1 ? nn[1] : nn[0]) + __shfl_xor_sync(0xffffffffu, h1 ? nn[0] : nn[1], 2);
    return p + __shfl_xor_sync(0xffffffffu, p, 1);
}

__device__ __forceinline__ int bfly_index(int lane)
{
    if (lane & 1) return -1;
    const int mi = ((lane & 4) ? 2 : 0) + ((lane & 2) ? 1 : 0);
    if (mi == 3) return -1;
    const int ki = (lane & 8) ? (mi < 2 ? 3 + mi : -1) : mi;
    if (ki < 0) return -1;
    return (lane & 16) ? (ki < 4 ? 5 + ki : -1) : ki;
}

// BS threads per tile, each owning PPT pixels of its warp's 8 x (4 PPT)
// block (lane (x, y) holds rows y, y + 4, ...): the PPT pixels' nine values
// are summed in the lane before one butterfly per visit.
template <int BS, int TW, int PPT>
__global__ void __launch_bounds__(BS) k_raster_bwd_px(Views V, const uint32_t* __restrict__ order,
                                                      const uint2* __restrict__ ranges,
                                                      const uint32_t* __restrict__ vals_sorted,
                                                      const uint32_t* __restrict__ pid_sorted,
                                                      const ProjRec* __restrict__ rec,
                                                      const float* __restrict__ tfinal,
                                                      const float* __restrict__ bg, const float* __restrict__ dl,
                                                      const uint32_t* __restrict__ nlast,
                                                      GradRec* __restrict__ gradrec, uint32_t* __restrict__ status,
                                                      uint32_t cap)
{
    if (!after_previous()) return;
    constexpr int NW = BS / 32;
    constexpr int BH = 4 * PPT;            // warp block height, pixels
    constexpr int TH = BS * PPT / TW;      // tile height, pixels
    constexpr int WPR = TW / 8;            // warp blocks per tile row
    constexpr int RPB = TH / BH;           // rows of warp blocks
    constexpr int BB = NW <= 8 ? 96 : 64;  // list entries per staged batch
    constexpr int IPT = (BB + BS - 1) / BS;   // staged entries per thread
    __shared__ float4 sA[2][BB];
    __shared__ float4 sB[2][BB];
    __shared__ float4 sD[2][BB];          // (conic a, b, c, blue)
    __shared__ uint32_t sE[2][BB];
    __shared__ uint32_t sM[2][BB];
    __shared__ float part[NW][BB][9];
    __shared__ int smax[NW];

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int64_t gt = order[blockIdx.x];   // longest lists first
    const int v = view_of_tile(V, gt);
    const ViewDesc& vd = V.v[v];
    const int lt = (int)(gt - vd.tile_base);
    const int ox = (lt % vd.TX) * TW, oy = (lt / vd.TX) * TH;
    const int px = ox + (w % WPR) * 8 + (lane & 7);
    const int py0 = oy + (w / WPR) * BH + (lane >> 3);
    const uint32_t wbit = 1u << w;
    const uint2 r = range_at(ranges, gt, cap, status);
    // pixel centres relative to the tile's first pixel (the staged means are too)
    const float fx = (float)(px - ox) + 0.5f;
    const int vi = bfly_index(lane);

    // per pixel k (row py0 + 4k): last blended entry, compensated T after
    // it, dL/dC, and U = sum_c dL/dC_c S_c with S_c the colour still to come
    // behind an entry (from T_final bg_c): dL/dalpha = T dL/dC . col -
    // U / (1 - alpha)
    uint32_t nl[PPT];
    float Th[PPT], Tl[PPT], d0[PPT], d1[PPT], d2[PPT], U[PPT], fy[PPT];
    int mx_nl = 0;
#pragma unroll
    for (int k = 0; k < PPT; k++) {
        const int py = py0 + 4 * k;
        fy[k] = (float)(py - oy) + 0.5f;
        nl[k] = 0;
        Th[k] = 1.f; Tl[k] = 0.f; d0[k] = 0.f; d1[k] = 0.f; d2[k] = 0.f; U[k] = 0.f;
        if (px < vd.W && py < vd.H) {
            const int64_t pix = vd.pix_base + (int64_t)py * vd.W + px;
            nl[k] = nlast[pix];
            Th[k] = tfinal[pix];
            d0[k] = dl[3 * pix]; d1[k] = dl[3 * pix + 1]; d2[k] = dl[3 * pix + 2];
        }
        if (bg) U[k] = Th[k] * fmaf(d0[k], bg[0], fmaf(d1[k], bg[1], d2[k] * bg[2]));
        mx_nl = max(mx_nl, (int)nl[k]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx_nl = max(mx_nl, __shfl_xor_sync(0xffffffffu, mx_nl, o));
    if (lane == 0) smax[w] = mx_nl;
    __syncthreads();
    int L = 0;
#pragma unroll
    for (int i = 0; i < NW; i++) L = max(L, smax[i]);
    L = min(L, (int)(r.y - r.x));

    // Batches from the back; the batch below the current one is gathered into
    // registers while the current one is processed, then stored to the other
    // buffer: two barriers per batch.  An entry's mask keeps the warps whose
    // block its box touches and one of whose pixels blended at or past it:
    // exactly the warps that visit it.
    auto stage = [&](int bbx, int buf, int i, const ProjRec& q, uint32_t e) {
        uint32_t live = 0;
#pragma unroll
        for (int k = 0; k < NW; k++) live |= (bbx + i < smax[k] ? 1u : 0u) << k;
        sA[buf][i] = pair_coefs(tile_mean(q.a.x, q.c.z, ox), tile_mean(q.a.y, q.c.w, oy), q.a.z, q.a.w, q.b.x);
        sB[buf][i] = make_float4(pair_c2(q.b.x), q.b.y, q.b.z, q.b.w);
        sD[buf][i] = make_float4(q.a.z, q.a.w, q.b.x, q.c.x);
        sE[buf][i] = e;
        sM[buf][i] = warp_block_mask(q.a.x, q.a.y, q.a.z, q.a.w, q.b.x, q.b.y, ox, oy, WPR, RPB, BH) & live;
    };
    int bb = ((L + BB - 1) / BB - 1) * BB;
    if (bb >= 0) {
        const int cnt0 = min(BB, L - bb);
        for (int i = tid; i < cnt0; i += BS) {
            const uint32_t k = r.x + bb + i;
            stage(bb, 0, i, rec_at(rec, pid_sorted[k], V.pairs, status), vals_sorted[k]);
        }
    }
    __syncthreads();
    for (int cur = 0; bb >= 0; bb -= BB, cur ^= 1) {
        const int cnt = min(BB, L - bb);
        const float4* __restrict__ cA = sA[cur];
        const float4* __restrict__ cB = sB[cur];
        const float4* __restrict__ cD = sD[cur];
        const uint32_t* __restrict__ cM = sM[cur];
        // gathers for the next (lower) batch, all entries full since bb > 0
        ProjRec qn[IPT];
        uint32_t en[IPT];
        if (bb > 0) {
#pragma unroll
            for (int u = 0; u < IPT; u++) {
                const int i = tid + u * BS;
                if (i < BB) {
                    const uint32_t k = r.x + bb - BB + i;
                    en[u] = vals_sorted[k];
                    qn[u] = rec_at(rec, pid_sorted[k], V.pairs, status);
                }
            }
        }
        for (int c = (cnt - 1) >> 5; c >= 0; c--) {
            // entries of this chunk whose box touches this warp's block,
            // before the last pair any of the warp's pixels blended
            const int jl = 32 * c + lane;
            uint32_t bits = __ballot_sync(0xffffffffu, jl < cnt && (cM[jl] & wbit));
            while (bits) {
                const int jj = 31 - __clz(bits);
                bits &= ~(1u << jj);
                const int j = 32 * c + jj;
                const float4 a = cA[j];
                const float4 b = cB[j];
                const float dx = pix_offset(fx, a.x);
                const PowX px2 = pair_power2_x(dx, a.z, a.w);   // shared by the lane's pixels
                // the skip tests of the lane's pixels first; the nine sums
                // are zeroed and formed only when a pixel of the warp blends
                float dyk[PPT], Gk[PPT], ak[PPT];
                bool hk[PPT], any = false;
#pragma unroll
                for (int k = 0; k < PPT; k++) {
                    dyk[k] = pix_offset(fy[k], a.y);
                    const float p2 = pair_power2_y(px2, dyk[k], b.x);
                    Gk[k] = ex2_approx(p2);
                    ak[k] = __fmul_rn(b.y, Gk[k]);
                    // one test for the pixel's three skips (exp2 taken for
                    // every pixel): no nested divergent branches
                    hk[k] = bb + j < (int)nl[k] && p2 >= kPow2Min && ak[k] >= kAlphaMin;
                    any |= hk[k];
                }
                float x = 0.f;
                if (__any_sync(0xffffffffu, any)) {
                    float g[9];
#pragma unroll
                    for (int i = 0; i < 9; i++) g[i] = 0.f;
#pragma unroll
                    for (int k = 0; k < PPT; k++) {
                        if (!hk[k]) continue;
                        const float araw = ak[k], G = Gk[k], dy = dyk[k];
                        const float alpha = fminf(kAlphaMax, araw);
                        const float cb = cD[j].w;
                        // compensated T before this entry
                        const float rom = div_one_minus(alpha, Th[k], Tl[k]);
                        const float wgt = alpha * Th[k];
                        g[6] = fmaf(wgt, d0[k], g[6]);
                        g[7] = fmaf(wgt, d1[k], g[7]);
                        g[8] = fmaf(wgt, d2[k], g[8]);
                        const float dcol = fmaf(d0[k], b.z, fmaf(d1[k], b.w, d2[k] * cb));
                        const float da = fmaf(Th[k], dcol, -U[k] * rom);
                        U[k] = fmaf(wgt, dcol, U[k]);
                        // moments of dp = dL/dpower (zero where the 0.99
                        // clamp holds); the conic and the constant factors
                        // are applied per entry after the reduction
                        const float dam = araw <= kAlphaMax ? da : 0.f;
                        g[5] = fmaf(dam, G, g[5]);
                        const float dp = dam * araw;
                        const float ydp = dy * dp;
                        g[0] += dp;
                        g[1] += ydp;
                        g[4] = fmaf(dy, ydp, g[4]);
                    }
                    // the lane's pixels share dx: sum dx dp = dx S, sum dx^2 dp
                    // = dx (dx S), sum dx dy dp = dx sum dy dp
                    g[0] *= dx;
                    g[2] = dx * g[0];
                    g[3] = dx * g[1];
                    x = bfly9(g, lane);
                }
                // every visiting warp fills its slot (zeros when none of its
                // pixels blended the entry)
                if (vi >= 0) part[w][j][vi] = x;
            }
        }
        __syncthreads();
        // one thread per entry adds the visiting warps' partial sums in warp
        // order and writes the entry's record (two 16-byte stores and one
        // 4-byte store).  Slots 0-4 hold sums of dp (dx, dy, dx^2, dx dy,
        // dy^2): dL/dmean = conic (sum dx dp, sum dy dp) and dL/dconic =
        // -(sum dx^2 dp / 2, sum dx dy dp, sum dy^2 dp / 2).
        for (int j = tid; j < cnt; j += BS) {
            float sm[9];
#pragma unroll
            for (int c = 0; c < 9; c++) sm[c] = 0.f;
            for (uint32_t m = sM[cur][j]; m; m &= m - 1u) {     // visiting warps, in warp order
                const int i = __ffs(m) - 1;
#pragma unroll
                for (int c = 0; c < 9; c++) sm[c] += part[i][j][c];
            }
            const float4 cd = sD[cur][j];
            const uint32_t e = sE[cur][j];
            if (GS_DCHECK(e < cap, status)) {
                float4* o = reinterpret_cast<float4*>(gradrec + e);
                o[0] = make_float4(fmaf(cd.x, sm[0], cd.y * sm[1]), fmaf(cd.y, sm[0], cd.z * sm[1]), -0.5f * sm[2],
                                   -sm[3]);
                o[1] = make_float4(-0.5f * sm[4], sm[5], sm[6], sm[7]);
                reinterpret_cast<float*>(o + 2)[0] = sm[8];
            }
        }
        if (bb > 0) {
#pragma unroll
            for (int u = 0; u < IPT; u++) {
                const int i = tid + u * BS;
                if (i < BB) stage(bb - BB, cur ^ 1, i, qn[u], en[u]);
            }
        }
        __syncthreads();
    }
    // entries past every pixel's last blended pair receive zero gradients
    for (uint32_t k = r.x + (uint32_t)L + tid; k < r.y; k += BS) {
        GradRec o;
        o.a = o.b = o.c = make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t e = vals_sorted[k];
        if (GS_DCHECK(e < cap, status)) gradrec[e] = o;
    }
}

void launch_raster_bwd_px(const Plan& P, const WsPtrs& w, const float* bg, const float* dl, cudaStream_t st)
{
    const Views& V = P.views;
    const unsigned grid = (unsigned)V.tiles;
    const int ppt = tile_ppt(P);
#define GS_RBP(BS, TW, PPT)                                                                                  \
    launch_after(k_raster_bwd_px<BS, TW, PPT>, grid, BS, 0, st, V, w.tile_order, w.ranges, w.vals_sorted,    \
                 w.pid_sorted, w.rec, w.tfinal, bg, dl, w.nlast, w.gradrec, &w.hdr->status,                  \
                 (uint32_t)P.cap)
#define GS_RBB(TW, TH, GL, BH)                                                                                   \
    launch_after(k_raster_bwd_blocks<TW, TH, GL, BH>, grid, BwdBlocks<TW, TH, GL, BH>::kThreads, 0, st, V,         \
                 w.tile_order, w.ranges, w.vals_sorted, w.pid_sorted, w.rec, w.tfinal, bg, dl, w.nlast,      \
                 w.gradrec, &w.hdr->status, (uint32_t)P.cap)
    // 16-wide tiles with one pixel per thread (the default) walk 8x4 blocks by lane
    // groups, and so do two pixels per thread with BF16 moments (their error against 64
    // bits is that of the other order of summation, 4.1e-7 to 2.6e-6 of the records' RMS;
    // FP32 moments keep the order).  All kernels of one order write the same bits, so a
    // grid takes the one that suits it (us, measured on rooms of 10 m and sites of 30 m,
    // 20,000 to 3M Gaussians, 64x64 to 1920x1080):
    //  - GL = 8 (four visits per warp) needs two waves of resident blocks to hide a tile's
    //    chain, else GL = 16: 200k Gaussians on 3,600 tiles 101 / 116, 5,700 tiles 57 / 72,
    //    2,040 tiles 141 / 111 (400k).  The tile count alone does not separate them: where
    //    few of the tiles are long, GL = 16 is faster up to about 4,000 tiles (1M site on
    //    3,600 tiles 254 against 229, 400k on 3,600 110 against 98).
    //  - Below that, lists so long that one tile's chain is the launch's time take a warp
    //    per block: 200k on 60 tiles 867 -> 776, 1M on 60 2,416 -> 1,660, 1M on 240
    //    986 -> 889; but 400k on 240 510 / 576.  (16x32 tiles have 16 warps and take it
    //    later: 400k on 30 2,097 -> 1,863, 400k on 75 1,172 / 1,251.)
    //  - Two pixels per thread, FP32: 8x8 blocks from two waves on (400k room on 3,600
    //    tiles 266 -> 214, 3M on 8,160 960 -> 827; sites on 3,600 within 1%) and for
    //    short lists (20k on 920 tiles 24.8 -> 23.2); in between a warp per block is
    //    faster (1M on 240 tiles 1,284 against 1,748, 3M on 2,040 739 against 864).
    //    16x32 tiles: from three waves on (1M on 2,900 tiles 347 -> 312), from two with
    //    short lists (1,840 tiles: 400k room 281 -> 236, 400k site 145 / 159, 3M 841 / 938).
    const bool blocks = ppt == 1 || (ppt == 2 && P.mom_bf16), tall = V.th == 32;
    const int64_t wave = (int64_t)P.sm_count * BwdBlocks<16, 16, 8, 4>::kBlocksPerSM * 256 / (V.tw * V.th);
    const bool full = V.tiles >= 2 * wave;
    const bool few_long = !full && V.pairs >= (tall ? 12288 : 2560) * V.tiles;
    const bool blocks8 = tall ? V.tiles >= 3 * wave || (full && V.pairs <= 256 * V.tiles)
                              : full || V.pairs <= 384 * V.tiles;
    if (V.tw == 8) {
        if (ppt == 1) GS_RBP(64, 8, 1);
        else GS_RBP(32, 8, 2);
    } else if (!tall) {
        if (blocks && full) GS_RBB(16, 16, 8, 4);
        else if (blocks && few_long) GS_RBP(256, 16, 1);
        else if (blocks) GS_RBB(16, 16, 16, 4);
        else if (ppt == 2 && blocks8) GS_RBB(16, 16, 16, 8);
        else if (ppt == 2) GS_RBP(128, 16, 2);
        else GS_RBP(64, 16, 4);
    } else {
        if (blocks && full) GS_RBB(16, 32, 8, 4);
        else if (blocks && few_long) GS_RBP(512, 16, 1);
        else if (blocks) GS_RBB(16, 32, 16, 4);
        else if (ppt == 2 && blocks8) GS_RBB(16, 32, 16, 8);
        else if (ppt == 2) GS_RBP(256, 16, 2);
        else GS_RBP(128, 16, 4);
    }
#undef GS_RBP
#undef GS_RBB
}

}  // namespace gs
