// densify.cu -- default densification (VkSplat Sec. 4.6, which follows the
// 3DGS default strategy) and the opacity reset, on the chunk-major scene
// layout.
//
// gs_densify_count decides every Gaussian's fate (kept as is, cloned, split and
// kept) and scans the three counts together into a list of the output rows'
// sources; gs_densify_apply gathers by that list, one thread per output row and
// group of arrays.  Decisions are binary32 comparisons of stored (activated)
// values, so they are exact.
#include <type_traits>

#include "gs_internal.cuh"

namespace gs {

struct DensifyK {
    float grad_thr;     // grow_grad2d
    float small_thr;    // grow_scale3d * scene_scale (binary32 product)
    float prune_opa;
    float big_thr;      // prune_scale3d * scene_scale
    float factor;       // split_factor
    int grow, prune_big;
};

// Fates of a Gaussian, a byte each in the scratch.
constexpr uint32_t kKeep = 1u, kClone = 2u, kSplit = 4u;

struct DensifyScratch {
    int64_t* counts;    // [4]: kept, clones, splits, total
    uint8_t* fate;      // [n, padded to whole blocks]
    uint32_t* part;     // [3][blocks]: kept, clones, splits per block, then their exclusive scans
    uint32_t* src;      // [2 n]: source row of each output row
};

static int64_t ds_blocks(int64_t n) { return (n + kScanBlock - 1) / kScanBlock; }

static size_t ds_align(size_t x) { return (x + 255) & ~(size_t)255; }

static size_t ds_layout(int64_t n, void* base, DensifyScratch* d)
{
    char* p = static_cast<char*>(base);
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = ds_align(o + bytes);
        return p ? p + at : nullptr;
    };
    char* counts = take(4 * sizeof(int64_t));
    char* fate = take((size_t)ds_blocks(n) * kScanBlock);
    char* part = take(3 * 4 * (size_t)ds_blocks(n));
    char* src = take(2 * 4 * (size_t)n);
    if (d) {
        d->counts = reinterpret_cast<int64_t*>(counts);
        d->fate = reinterpret_cast<uint8_t*>(fate);
        d->part = reinterpret_cast<uint32_t*>(part);
        d->src = reinterpret_cast<uint32_t*>(src);
    }
    return o;
}

// The three counts of up to 2^20 Gaussians in one 64-bit word.
__device__ __forceinline__ unsigned long long ds_pack(uint32_t f)
{
    return (unsigned long long)(f & kKeep) | (unsigned long long)((f & kClone) >> 1) << 21 |
           (unsigned long long)((f & kSplit) >> 2) << 42;
}
__device__ __forceinline__ uint32_t ds_count(unsigned long long x, int k) { return (uint32_t)(x >> (21 * k)) & 0x1FFFFFu; }

// Fates of one scan block's Gaussians, and its three counts.
__global__ void __launch_bounds__(kScanThreads) k_densify_decide(int64_t n, const float4* __restrict__ geom,
                                                                 const float2* __restrict__ stats, DensifyK K,
                                                                 uint8_t* __restrict__ fate,
                                                                 uint32_t* __restrict__ part)
{
    if (!after_previous()) return;
    __shared__ unsigned long long ws[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanBlock;
    unsigned long long sum = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int64_t i = base + u * kScanThreads + threadIdx.x;
        uint32_t f = 0;
        if (i < n) {
            const float4 so = geom[2 * n + i];
            const float2 st = stats[i];
            const float avg = __fdiv_rn(st.x, fmaxf(st.y, 1.0f));
            const bool high = K.grow && avg > K.grad_thr;
            const float ms = fmaxf(fmaxf(so.x, so.y), so.z);
            const bool small = ms <= K.small_thr;
            const bool clone = high && small, split = high && !small;
            const bool low_o = so.w < K.prune_opa;
            const bool big = K.prune_big && ms > K.big_thr;
            const bool big_split = K.prune_big && __fdiv_rn(ms, K.factor) > K.big_thr;
            f = (!split && !(low_o || big) ? kKeep : 0u) | (clone && !(low_o || big) ? kClone : 0u) |
                (split && !(low_o || big_split) ? kSplit : 0u);
        }
        fate[i] = (uint8_t)f;
        sum += ds_pack(f);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x < 3) {
        unsigned long long t = 0;
        for (int w = 0; w < kScanThreads / 32; w++) t += ws[w];
        part[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = ds_count(t, threadIdx.x);
    }
}

// Single block: exclusive scans of the blocks' three counts, and the totals.
__global__ void __launch_bounds__(1024) k_densify_scan(int64_t blocks, uint32_t* __restrict__ part,
                                                       int64_t* __restrict__ counts)
{
    if (!after_previous()) return;
    __shared__ uint32_t ws[32];
    __shared__ uint32_t tot[3];
    for (int k = 0; k < 3; k++) {
        uint32_t carry = 0;
        for (int64_t b = 0; b < blocks; b += 1024) {
            const int64_t i = b + threadIdx.x;
            const uint32_t v = i < blocks ? part[k * blocks + i] : 0u;
            uint32_t t;
            const uint32_t ex = block_excl_scan<1024>(v, ws, &t);
            if (i < blocks) part[k * blocks + i] = carry + ex;
            carry += t;
            __syncthreads();
        }
        if (threadIdx.x == 0) tot[k] = carry;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int64_t na = tot[0], nb = tot[1], nc = tot[2];
        counts[0] = na;
        counts[1] = nb;
        counts[2] = nc;
        counts[3] = na + nb + 2 * nc;
    }
}

// Source rows of the outputs: thread t takes 8 neighbouring Gaussians of its block.
__global__ void __launch_bounds__(kScanThreads) k_densify_index(const uint8_t* __restrict__ fate,
                                                                const uint32_t* __restrict__ part,
                                                                const int64_t* __restrict__ counts,
                                                                uint32_t* __restrict__ src)
{
    if (!after_previous()) return;
    static_assert(kScanItems == 8, "eight fates in one 64-bit load");
    __shared__ unsigned long long ws[kScanThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * kScanBlock + threadIdx.x * kScanItems;
    const unsigned long long f8 = *reinterpret_cast<const unsigned long long*>(fate + i0);
    unsigned long long own = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; u++) own += ds_pack((uint32_t)(f8 >> (8 * u)) & 7u);
    unsigned long long x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    x -= own;
    for (int k = 0; k < w; k++) x += ws[k];
    const int64_t na = counts[0], nb = counts[1], nc = counts[2];
    const int64_t nblk = gridDim.x;
    int64_t a = part[blockIdx.x] + ds_count(x, 0), b = na + part[nblk + blockIdx.x] + ds_count(x, 1),
            c = na + nb + part[2 * nblk + blockIdx.x] + ds_count(x, 2);
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const uint32_t f = (uint32_t)(f8 >> (8 * u)) & 7u, i = (uint32_t)(i0 + u);
        if (f & kKeep) src[a++] = i;
        if (f & kClone) src[b++] = i;
        if (f & kSplit) {
            src[c + nc] = i;
            src[c++] = i;
        }
    }
}

// Output row j of one group of arrays (blockIdx.y: 0 geometry and statistics, 1 SH,
// 2 and 3 the moments), gathered from row src[j]; the output ranges (kept, clones,
// first and second split products) say what becomes of it.  Bound by HBM: one
// read and one write of every row (2.4 GB at 3M Gaussians, BF16).  A thread per
// input Gaussian that copied its whole row up to three times, lane by lane, took
// 737 us there, this 393 us: neighbouring lanes now write neighbouring rows in
// every range and each thread has the loads of one array in flight.
template <bool SH16, bool MOM16>
__global__ void __launch_bounds__(256) k_densify_apply(SceneDesc in, SceneDesc out, const uint32_t* __restrict__ src,
                                                       const int64_t* __restrict__ counts,
                                                       const float* __restrict__ eps, float factor)
{
    if (!after_previous()) return;
    const int64_t n = in.n, m = out.n;
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m || counts[3] != m) return;   // wrong output size: write nothing
    const int64_t i = src[j];
    const int64_t na = counts[0], nb = counts[1], nc = counts[2];
    if (blockIdx.y == 0) {
        float4 g0 = in.geom[i], g2 = in.geom[2 * n + i];
        const float4 g1 = in.geom[n + i];
        if (j >= na + nb) {
            // R(q) of the normalised quaternion (w, x, y, z), as in the projection
            const float qn = rsqrtf(g1.x * g1.x + g1.y * g1.y + g1.z * g1.z + g1.w * g1.w);
            const float w = g1.x * qn, x = g1.y * qn, y = g1.z * qn, z = g1.w * qn;
            const float R[9] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y),
                                2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x),
                                2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)};
            const float* e = eps + 6 * i + (j >= na + nb + nc ? 3 : 0);
            const float lx = g2.x * e[0], ly = g2.y * e[1], lz = g2.z * e[2];
            g0 = make_float4(g0.x + (R[0] * lx + R[1] * ly + R[2] * lz), g0.y + (R[3] * lx + R[4] * ly + R[5] * lz),
                             g0.z + (R[6] * lx + R[7] * ly + R[8] * lz), g0.w);
            g2 = make_float4(__fdiv_rn(g2.x, factor), __fdiv_rn(g2.y, factor), __fdiv_rn(g2.z, factor), g2.w);
        }
        out.geom[j] = g0;
        out.geom[m + j] = g1;
        out.geom[2 * m + j] = g2;
        if (out.stats) out.stats[j] = make_float2(0.f, 0.f);
    } else if (blockIdx.y == 1) {
        constexpr int C = SH16 ? 6 : 12;      // 16-byte chunks
        const uint4* s = static_cast<const uint4*>(in.sh);
        uint4* d = static_cast<uint4*>(out.sh);
        uint4 x[C];
#pragma unroll
        for (int k = 0; k < C; k++) x[k] = s[k * n + i];
#pragma unroll
        for (int k = 0; k < C; k++) d[k * m + j] = x[k];
    } else {
        // a new Gaussian starts with zero moments
        using M = typename std::conditional<MOM16, uint2, uint4>::type;
        const M* s = static_cast<const M*>(blockIdx.y == 2 ? in.m : in.v);
        M* d = static_cast<M*>(blockIdx.y == 2 ? out.m : out.v);
        M x[15];
#pragma unroll
        for (int k = 0; k < 15; k++) {
            x[k] = M{};
            if (j < na) x[k] = s[k * n + i];
        }
#pragma unroll
        for (int k = 0; k < 15; k++) d[k * m + j] = x[k];
    }
}

template <bool MOM16>
__global__ void k_reset_opacity(SceneDesc sc, float value)
{
    const int64_t n = sc.n;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float4 so = sc.geom[2 * n + i];
    so.w = fminf(so.w, value);
    sc.geom[2 * n + i] = so;
    if (MOM16) {
        uint2* m = static_cast<uint2*>(sc.m);
        uint2* v = static_cast<uint2*>(sc.v);
        m[2 * n + i].y &= 0x0000FFFFu;   // the fourth bf16 is the logit-opacity moment
        v[2 * n + i].y &= 0x0000FFFFu;
    } else {
        static_cast<float4*>(sc.m)[2 * n + i].w = 0.f;
        static_cast<float4*>(sc.v)[2 * n + i].w = 0.f;
    }
}

static SceneDesc ds_scene(const gs_scene_buf& b)
{
    SceneDesc s;
    s.n = b.n;
    s.base = 0;
    s.geom = static_cast<float4*>(b.geom);
    s.sh = b.sh;
    s.m = b.m;
    s.v = b.v;
    s.stats = static_cast<float2*>(b.stats);
    return s;
}

static bool ds_cfg_ok(const gs_densify_cfg* c)
{
    auto fin = [](float x) { return x == x && x - x == 0.0f; };
    return c && fin(c->grow_grad2d) && fin(c->grow_scale3d) && fin(c->prune_opa) && fin(c->prune_scale3d) &&
           fin(c->scene_scale) && fin(c->split_factor) && c->scene_scale > 0.f && c->split_factor > 0.f &&
           c->grow_grad2d >= 0.f && c->grow_scale3d > 0.f && c->prune_scale3d > 0.f;
}

static bool ds_scene_ok(const gs_scene_buf* s)
{
    return s && s->n >= 1 && s->n < ((int64_t)1 << 31) && s->geom && s->sh && s->m && s->v;
}

static gs_status ds_launch_status()
{
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

}  // namespace gs

using namespace gs;

extern "C" {

size_t gs_densify_scratch_bytes(int64_t n)
{
    if (n < 1) return 0;
    return ds_layout(n, nullptr, nullptr);
}

gs_status gs_densify_count(const gs_scene_buf* scene, int32_t storage_flags, const gs_densify_cfg* cfg,
                           void* scratch, void* stream)
{
    (void)storage_flags;
    if (!ds_scene_ok(scene) || !scene->stats || !scratch || !ds_cfg_ok(cfg)) return GS_ERR_INVALID_ARG;
    const int64_t n = scene->n;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    DensifyScratch d;
    ds_layout(n, scratch, &d);
    DensifyK K;
    K.grad_thr = cfg->grow_grad2d;
    K.small_thr = cfg->grow_scale3d * cfg->scene_scale;
    K.prune_opa = cfg->prune_opa;
    K.big_thr = cfg->prune_scale3d * cfg->scene_scale;
    K.factor = cfg->split_factor;
    K.grow = cfg->grow != 0;
    K.prune_big = cfg->prune_big != 0;
    const unsigned blocks = (unsigned)ds_blocks(n);
    launch_after(k_densify_decide, blocks, kScanThreads, 0, st, n, static_cast<const float4*>(scene->geom),
                 static_cast<const float2*>(scene->stats), K, d.fate, d.part);
    launch_after(k_densify_scan, 1, 1024, 0, st, blocks, d.part, d.counts);
    launch_after(k_densify_index, blocks, kScanThreads, 0, st, d.fate, d.part, d.counts, d.src);
    return ds_launch_status();
}

gs_status gs_densify_counts(const void* scratch, int64_t counts[4], void* stream)
{
    if (!scratch || !counts) return GS_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(counts, scratch, 4 * sizeof(int64_t), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return GS_ERR_CUDA;
    return cudaStreamSynchronize(st) == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status gs_densify_apply(const gs_scene_buf* in, int32_t storage_flags, const gs_densify_cfg* cfg,
                           const float* eps, const void* scratch, gs_scene_buf* out, void* stream)
{
    if (!ds_scene_ok(in) || !ds_scene_ok(out) || !eps || !scratch || !ds_cfg_ok(cfg)) return GS_ERR_INVALID_ARG;
    const int64_t n = in->n;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    DensifyScratch d;
    ds_layout(n, const_cast<void*>(scratch), &d);
    const SceneDesc si = ds_scene(*in), so = ds_scene(*out);
    const dim3 grid((unsigned)((so.n + 255) / 256), 4);
    const bool sh16 = storage_flags & GS_STORE_SH_BF16, mom16 = storage_flags & GS_STORE_MOMENTS_BF16;
#define GS_DA(A, B) launch_after(k_densify_apply<A, B>, grid, 256, 0, st, si, so, d.src, d.counts, eps, cfg->split_factor)
    if (sh16 && mom16) GS_DA(true, true);
    else if (sh16) GS_DA(true, false);
    else if (mom16) GS_DA(false, true);
    else GS_DA(false, false);
#undef GS_DA
    return ds_launch_status();
}

gs_status gs_reset_opacity(const gs_scene_buf* scene, int32_t storage_flags, float value, void* stream)
{
    if (!ds_scene_ok(scene) || !(value == value)) return GS_ERR_INVALID_ARG;
    const SceneDesc s = ds_scene(*scene);
    const unsigned blocks = (unsigned)((scene->n + 255) / 256);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (storage_flags & GS_STORE_MOMENTS_BF16) k_reset_opacity<true><<<blocks, 256, 0, st>>>(s, value);
    else k_reset_opacity<false><<<blocks, 256, 0, st>>>(s, value);
    return ds_launch_status();
}

}  // extern "C"
