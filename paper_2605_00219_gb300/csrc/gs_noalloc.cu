// gs_noalloc.cu -- L1 loss and gradient that needs no device allocation.
//
// Some callers cannot allocate device memory at all: a host framework that
// owns every byte of the GPU through its own pool and forbids libraries from
// calling cudaMalloc, a real-time renderer whose frame loop must never block
// on the allocator, or code that runs while allocation is disallowed.  Such a
// caller can still compute the L1 loss of its rendered images and the
// gradient dL/dC with gs_loss_l1_noalloc(), which needs no plan and no
// workspace: its only scratch (one partial sum per thread block and a
// completion counter) lives in the static device array below, which the
// library image carries and every GPU that loads the library keeps until the
// process exits.
//
// The array is shared by all calls on a device and keeps whatever the last
// call left in it; the counter is cleared before every launch.  Calls whose
// executions overlap on the GPU (different streams, no ordering between
// them) race on the array and must not be issued.
#include <cfloat>
#include <mutex>

#include "gs_internal.cuh"

namespace {

constexpr int kNaThreads = 256;
constexpr int kNaItems = 8;                               // values per thread and tile
constexpr int kNaTile = kNaThreads * kNaItems;
// 8 blocks per SM: every block is resident, and the last one adds at most this
// many partial sums
constexpr int kNaMaxBlocks = 152 * 8;
constexpr int kNaMaxDevices = 64;

// [0] completion counter, [1..63] unused (keeps the partials 256-byte
// aligned), [64 ..] one float partial sum per thread block.
static __device__ __align__(256) uint32_t g_l1_noalloc_scratch[64 + kNaMaxBlocks];

std::mutex g_setup_mutex;
uint32_t* g_scratch_addr[kNaMaxDevices];

// Device address of the scratch array on the current device.  In host code
// the array's name is only a host-side stand-in, so the address is looked up
// once per device with cudaGetSymbolAddress (with that device current) and
// cached.  It is the address in the device's primary context; a device reset
// or another current context would make it stale, which the header rules
// out for callers.
gs_status scratch_on_current_device(uint32_t** out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNaMaxDevices) {
        cudaGetLastError();
        return GS_ERR_CUDA;
    }
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_addr[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_l1_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            return GS_ERR_CUDA;
        }
        g_scratch_addr[dev] = static_cast<uint32_t*>(p);
    }
    *out = g_scratch_addr[dev];
    return GS_OK;
}

__device__ __forceinline__ float na_sign(float d, float inv_n) { return d > 0.f ? inv_n : (d < 0.f ? -inv_n : 0.f); }

// Bound by HBM (12 bytes a value).  Blocks stride over tiles of 2,048 values, four
// values per access when the three arrays are 16-byte aligned (VEC); a thread
// adds its eight values of a tile to a Kahan-compensated total.  The last block to
// finish adds the blocks' sums across its threads (compensated, fixed order).
// 1920 x 1080 x 3 values: 76 -> 13 us; one block per tile had left 3,038
// partial sums to one thread.
template <bool VEC>
__global__ void __launch_bounds__(kNaThreads) k_loss_l1_noalloc(const float* __restrict__ image,
                                                                const float* __restrict__ target,
                                                                float* __restrict__ dl, int64_t n, float inv_n,
                                                                uint32_t* __restrict__ scratch,
                                                                float* __restrict__ loss_out)
{
    __shared__ float ws[kNaThreads / 32], wl[kNaThreads / 32];
    __shared__ bool is_last;
    uint32_t* counter = scratch;
    float* part = reinterpret_cast<float*>(scratch + 64);
    float s = 0.f, comp = 0.f;
    for (int64_t base = (int64_t)blockIdx.x * kNaTile; base < n; base += (int64_t)gridDim.x * kNaTile) {
        float t = 0.f;
        if (VEC && base + kNaTile <= n) {
            const int64_t i0 = base / 4 + threadIdx.x, i1 = i0 + kNaThreads;
            const float4 a0 = reinterpret_cast<const float4*>(image)[i0], a1 = reinterpret_cast<const float4*>(image)[i1];
            const float4 b0 = reinterpret_cast<const float4*>(target)[i0], b1 = reinterpret_cast<const float4*>(target)[i1];
            const float4 d0 = make_float4(a0.x - b0.x, a0.y - b0.y, a0.z - b0.z, a0.w - b0.w);
            const float4 d1 = make_float4(a1.x - b1.x, a1.y - b1.y, a1.z - b1.z, a1.w - b1.w);
            reinterpret_cast<float4*>(dl)[i0] =
                make_float4(na_sign(d0.x, inv_n), na_sign(d0.y, inv_n), na_sign(d0.z, inv_n), na_sign(d0.w, inv_n));
            reinterpret_cast<float4*>(dl)[i1] =
                make_float4(na_sign(d1.x, inv_n), na_sign(d1.y, inv_n), na_sign(d1.z, inv_n), na_sign(d1.w, inv_n));
            t = ((fabsf(d0.x) + fabsf(d0.y)) + (fabsf(d0.z) + fabsf(d0.w))) +
                ((fabsf(d1.x) + fabsf(d1.y)) + (fabsf(d1.z) + fabsf(d1.w)));
        } else {
#pragma unroll
            for (int i = 0; i < kNaItems; i++) {
                const int64_t idx = base + i * kNaThreads + threadIdx.x;
                if (idx < n) {
                    const float d = image[idx] - target[idx];
                    dl[idx] = na_sign(d, inv_n);
                    t += fabsf(d);
                }
            }
        }
        // (an infinite total has no error term: infinity - infinity)
        const float y = t - comp, u = s + y;
        comp = u <= FLT_MAX ? (u - s) - y : 0.f;
        s = u;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int i = 0; i < kNaThreads / 32; i++) t += ws[i];
        part[blockIdx.x] = t;
        __threadfence();
        is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    // the blocks' sums as unevaluated pairs (hi, lo), so that the last levels,
    // at the total's magnitude, round once (lo stays finite when hi is not)
    float hi = 0.f, lo = 0.f;
    auto add = [&](float h2, float l2) {
        float e;
        gs::two_sum(hi, h2, hi, e);
        lo += l2 + (hi <= FLT_MAX ? e : 0.f);
    };
    for (unsigned i = threadIdx.x; i < gridDim.x; i += kNaThreads) add(((volatile float*)part)[i], 0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_down_sync(0xffffffffu, hi, o), l2 = __shfl_down_sync(0xffffffffu, lo, o);
        add(h2, l2);
    }
    if ((threadIdx.x & 31) == 0) {
        ws[threadIdx.x >> 5] = hi;
        wl[threadIdx.x >> 5] = lo;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kNaThreads / 32; i++) add(ws[i], wl[i]);
        *loss_out = (hi + lo) * inv_n;
        *counter = 0u;
    }
}

}  // namespace

extern "C" gs_status gs_loss_l1_noalloc(const float* image, const float* target, float* dL_dimage, float* loss,
                                        int64_t n_values, void* stream)
{
    if (!image || !target || !dL_dimage || !loss) return GS_ERR_INVALID_ARG;
    if (n_values <= 0 || n_values > GS_L1_NOALLOC_MAX_VALUES) return GS_ERR_INVALID_ARG;
    uint32_t* scratch = nullptr;
    const gs_status e = scratch_on_current_device(&scratch);
    if (e != GS_OK) return e;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(scratch, 0, sizeof(uint32_t), st) != cudaSuccess) {
        cudaGetLastError();
        return GS_ERR_CUDA;
    }
    const int64_t blocks = std::min<int64_t>((n_values + kNaTile - 1) / kNaTile, kNaMaxBlocks);
    const bool vec = ((reinterpret_cast<uintptr_t>(image) | reinterpret_cast<uintptr_t>(target) |
                       reinterpret_cast<uintptr_t>(dL_dimage)) & 15u) == 0;
    const float inv_n = 1.0f / (float)n_values;
    if (vec)
        k_loss_l1_noalloc<true><<<(unsigned)blocks, kNaThreads, 0, st>>>(image, target, dL_dimage, n_values, inv_n,
                                                                         scratch, loss);
    else
        k_loss_l1_noalloc<false><<<(unsigned)blocks, kNaThreads, 0, st>>>(image, target, dL_dimage, n_values, inv_n,
                                                                          scratch, loss);
    if (cudaPeekAtLastError() != cudaSuccess) {
        cudaGetLastError();
        return GS_ERR_CUDA;
    }
    return GS_OK;
}
