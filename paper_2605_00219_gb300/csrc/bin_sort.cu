// bin_sort.cu -- tiling and sorting (VkSplat Sec. 4.1, Sec. 4.4; Table 2
// "Tiling/Sorting": index offset, generate keys, sorting, tile ranges).
//
// The sorted lists are the 32-bit keys (tile << shift | depth code >> drop)
// of Sec. 4.4 in stable order, i.e. ordered by (view, tile, depth code,
// emission slot): the tile is the key's leading part, so the sort is done
// as a bucketing by tile followed by a sort of each tile's short list.
//
//   index offset : exclusive scan of the per-pair tile counts, in
//                  Gaussian-major pair order: a Gaussian's intersections in all
//                  views are consecutive emission slots.  Sums per 1,024 pairs,
//                  one block scans them, and the emission scans its pairs (no
//                  inter-block waiting, no second pass over the counts)
//   tile ranges  : the projection's traversal already counted the entries of
//                  every tile; their exclusive scan gives each tile's
//                  [start, end) in the sorted arrays and its scatter cursor
//   generate keys: from the tile spans the projection kept, each intersection
//                  goes to its rank's or the next free place of its tile (depth
//                  code and emission slot), and its pair to the emission slot
//   sorting      : a thread block, a part of one or a warp sorts a tile's
//                  entries by (depth code, emission slot) -- unique, so the
//                  arrival order of the atomics does not matter -- and writes
//                  the keys, emission slots and pairs: 32-bit words of depth
//                  code and arrival index sorted in registers and merged in
//                  shared memory, ties put in order afterwards; 64-bit keys
//                  where the words are too short; longer lists in chunks,
//                  merged in global memory piece by piece
// K never leaves the device: every kernel reads it from the workspace header
// and grids are sized by the plan.  When K exceeds the capacity nothing is
// emitted and every tile list is empty (GS_STATUS_CAPACITY reports it).
#include "gs_internal.cuh"

namespace gs {

// ---------------------------------------------------------------------------
// Emission slots, tile ranges and launch order
// ---------------------------------------------------------------------------

// Launch order of the raster kernels and the tile sort: tiles by decreasing list
// length, bucketed by floor(log2(length + 1)).  Blocks are dispatched roughly in
// index order, so the longest tiles start first and the short ones fill the
// tail (longest-processing-time scheduling).  Within a bucket the order
// follows shared-memory atomics; it decides only when a tile runs, never its
// result.
__device__ __forceinline__ int len_bucket(uint32_t len) { return 31 - __clz(len + 1u); }

// The sort's size classes are runs of buckets: long >= 2047 entries (buckets
// 11+), medium 1023-2046 (10), short 255-1022 (8, 9), tiny <= 254 (0-7).  One
// thread: the class sizes, and each bucket's first place in the order (in place).
__device__ __forceinline__ void order_places(uint32_t* cnt, WsHeader* hdr)
{
    uint32_t cls[4] = {0u, 0u, 0u, 0u};
    uint32_t run = 0;
    for (int b = 31; b >= 0; b--) {
        const uint32_t c = cnt[b];
        cls[b >= 11 ? 0 : b == 10 ? 1 : b >= 8 ? 2 : 3] += c;
        cnt[b] = run;
        run += c;
    }
    for (int c = 0; c < 4; c++) hdr->sort_class[c] = cls[c];
}

// Intersections of one group of kPairGroup pairs, summed by one warp.
__device__ __forceinline__ uint32_t pair_group_sum(const uint32_t* __restrict__ count, int64_t pairs, int64_t group)
{
    // (every load of the group in flight at once)
    uint32_t c[kPairGroup / 32], s = 0;
#pragma unroll
    for (int k = 0; k < kPairGroup / 32; k++) {
        const int64_t q = group * kPairGroup + 32 * k + (threadIdx.x & 31);
        c[k] = q < pairs ? count[q] : 0u;
    }
#pragma unroll
    for (int k = 0; k < kPairGroup / 32; k++) s += c[k];
    return __reduce_add_sync(0xffffffffu, s);
}

// Exclusive scan in place of the pair groups' intersection counts by one block of
// 1,024 threads (each warp one run of them: sums, then prefixes), K, the
// offsets' last entry and the capacity check: k_eff = K when it fits, else 0
// (nothing is emitted) with GS_STATUS_CAPACITY.  Returns whether K fits.
__device__ bool scan_gpart(uint32_t* __restrict__ gpart, int64_t blocks, WsHeader* __restrict__ hdr,
                           uint32_t* __restrict__ total_at, uint32_t cap, unsigned long long* ws)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t per = ((blocks + 31) / 32 + 31) & ~(int64_t)31;       // whole warp accesses
    const int64_t b0 = min(per * w, blocks), b1 = min(b0 + per, blocks);
    unsigned long long sum = 0;
#pragma unroll 4
    for (int64_t i = b0 + lane; i < b1; i += 32) sum += gpart[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) ws[w] = sum;
    __syncthreads();
    unsigned long long before = 0, total = 0;
    for (int k = 0; k < 32; k++) {
        if (k < w) before += ws[k];
        total += ws[k];
    }
    uint32_t carry = (uint32_t)before;
#pragma unroll 4
    for (int64_t i0 = b0; i0 < b1; i0 += 32) {
        const uint32_t v = i0 + lane < b1 ? gpart[i0 + lane] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (i0 + lane < b1) gpart[i0 + lane] = carry + x - v;
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    const bool fits = total <= cap;
    if (threadIdx.x == 0) {
        hdr->k_required = total;
        hdr->k_eff = fits ? (uint32_t)total : 0u;
        if (!fits) atomicOr(&hdr->status, GS_STATUS_CAPACITY);
        *total_at = (uint32_t)total;
    }
    return fits;
}

// Range of a tile: its list, empty when the tile is or when K exceeds the capacity.
__device__ __forceinline__ uint2 tile_range(uint32_t start, uint32_t len, bool fits)
{
    return fits && len ? make_uint2(start, start + len) : make_uint2(0u, 0u);
}

// Up to kScanBlock tiles, one block: emission-slot scan, K, and for every tile
// its start (exclusive scan of both counters), range, the cursor of the other
// pairs' entries (start + the ranked entries, written over their counter) and its
// place in the launch order.  Latency-bound; seven launches of the same work took
// 25 us at 64 tiles and 36 us at 3,600 (8 us here, and 4 us of k_sort_sums).
__global__ void __launch_bounds__(1024) k_sort_setup(const uint32_t* __restrict__ count, int64_t pairs, bool summed,
                                                     uint32_t* gpart, int64_t gblocks, int tiles,
                                                     uint32_t* cnt, uint32_t* __restrict__ tile_cur,
                                                     uint2* __restrict__ ranges, uint32_t* __restrict__ order,
                                                     uint32_t* __restrict__ total_at, WsHeader* __restrict__ hdr,
                                                     uint32_t cap)
{
    if (!after_previous()) return;
    constexpr int IT = kScanBlock / 1024;
    __shared__ unsigned long long ws64[32];
    __shared__ uint32_t ws[32], hist[32];
    __shared__ uint32_t buf[kScanBlock];
    if (threadIdx.x < 32) hist[threadIdx.x] = 0;
    uint32_t c0[IT], len[IT];
#pragma unroll
    for (int k = 0; k < IT; k++) {
        const int t = k * 1024 + threadIdx.x;
        c0[k] = t < tiles ? cnt[t] : 0u;
        len[k] = t < tiles ? c0[k] + cnt[tiles + t] : 0u;
        buf[t] = len[k];
    }
    if (!summed) {
        for (int64_t g = threadIdx.x >> 5; g < gblocks; g += 32) {
            const uint32_t t = pair_group_sum(count, pairs, g);
            if ((threadIdx.x & 31) == 0) gpart[g] = t;
        }
        __syncthreads();
    }
    const bool fits = scan_gpart(gpart, gblocks, hdr, total_at, cap, ws64);     // (synchronises)
    uint32_t own[IT], s = 0;
#pragma unroll
    for (int k = 0; k < IT; k++) {
        own[k] = s;
        s += buf[threadIdx.x * IT + k];
    }
    const uint32_t ex = block_excl_scan<1024>(s, ws, nullptr);
#pragma unroll
    for (int k = 0; k < IT; k++) buf[threadIdx.x * IT + k] = ex + own[k];
#pragma unroll
    for (int k = 0; k < IT; k++)
        if (k * 1024 + (int)threadIdx.x < tiles) atomicAdd(&hist[len_bucket(fits ? len[k] : 0u)], 1u);
    __syncthreads();
    if (threadIdx.x == 0) order_places(hist, hdr);
#pragma unroll
    for (int k = 0; k < IT; k++) {
        const int t = k * 1024 + threadIdx.x;
        if (t < tiles) {
            const uint32_t s0 = buf[t];
            tile_cur[t] = s0;
            ranges[t] = tile_range(s0, len[k], fits);
            cnt[tiles + t] = s0 + c0[k];
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < IT; k++) {
        const int t = k * 1024 + threadIdx.x;
        if (t < tiles) order[atomicAdd(&hist[len_bucket(fits ? len[k] : 0u)], 1u)] = (uint32_t)t;
    }
}

// More pairs or tiles: sums first.  Blocks below gblocks16: the sums of 16 pair
// groups, one per warp; the others (more than kScanBlock tiles, the same work in
// three launches): sum and list-length histogram of kScanBlock tiles per block
// (part: [blocks] sums, then [blocks][32] buckets);
__global__ void __launch_bounds__(kScanThreads) k_sort_sums(const uint32_t* __restrict__ count, int64_t pairs,
                                                            uint32_t* __restrict__ gpart, int64_t gblocks,
                                                            unsigned gblocks16, int64_t tiles,
                                                            const uint32_t* __restrict__ cnt,
                                                            uint32_t* __restrict__ part)
{
    if (!after_previous()) return;
    __shared__ uint32_t ws[32], hist[32];
    if (blockIdx.x < gblocks16) {
        const int64_t g = (int64_t)blockIdx.x * (kScanThreads / 32) + (threadIdx.x >> 5);
        if (g < gblocks) {
            const uint32_t t = pair_group_sum(count, pairs, g);
            if ((threadIdx.x & 31) == 0) gpart[g] = t;
        }
        return;
    }
    const int64_t blk = blockIdx.x - gblocks16, blocks = gridDim.x - gblocks16;
    if (threadIdx.x < 32) hist[threadIdx.x] = 0;
    __syncthreads();
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        const int64_t t = blk * kScanBlock + k * kScanThreads + threadIdx.x;
        if (t < tiles) {
            const uint32_t len = cnt[t] + cnt[tiles + t];
            s += len;
            atomicAdd(&hist[len_bucket(len)], 1u);
        }
    }
    uint32_t tot;
    block_excl_scan<kScanThreads>(s, ws, &tot);      // (synchronises)
    if (threadIdx.x == 0) part[blk] = tot;
    if (threadIdx.x < 32) part[blocks + 32 * blk + threadIdx.x] = hist[threadIdx.x];
}

// one block: the emission-slot scan and K, the blocks' tile starts, and each
// (block, bucket)'s first place in the order (when K exceeds the capacity every
// list is empty: all tiles in bucket 0);
__global__ void __launch_bounds__(1024) k_sort_parts(uint32_t* __restrict__ gpart, int64_t gblocks, int64_t tiles,
                                                     uint32_t* __restrict__ part, int64_t nparts,
                                                     uint32_t* __restrict__ total_at, WsHeader* __restrict__ hdr,
                                                     uint32_t cap)
{
    if (!after_previous()) return;
    __shared__ unsigned long long ws64[32];
    __shared__ uint32_t ws[32], place[32];
    const bool fits = scan_gpart(gpart, gblocks, hdr, total_at, cap, ws64);
    uint32_t carry = 0;
    for (int64_t b = 0; b < nparts; b += 1024) {
        const int64_t i = b + threadIdx.x;
        const uint32_t v = i < nparts ? part[i] : 0u;
        uint32_t tot;
        const uint32_t ex = block_excl_scan<1024>(v, ws, &tot);
        if (i < nparts) part[i] = carry + ex;
        carry += tot;
        __syncthreads();
    }
    uint32_t* hist = part + nparts;
    const int b = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        uint32_t c = 0;
        for (int64_t i = 0; i < nparts; i++) {
            if (!fits) hist[32 * i + b] = b ? 0u : (uint32_t)min((int64_t)kScanBlock, tiles - i * kScanBlock);
            c += hist[32 * i + b];
        }
        place[b] = c;
        __syncwarp();
        if (threadIdx.x == 0) order_places(place, hdr);
        __syncwarp();
        uint32_t run = place[b];
        for (int64_t i = 0; i < nparts; i++) {
            const uint32_t h = hist[32 * i + b];
            hist[32 * i + b] = run;
            run += h;
        }
    }
}

// starts, ranges, cursors and places.
__global__ void __launch_bounds__(kScanThreads) k_tile_down(int64_t tiles, uint32_t* cnt,
                                                            const uint32_t* __restrict__ part,
                                                            uint32_t* __restrict__ tile_cur,
                                                            uint2* __restrict__ ranges, uint32_t* __restrict__ order,
                                                            const WsHeader* __restrict__ hdr)
{
    if (!after_previous()) return;
    __shared__ uint32_t ws[32], hist[32];
    __shared__ uint32_t buf[kScanBlock];
    const int64_t base = (int64_t)blockIdx.x * kScanBlock;
    if (threadIdx.x < 32) hist[threadIdx.x] = part[gridDim.x + 32 * (int64_t)blockIdx.x + threadIdx.x];
    const bool fits = hdr->k_eff == hdr->k_required;
    uint32_t c0[kScanItems], len[kScanItems];
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        const int l = k * kScanThreads + threadIdx.x;
        c0[k] = base + l < tiles ? cnt[base + l] : 0u;
        len[k] = base + l < tiles ? c0[k] + cnt[tiles + base + l] : 0u;
        buf[l] = len[k];
    }
    __syncthreads();
    uint32_t own[kScanItems], s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        own[k] = s;
        s += buf[threadIdx.x * kScanItems + k];
    }
    const uint32_t ex = block_excl_scan<kScanThreads>(s, ws, nullptr) + part[blockIdx.x];
#pragma unroll
    for (int k = 0; k < kScanItems; k++) buf[threadIdx.x * kScanItems + k] = ex + own[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        const int l = k * kScanThreads + threadIdx.x;
        const int64_t t = base + l;
        if (t < tiles) {
            const uint32_t s0 = buf[l];
            tile_cur[t] = s0;
            ranges[t] = tile_range(s0, len[k], fits);
            cnt[tiles + t] = s0 + c0[k];
            order[atomicAdd(&hist[len_bucket(fits ? len[k] : 0u)], 1u)] = (uint32_t)t;
        }
    }
}

// ---------------------------------------------------------------------------
// Generate keys into tile buckets
// ---------------------------------------------------------------------------

constexpr int kEmitThreads = 256;
// Tiles of a one- or two-band pair that its own lane places.
constexpr uint32_t kEmitLane = 16;

// One thread per Gaussian-major pair q: its intersections take emission
// slots offset[q] + i in traversal order; each is placed in its tile's list
// (depth code and emission slot), and the view-major pair index is recorded
// at its emission slot.  The tiles come from the pair's tile span.  A ranked
// pair's entries go to tile start + the rank the projection took; the other
// pairs' entries take the next free place after the ranked ones (an atomic
// cursor per tile), and the rare pair of more than two bands repeats the
// traversal from its binning geometry.  A pair of more than kEmitLane tiles or
// two bands is placed by its whole warp: one lane's serial walk of the largest
// footprints was a third of the launch on a room of 200k Gaussians (32 -> 22 us).
// 3M Gaussians, 4 views: 265 us with the slot scan inside, against 240 + 49 us for
// the emission and a separate scan (5 blocks per SM; 6 / 4: 274 / 285 us).
//
// The pair's first emission slot is its group's scanned sum, the counts of the
// group's earlier blocks (at most three), and a scan of the block's own counts.  It is
// written to offset for the backward.
__global__ void __launch_bounds__(kEmitThreads, 5) k_emit(Views V, const uint32_t* __restrict__ count,
                                                 const uint32_t* __restrict__ gpart,
                                                 uint32_t* __restrict__ offset, const ProjRec* __restrict__ rec,
                                                 const uint4* __restrict__ span, const uint4* __restrict__ rank,
                                                 const uint32_t* __restrict__ tile_start, uint32_t* tile_over,
                                                 uint2* __restrict__ bucket, uint32_t* __restrict__ pid,
                                                 WsHeader* __restrict__ hdr)
{
    if (!after_previous()) return;
    __shared__ uint32_t ws[32], earlier[kEmitThreads / 32];
    const int64_t qb = (int64_t)blockIdx.x * kEmitThreads, qi = qb + threadIdx.x;
    // the pair's loads are issued together, before any of them is tested
    // (one memory round trip instead of three); span and ranks are stale
    // for a pair without tiles and a pair that is not ranked, and unused
    const unsigned long long kreq = hdr->k_required;
    const uint32_t keff = hdr->k_eff;
    const bool valid = qi < V.pairs;
    const uint32_t cnt = valid ? count[qi] : 0u;
    uint4 sp, rk4;
    if (valid) {
        sp = span[qi];
        rk4 = rank[qi];
    }
    uint32_t pre = 0;
    for (int64_t q = qi - kEmitThreads; q >= qb - qb % kPairGroup; q -= kEmitThreads) pre += count[q];
    pre = __reduce_add_sync(0xffffffffu, pre);
    if ((threadIdx.x & 31) == 0) earlier[threadIdx.x >> 5] = pre;
    uint32_t off = gpart[qb / kPairGroup] + block_excl_scan<kEmitThreads>(cnt, ws, nullptr);   // (synchronises)
#pragma unroll
    for (int k = 0; k < kEmitThreads / 32; k++) off += earlier[k];
    if (valid) offset[qi] = off;
    if (keff != kreq) return;     // over capacity: nothing is emitted
    int s = 0;
    while (s + 1 < V.n_scenes && V.qbase[s + 1] <= qi) s++;
    const uint32_t nv = (uint32_t)V.nv[s];
    const uint32_t local = (uint32_t)(qi - V.qbase[s]);     // pairs < 2^31
    const uint32_t g = local / nv;
    const int v = cnt ? V.view_of[s][local - g * nv] : 0;
    const ViewDesc& vd = V.v[v];
    const uint32_t p = (uint32_t)vd.pair_base + g;
    const uint32_t nb = (sp.x >> 24) & 3u;
    // a pair of many tiles is placed by the whole warp, below
    const bool wide = cnt != 0 && (nb == kSpanMany || cnt > kEmitLane);
    if (cnt != 0 && !wide) {
        const uint32_t low = (sp.x & 0x7FFFFFu) >> vd.drop;
        uint32_t* cur = tile_over + vd.tile_base;
        const bool rows = (sp.x >> 26) & 1u;
        const uint32_t TX = (uint32_t)vd.TX;
        const uint32_t c0 = sp.y & 0xFFFFu, c1 = sp.y >> 16;
        if ((sp.x >> 27) & 1u) {
            // ranked: at most kRankMax tiles, no atomics
            const uint32_t rk[kRankMax] = {rk4.x, rk4.y, rk4.z, rk4.w};
            const uint32_t* __restrict__ st0 = tile_start + vd.tile_base;
#pragma unroll
            for (uint32_t u = 0; u < kRankMax; u++) {
                const uint32_t e = off + u;
                if (u < cnt) {
                    const uint32_t slot = st0[span_tile(u, rows, TX, c0, c1, sp.z, sp.w)] + rk[u];
                    if (GS_DCHECK(slot < hdr->k_eff && e < hdr->k_eff, &hdr->status)) {
                        bucket[slot] = make_uint2(low, e);
                        pid[e] = p;
                    }
                }
            }
        } else {
            // one or two bands: the cursors taken four at a time so that the
            // atomics' round trips overlap
            for (uint32_t i0 = 0; i0 < cnt; i0 += 4) {
                uint32_t slot[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const uint32_t i = i0 + u;
                    if (i < cnt) slot[u] = atomicAdd(cur + span_tile(i, rows, TX, c0, c1, sp.z, sp.w), 1u);
                }
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const uint32_t i = i0 + u, e = off + i;
                    if (i < cnt && GS_DCHECK(slot[u] < hdr->k_eff && e < hdr->k_eff, &hdr->status)) {
                        bucket[slot[u]] = make_uint2(low, e);
                        pid[e] = p;
                    }
                }
            }
        }
    }
    for (uint32_t m = __ballot_sync(0xffffffffu, wide); m; m &= m - 1u) {
        const int k = __ffs(m) - 1;
        auto from = [&](uint32_t x) { return __shfl_sync(0xffffffffu, x, k); };
        const uint4 ks = make_uint4(from(sp.x), from(sp.y), from(sp.z), from(sp.w));
        const uint32_t koff = from(off), kcnt = from(cnt), kp = from(p);
        const ViewDesc& kd = V.v[from((uint32_t)v)];
        const uint32_t low = (ks.x & 0x7FFFFFu) >> kd.drop;
        uint32_t* cur = tile_over + kd.tile_base;
        auto place = [&](uint32_t i, uint32_t tile) {
            const uint32_t e = koff + i, slot = atomicAdd(cur + tile, 1u);
            if (GS_DCHECK(slot < hdr->k_eff && e < hdr->k_eff, &hdr->status)) {
                bucket[slot] = make_uint2(low, e);
                pid[e] = kp;
            }
        };
        if (((ks.x >> 24) & 3u) == kSpanMany) {
            // the traversal again, from the binning geometry (same bits)
            const float4 ra = rec[kp].a;
            BinGeom gm;
            gm.mx = ra.x; gm.my = ra.y;
            gm.a = __uint_as_float(ks.y); gm.b = __uint_as_float(ks.z); gm.c = __uint_as_float(ks.w);
            gm.det = FS(FM(gm.a, gm.c), FM(gm.b, gm.b));
            gm.r2 = cull_r2(rec[kp].b.y);
            gm.mant = ks.x & 0x7FFFFFu;
            gm.valid = 1;
            warp_scanline(gm, V.tw, V.th, kd.TX, kd.TY, place);
        } else {
            const bool rows = (ks.x >> 26) & 1u;
            for (uint32_t i = threadIdx.x & 31; i < kcnt; i += 32)
                place(i, span_tile(i, rows, (uint32_t)kd.TX, ks.y & 0xFFFFu, ks.y >> 16, ks.z, ks.w));
        }
    }
}

// ---------------------------------------------------------------------------
// Per-tile sort
// ---------------------------------------------------------------------------

__device__ __forceinline__ unsigned long long sort_key(uint32_t low, uint32_t e)
{
    return ((unsigned long long)low << 32) | e;
}

// Ascending sort of N (a multiple of 8, 8 <= N <= 8 * blockDim.x) 64-bit
// keys in shared memory, block merge sort: thread t < N / 8 owns the 8 keys
// [8t, 8t + 8); it sorts them with a 19-comparator network in registers,
// then, at each merge level of run width w, finds where its 8 outputs start
// in the merge of its two runs (merge-path binary search on the output
// diagonal) and merges them sequentially.  The last run of a level may be
// short or alone (then it is already merged), so no padding to a power of
// two is sorted.  While two runs fit in one warp's 256 keys (w <= 128) only
// that warp reads and writes them, so the level synchronises the warp; a
// level that reads wider runs synchronises the group, also before its
// reads.  The caller synchronises the group before.
template <typename Key>
__device__ __forceinline__ void cmpx(Key& a, Key& b)
{
    const Key lo = a < b ? a : b, hi = a < b ? b : a;
    a = lo;
    b = hi;
}

// The threads that sort one list: the whole block, half of it (a named
// barrier of its own) or one warp.  t is the thread's index in the group.
struct SortGroup {
    int t, n, bar;
    __device__ __forceinline__ void sync() const
    {
        if (n == 32) __syncwarp();
        else if (bar == 0) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(n) : "memory");
    }
};

// Whether any thread of the group has the flag (synchronises the group; a warp's
// shared-memory accesses are not ordered by it).
__device__ __forceinline__ bool group_any(const SortGroup& g, bool flag)
{
    if (g.n == 32) return __any_sync(0xffffffffu, flag);
    if (g.bar == 0) return __syncthreads_or(flag);
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.u32 q, %1, 0;\nbar.red.or.pred p, %2, %3, q;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(r)
        : "r"((uint32_t)flag), "r"(g.bar), "r"(g.n)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ SortGroup whole_block() { return SortGroup{(int)threadIdx.x, (int)blockDim.x, 0}; }

// Merge levels of the block merge sort from run width w0 (every run of w0 keys
// sorted, the group synchronised): threads t < N / IT place IT outputs each.
template <int IT, typename Key>
__device__ __forceinline__ void merge_levels_smem(Key* s, int N, int w0, const SortGroup& g)
{
    const int nt = N / IT, t = g.t;
    Key r[IT];
    for (int w = w0; w < N; w <<= 1) {
        const bool in_warp = 2 * w <= 32 * IT;
        const int base = (IT * t) & ~(2 * w - 1), diag = IT * t - base;
        const int la = min(w, N - base), lb = max(0, min(w, N - base - w));
        const bool merge = t < nt && lb > 0;   // a lone last run stays in place
        if (merge) {
            const Key* A = s + base;
            const Key* B = s + base + w;
            int lo = max(0, diag - lb), hi = min(diag, la);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (A[mid] <= B[diag - 1 - mid]) lo = mid + 1;
                else hi = mid;
            }
            int a = lo, b = diag - lo;
            Key ha = a < la ? A[a] : Key(0), hb = b < lb ? B[b] : Key(0);
#pragma unroll
            for (int k = 0; k < IT; k++) {
                const bool take_a = b >= lb || (a < la && ha <= hb);
                r[k] = take_a ? ha : hb;
                if (take_a) {
                    a++;
                    ha = a < la ? A[a] : Key(0);
                } else {
                    b++;
                    hb = b < lb ? B[b] : Key(0);
                }
            }
        }
        if (in_warp) __syncwarp();
        else g.sync();
        if (merge) {
            if constexpr (sizeof(Key) == 4) {
#pragma unroll
                for (int k = 0; k < IT; k += 4)
                    *reinterpret_cast<uint4*>(s + IT * t + k) = make_uint4(r[k], r[k + 1], r[k + 2], r[k + 3]);
            } else {
#pragma unroll
                for (int k = 0; k < IT; k++) s[IT * t + k] = r[k];
            }
        }
        // the next level (width 2w) reads other warps' keys unless its runs
        // still fit in one warp
        if (4 * w <= 32 * IT) __syncwarp();
        else g.sync();
    }
    g.sync();
}

template <typename Key>
__device__ __forceinline__ void sort8(Key* r)
{
    cmpx(r[0], r[1]); cmpx(r[2], r[3]); cmpx(r[4], r[5]); cmpx(r[6], r[7]);
    cmpx(r[0], r[2]); cmpx(r[1], r[3]); cmpx(r[4], r[6]); cmpx(r[5], r[7]);
    cmpx(r[1], r[2]); cmpx(r[5], r[6]);
    cmpx(r[0], r[4]); cmpx(r[1], r[5]); cmpx(r[2], r[6]); cmpx(r[3], r[7]);
    cmpx(r[2], r[4]); cmpx(r[3], r[5]);
    cmpx(r[1], r[2]); cmpx(r[3], r[4]); cmpx(r[5], r[6]);
}

__device__ void block_merge_sort_smem(unsigned long long* s, int N, const SortGroup& g)
{
    constexpr int IT = 8;
    unsigned long long r[IT];
    if (g.t < N / IT) {
#pragma unroll
        for (int k = 0; k < IT; k++) r[k] = s[IT * g.t + k];
        sort8(r);
#pragma unroll
        for (int k = 0; k < IT; k++) s[IT * g.t + k] = r[k];
    }
    __syncwarp();
    merge_levels_smem<IT>(s, N, IT, g);
}

// Ascending sort of a warp's 256 keys in registers, lane l holding [8l, 8l + 8):
// 8 keys by the network, then bitonic merges of run width 8, 16, ... up to `most`
// keys, which lie in the first most / 8 lanes (each: the mirrored exchange, then halving
// exchanges, across lanes by shuffles and within a lane in registers).  No shared-memory
// round trips.
__device__ __forceinline__ void warp_sort256(uint32_t* r, int lane, int most)
{
    sort8(r);
#pragma unroll
    for (int w = 1; w < 32; w <<= 1) {          // run width in lanes
        if (8 * w >= most) break;
        uint32_t y[8];
#pragma unroll
        for (int k = 0; k < 8; k++) y[k] = __shfl_xor_sync(0xffffffffu, r[7 - k], 2 * w - 1);
#pragma unroll
        for (int k = 0; k < 8; k++) r[k] = (lane & w) ? max(r[k], y[k]) : min(r[k], y[k]);
#pragma unroll
        for (int d = w >> 1; d > 0; d >>= 1)
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const uint32_t z = __shfl_xor_sync(0xffffffffu, r[k], d);
                r[k] = (lane & d) ? max(r[k], z) : min(r[k], z);
            }
#pragma unroll
        for (int k = 0; k < 4; k++) cmpx(r[k], r[k + 4]);
        cmpx(r[0], r[2]); cmpx(r[1], r[3]); cmpx(r[4], r[6]); cmpx(r[5], r[7]);
        cmpx(r[0], r[1]); cmpx(r[2], r[3]); cmpx(r[4], r[5]); cmpx(r[6], r[7]);
    }
}

// (depth code, emission slot) lists in two layouts: one uint2 per entry, or
// two u32 arrays.
struct PackedList {
    uint2* kv;
    __device__ unsigned long long get(uint32_t i) const { const uint2 x = kv[i]; return sort_key(x.x, x.y); }
    __device__ void put(uint32_t i, unsigned long long x) const { kv[i] = make_uint2((uint32_t)(x >> 32), (uint32_t)x); }
};
struct SplitList {
    uint32_t* k;
    uint32_t* v;
    __device__ unsigned long long get(uint32_t i) const { return sort_key(k[i], v[i]); }
    __device__ void put(uint32_t i, unsigned long long x) const { k[i] = (uint32_t)(x >> 32); v[i] = (uint32_t)x; }
};

// One merge level of run width `run` (a power of two, at least kTileSortMax) over a
// list of n entries at s0, kTileSortMax outputs at a time: where each such piece
// starts in its two runs by one binary search per thread, all at once; then both parts
// of a piece read to shared memory and merged there, 8 outputs a thread.  (A search
// per entry in global memory took 165 us a level for a list of 21,000.)
template <class Src, class Dst>
__device__ void merge_level(const Src& src, const Dst& dst, uint32_t s0, uint32_t n, uint32_t run,
                            unsigned long long* sk, uint32_t* split)
{
    constexpr uint32_t P = kTileSortMax, IT = 8;
    static_assert(P == IT * kTileSortThreads, "every thread merges 8 outputs of a piece");
    const uint32_t pieces = (n + P - 1) / P;
    for (uint32_t j0 = 0; j0 < pieces; j0 += kTileSortThreads) {
        for (uint32_t j = j0 + threadIdx.x; j <= j0 + kTileSortThreads && j < pieces; j += blockDim.x) {
            const uint32_t base = (j * P) & ~(2u * run - 1u), diag = j * P - base;
            const uint32_t la = min(run, n - base), lb = min(run, n - base - la);
            uint32_t lo = diag > lb ? diag - lb : 0u, hi = min(diag, la);
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (src.get(s0 + base + mid) < src.get(s0 + base + la + diag - 1u - mid)) lo = mid + 1u;
                else hi = mid;
            }
            split[j - j0] = lo;
        }
        __syncthreads();
        const uint32_t j1 = min(pieces, j0 + (uint32_t)kTileSortThreads);
        for (uint32_t j = j0; j < j1; j++) {
            const uint32_t base = (j * P) & ~(2u * run - 1u), diag = j * P - base;
            const uint32_t la = min(run, n - base), lb = min(run, n - base - la);
            const uint32_t end = min(diag + P, la + lb);
            const uint32_t a0 = split[j - j0], a1 = end < la + lb ? split[j + 1 - j0] : la;
            const uint32_t b0 = diag - a0, b1 = end - a1, na = a1 - a0, m = end - diag;
#pragma unroll
            for (uint32_t k = 0; k < IT; k++) {
                const uint32_t i = threadIdx.x + k * kTileSortThreads;
                if (i < m) sk[i] = src.get(s0 + base + (i < na ? a0 + i : la + b0 + i - na));
            }
            __syncthreads();
            const uint32_t nb = b1 - b0, d = min(IT * threadIdx.x, m);
            uint32_t lo = d > nb ? d - nb : 0u, hi = min(d, na);
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (sk[mid] < sk[na + d - 1u - mid]) lo = mid + 1u;
                else hi = mid;
            }
            uint32_t a = lo, b = d - lo;
#pragma unroll
            for (uint32_t k = 0; k < IT; k++) {
                if (d + k >= m) break;
                const unsigned long long ha = a < na ? sk[a] : ~0ull, hb = b < nb ? sk[na + b] : ~0ull;
                const bool take_a = b >= nb || (a < na && ha < hb);
                dst.put(s0 + base + diag + d + k, take_a ? ha : hb);
                a += take_a ? 1u : 0u;
                b += take_a ? 0u : 1u;
            }
            __syncthreads();
        }
    }
}

// The tile sort (longest lists launched first).  Input: the tile's bucket [s0, s1) of
// (depth code, emission slot) in atomic arrival order.  Output at the same positions: keys_sorted = tile << shift | depth
// code, vals_sorted = emission slot, pid_sorted = the slot's pair.
//
// A run of n <= IT g.n entries at b, sorted by the group on 32-bit words (depth code,
// arrival index) where the two fit: 256 words at a time sorted in a warp's registers,
// wider runs by merges in shared memory (`key`: IT g.n words).  Equal depth codes (17%
// of the entries at 3M Gaussians, 1080p, in runs of two or three) then still have
// arrival order, and each entry of a run counts the run's smaller emission slots.
// put(position, depth code, emission slot, pair(slot)) takes the sorted entries.  False, with
// nothing put, if `bits` of depth code leave no room for the index or more than
// kTieRun entries share a code: the caller sorts 64-bit keys then.  On a wall seen
// head-on every list is such a one; its runs show in 256 sorted words already, before
// the merges (3M Gaussians, 4x1080p, whole sort 1,174 -> 1,105 us; 1,105 with 64-bit
// keys only).
constexpr int kTieRun = 32;

template <int IT, typename Pair, typename Put>
__device__ __forceinline__ bool sort_words(const uint2* b, int n, int bits, uint32_t* key, const SortGroup& g,
                                           Pair pair, Put put)
{
    const int ib = 32 - __clz((n - 1) | 1);        // bits of the arrival index
    if (bits + ib > 32) return false;
    const int lane = g.t & 31;
    bool far = false;
#pragma unroll
    for (int c = 0; c < IT / 8; c++) {
        const int w0 = (g.t >> 5) * 32 * IT + 256 * c;
        if (w0 >= n) break;
        // the entries dealt to the first L lanes only, so a short list needs only
        // the merges of L lanes (the others hold padding)
        const int m = min(n - w0, 256);
        const int L = m <= 8 ? 1 : 1 << (32 - __clz((m - 1) >> 3));
        uint32_t r[8];
        uint2 q[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int i = L * k + lane;
            q[k] = lane < L && i < m ? b[w0 + i] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int i = L * k + lane;
            const bool in = lane < L && i < m;
            r[k] = in ? (q[k].x << ib) | (uint32_t)(w0 + i) : ~0u;
            if (IT == 8 && in) key[IT * g.n + w0 + i] = q[k].y;
        }
        warp_sort256(r, lane, 8 * L);
        if (n > 256) {
            const uint32_t ahead = __shfl_down_sync(0xffffffffu, r[0], kTieRun / 8);
            far |= 8 * lane + kTieRun < m && r[0] >> ib == ahead >> ib;
        }
        reinterpret_cast<uint4*>(key + w0 + 8 * lane)[0] = make_uint4(r[0], r[1], r[2], r[3]);
        reinterpret_cast<uint4*>(key + w0 + 8 * lane)[1] = make_uint4(r[4], r[5], r[6], r[7]);
    }
    if (n > 256) {      // (more than a warp's: a block barrier)
        if (group_any(g, far)) return false;
        merge_levels_smem<IT>(key, (n + IT - 1) / IT * IT, 256, g);
    } else {
        g.sync();
    }
    for (int i = g.t; i + kTieRun < n; i += g.n) far |= key[i] >> ib == key[i + kTieRun] >> ib;
    if (group_any(g, far)) return false;
    const uint32_t im = (1u << ib) - 1u;
    auto slot = [&](uint32_t i) { return IT == 8 ? key[IT * g.n + i] : b[i].y; };
    constexpr int F = IT / 8;                      // entries in flight per thread (4 took 10% more)
    for (int i0 = g.t; i0 < n; i0 += F * g.n) {
        uint32_t x[F], e[F], p[F];
#pragma unroll
        for (int k = 0; k < F; k++) {
            const int i = i0 + k * g.n;
            x[k] = i < n ? key[i] : 0u;
            e[k] = i < n ? slot(x[k] & im) : 0u;
        }
#pragma unroll
        for (int k = 0; k < F; k++) p[k] = i0 + k * g.n < n ? pair(e[k]) : 0u;
#pragma unroll
        for (int k = 0; k < F; k++) {
            const int i = i0 + k * g.n;
            if (i >= n) break;
            const uint32_t low = x[k] >> ib;
            int first = i, pos = i;
            while (first > 0 && key[first - 1] >> ib == low) first--;
            if (first < i || (i + 1 < n && key[i + 1] >> ib == low)) {
                pos = first;
                for (int j = first; j < n && key[j] >> ib == low; j++) pos += slot(key[j] & im) < e[k];
            }
            put(pos, low, e[k], p[k]);
        }
    }
    return true;
}

// One tile's list of n <= IT g.n entries, sorted by the group g in shared memory
// (sk: 4 IT g.n bytes, 8 of them for each entry where 64-bit keys may be sorted,
// n <= 8 g.n).  Words where they serve, 64-bit keys otherwise; false if neither.
// 3M Gaussians, 4x1080p, all lists: 462 us with 64-bit keys, 257 us; without the
// emission slots in shared memory (IT = 8) 10% more.
template <int IT>
__device__ __forceinline__ bool tile_sort_group(const Views& V, int64_t gt, uint32_t s0, uint32_t n, unsigned long long* sk,
                                const SortGroup& g, uint2* bucket, const uint32_t* __restrict__ pid,
                                uint32_t* keys_sorted, uint32_t* vals_sorted, uint32_t* __restrict__ pid_sorted,
                                uint32_t* status, uint32_t cap)
{
    (void)status;
    (void)cap;
    const ViewDesc& vd = V.v[view_of_tile(V, gt)];
    const uint32_t hi_bits = (uint32_t)(gt - vd.tile_base) << vd.shift;
    auto pair = [&](uint32_t e) { return GS_DCHECK(e < cap, status) ? pid[e] : 0u; };
    auto put = [&](int i, uint32_t low, uint32_t e, uint32_t p) {
        keys_sorted[s0 + i] = hi_bits | low;
        vals_sorted[s0 + i] = e;
        pid_sorted[s0 + i] = p;
    };
    if (sort_words<IT>(bucket + s0, (int)n, 23 - vd.drop, reinterpret_cast<uint32_t*>(sk), g, pair, put)) return true;
    if (IT > 8) return false;
    g.sync();
    const int N = (int)((n + 7u) & ~7u);    // the last thread's keys padded
    for (int i = g.t; i < N; i += g.n) {
        unsigned long long x = ~0ull;
        if (i < (int)n) {
            const uint2 b = bucket[s0 + i];
            x = sort_key(b.x, b.y);
        }
        sk[i] = x;
    }
    g.sync();
    block_merge_sort_smem(sk, N, g);
    for (int i = g.t; i < (int)n; i += g.n) put(i, (uint32_t)(sk[i] >> 32), (uint32_t)sk[i], pair((uint32_t)sk[i]));
    return true;
}

// A list too long for shared memory, sorted by the whole block: chunks sorted in
// shared memory into the (keys, vals) arrays (twice kTileSortMax entries as words,
// or kTileSortMax 64-bit keys), then merge levels alternating between the arrays and
// the bucket.  8 scenes, 81,600 tiles, 854 lists above 4,096 entries of 31M entries in
// all: 1,130 -> 660 us for the whole sort, of which merge_level's pieces gave 120.
__device__ void tile_sort_chunked(const Views& V, int64_t gt, uint32_t s0, uint32_t n, unsigned long long* sk,
                                  uint2* bucket, const uint32_t* __restrict__ pid, uint32_t* keys_sorted,
                                  uint32_t* vals_sorted, uint32_t* __restrict__ pid_sorted, uint32_t* status,
                                  uint32_t cap)
{
    (void)status;
    (void)cap;
    const ViewDesc& vd = V.v[view_of_tile(V, gt)];
    const uint32_t hi_bits = (uint32_t)(gt - vd.tile_base) << vd.shift;
    const SortGroup g = whole_block();
    const PackedList pk{bucket};
    const SplitList sp{keys_sorted, vals_sorted};
    __shared__ uint32_t split[kTileSortThreads + 1];
    const int bits = 23 - vd.drop;
    const uint32_t M = bits + 13 <= 32 ? 2u * kTileSortMax : kTileSortMax;
    static_assert(kTileSortMax == 4096, "13 bits index a chunk of words");
    for (uint32_t c0 = 0; c0 < n; c0 += M) {
        const uint32_t len = min(M, n - c0);
        auto put = [&](int i, uint32_t low, uint32_t e, uint32_t) { sp.put(s0 + c0 + i, sort_key(low, e)); };
        if (!sort_words<16>(bucket + s0 + c0, (int)len, bits, reinterpret_cast<uint32_t*>(sk), g,
                            [](uint32_t) { return 0u; }, put)) {
            // by 64-bit keys, in two halves merged through the bucket where long
            for (uint32_t h0 = 0; h0 < len; h0 += kTileSortMax) {
                const uint32_t hl = min((uint32_t)kTileSortMax, len - h0);
                __syncthreads();
                for (uint32_t i = threadIdx.x; i < kTileSortMax; i += blockDim.x)
                    sk[i] = i < hl ? pk.get(s0 + c0 + h0 + i) : ~0ull;
                __syncthreads();
                block_merge_sort_smem(sk, kTileSortMax, g);
                for (uint32_t i = threadIdx.x; i < hl; i += blockDim.x)
                    if (len > kTileSortMax) pk.put(s0 + c0 + h0 + i, sk[i]);
                    else sp.put(s0 + c0 + i, sk[i]);
            }
            __syncthreads();
            if (len > kTileSortMax) merge_level(pk, sp, s0 + c0, len, kTileSortMax, sk, split);
        }
        __syncthreads();
    }
    bool in_bucket = false;
    for (uint32_t run = M; run < n; run <<= 1) {
        if (in_bucket) merge_level(pk, sp, s0, n, run, sk, split);
        else merge_level(sp, pk, s0, n, run, sk, split);
        in_bucket = !in_bucket;
    }
    constexpr int F = 4;                           // entries in flight per thread
    for (uint32_t i0 = threadIdx.x; i0 < n; i0 += F * blockDim.x) {
        unsigned long long x[F];
        uint32_t p[F];
#pragma unroll
        for (int k = 0; k < F; k++) {
            const uint32_t i = i0 + k * blockDim.x;
            x[k] = i >= n ? 0ull : in_bucket ? pk.get(s0 + i) : sp.get(s0 + i);
        }
#pragma unroll
        for (int k = 0; k < F; k++) {
            const uint32_t e = (uint32_t)x[k];
            p[k] = i0 + k * blockDim.x < n && GS_DCHECK(e < cap, status) ? pid[e] : 0u;
        }
#pragma unroll
        for (int k = 0; k < F; k++) {
            const uint32_t i = i0 + k * blockDim.x;
            if (i >= n) break;
            keys_sorted[s0 + i] = hi_bits | (uint32_t)(x[k] >> 32);
            vals_sorted[s0 + i] = (uint32_t)x[k];
            pid_sorted[s0 + i] = p[k];
        }
    }
}

// The tile order lists the tiles by size class (see len_bucket): long lists
// (>= 2047 entries), medium (1023-2046), short (255-1022), tiny (<= 254).
// Blocks of 512 threads take one long list each, or two medium, four short or
// sixteen tiny ones, by halves, quarters (with a named barrier each) or warps.
// Three blocks (1,536 threads) per SM: 40 registers serve every list up to 4,096
// entries; the 16-key form of longer ones spills there (3M Gaussians, 4x1080p: two
// blocks 326 us, three 257, four 251; 8 scenes with 854 longer lists: 802, 660, 680).
// One launch for all classes: 2,000 Gaussians 10.0 + 3 us of launch -> 8.7 us against
// two kernels, 4x1080p 248 -> 257.
__global__ void __launch_bounds__(kTileSortThreads, 3) k_tile_sort(Views V, const uint32_t* __restrict__ order,
                                                                   const uint2* __restrict__ ranges, uint2* bucket,
                                                                   const uint32_t* __restrict__ pid,
                                                                   uint32_t* keys_sorted, uint32_t* vals_sorted,
                                                                   uint32_t* __restrict__ pid_sorted,
                                                                   const WsHeader* __restrict__ hdr, uint32_t* status,
                                                                   uint32_t cap)
{
    if (!after_previous()) return;
    extern __shared__ unsigned long long sk[];
    const uint32_t t = threadIdx.x;
    uint32_t first = 0, b = blockIdx.x, split = 1;     // the block's class: its first list, lists per block
    for (int c = 0; c < 4; c++, split = c == 3 ? 16u : 2u * split) {
        const uint32_t lists = hdr->sort_class[c], blocks = (lists + split - 1u) / split;
        if (b < blocks) {
            const uint32_t n_t = kTileSortThreads / split, part = t / n_t, m = split * b + part;
            if (m >= lists) return;
            const int64_t gt = order[first + m];
            const uint2 r = range_at(ranges, gt, cap, status);
            const uint32_t n = r.y - r.x;
            if (n == 0 || (c > 0 && n > 8u * n_t)) return;
            const SortGroup g{(int)(t - part * n_t), (int)n_t, c == 0 ? 0 : 1 + (int)part};
            bool done = false;
            if (n <= 8u * n_t)
                done = tile_sort_group<8>(V, gt, r.x, n, sk + 8u * n_t * part, g, bucket, pid, keys_sorted, vals_sorted,
                                          pid_sorted, status, cap);
            else if (n <= 2u * kTileSortMax)
                done = tile_sort_group<16>(V, gt, r.x, n, sk, g, bucket, pid, keys_sorted, vals_sorted, pid_sorted,
                                           status, cap);
            if (!done)
                tile_sort_chunked(V, gt, r.x, n, sk, bucket, pid, keys_sorted, vals_sorted, pid_sorted, status, cap);
            return;
        }
        b -= blocks;
        first += lists;
    }
}

// ---------------------------------------------------------------------------

void launch_bin_sort(const Plan& P, const WsPtrs& w, cudaStream_t st)
{
    const Views& V = P.views;
    const uint32_t cap = (uint32_t)P.cap;
    // emission-slot scan, K and the capacity check; tile starts, ranges, the other
    // pairs' cursors and the launch order
    uint32_t* const total_at = w.offset + V.pairs;
    const bool one = V.tiles <= kScanBlock;
    const bool sums = !one || P.pair_groups > 64;      // else the one block sums the pairs itself
    const unsigned nparts = one ? 0u : (unsigned)P.tile_scan_parts;
    if (sums) {
        const unsigned gb = (unsigned)((P.pair_groups + kScanThreads / 32 - 1) / (kScanThreads / 32));
        launch_after(k_sort_sums, gb + nparts, kScanThreads, 0, st, w.count, V.pairs, w.gpart, P.pair_groups, gb,
                     V.tiles, w.tile_cnt, w.tile_part);
    }
    if (one) {
        launch_after(k_sort_setup, 1, 1024, 0, st, w.count, V.pairs, sums, w.gpart, P.pair_groups, (int)V.tiles,
                     w.tile_cnt, w.tile_cur, w.ranges, w.tile_order, total_at, w.hdr, cap);
    } else {
        launch_after(k_sort_parts, 1, 1024, 0, st, w.gpart, P.pair_groups, V.tiles, w.tile_part, nparts, total_at,
                     w.hdr, cap);
        launch_after(k_tile_down, nparts, kScanThreads, 0, st, V.tiles, w.tile_cnt, w.tile_part, w.tile_cur, w.ranges,
                     w.tile_order, w.hdr);
    }
    // generate keys into the tile buckets
    {
        const int64_t blocks = (V.pairs + kEmitThreads - 1) / kEmitThreads;
        launch_after(k_emit, (unsigned)blocks, kEmitThreads, 0, st, V, w.count, w.gpart, w.offset, w.rec, w.span,
                     w.rank, w.tile_cur, w.tile_cnt + V.tiles, w.bucket, w.pid, w.hdr);
    }
    // sort each tile's list
    {
        const size_t smem = sizeof(unsigned long long) * kTileSortMax;              // 32 KB: no opt-in needed
        launch_after(k_tile_sort, (unsigned)V.tiles, kTileSortThreads, smem, st, V, w.tile_order, w.ranges, w.bucket,
                     w.pid, w.keys_sorted, w.vals_sorted, w.pid_sorted, w.hdr, &w.hdr->status, cap);
    }
}

}  // namespace gs
