// k_sort.cu -- exclusive scans and a stable LSD radix sort of 64-bit keys.
//
// These are the data-movement primitives behind cover bucketing (sort of
// (element, point) keys), node emission (sort of (node, point) keys) and the
// nerve (sort-unique of (node, node) keys). The sort is stable, so sorting a
// key on its high field only keeps the low field's incoming order.
#include <cooperative_groups.h>

#include <algorithm>
#include <utility>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace mgb {

namespace {

// A slot's flags as a scan value: bit 0 (member) in the low half, bit 1 (root)
// in the high half of the sum, so that one scan counts both.
struct SlotFlag {
    uint8_t v;
    __device__ operator int64_t() const { return (int64_t)(v & 1) | ((int64_t)(v >> 1) << 32); }
};

// ---------------------------------------------------------------- scan
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t* total)
{
    __shared__ int64_t warp_sums[kScanThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < kScanThreads / 32 ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < kScanThreads / 32) warp_sums[lane] = w;
    }
    __syncthreads();
    const int64_t before = warp ? warp_sums[warp - 1] : 0;
    *total = warp_sums[kScanThreads / 32 - 1];
    __syncthreads();
    return before + x - v;
}

template <class T>
__global__ void __launch_bounds__(kScanThreads) scan_reduce_kernel(const T* __restrict__ in, int64_t n,
                                                                   int64_t* __restrict__ sums)
{
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t idx = base + (int64_t)threadIdx.x * kScanItems + i;
        if (idx < n) s += (int64_t)in[idx];
    }
    int64_t total;
    block_exclusive_scan(s, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

template <class T>
__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(const T* __restrict__ in, int64_t n,
                                                                  const int64_t* __restrict__ offs,
                                                                  int64_t* __restrict__ out)
{
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t v[kScanItems];
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t idx = base + (int64_t)threadIdx.x * kScanItems + i;
        v[i] = idx < n ? (int64_t)in[idx] : 0;
        s += v[i];
    }
    int64_t total;
    int64_t run = block_exclusive_scan(s, &total) + offs[blockIdx.x];
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t idx = base + (int64_t)threadIdx.x * kScanItems + i;
        if (idx < n) out[idx] = run;
        run += v[i];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) out[n] = run;
}

// Exclusive scan of up to kScanOneMax values in one CTA (one launch, no
// scratch): thread t scans kScanOneItems consecutive values, read as whole
// 128-byte lines by the warp.
constexpr int kScanOneThreads = 1024;
constexpr int kScanOneItems = 8;
constexpr int64_t kScanOneMax = kScanOneThreads * kScanOneItems;

template <class T>
__global__ void __launch_bounds__(kScanOneThreads) scan_one_kernel(const T* __restrict__ in, int64_t n,
                                                                   int64_t* __restrict__ out)
{
    __shared__ int64_t warp_sums[kScanOneThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t b = (int64_t)tid * kScanOneItems;
    int64_t it[kScanOneItems];
    int64_t v = 0;
#pragma unroll
    for (int i = 0; i < kScanOneItems; ++i) it[i] = b + i < n ? (int64_t)in[b + i] : 0;
#pragma unroll
    for (int i = 0; i < kScanOneItems; ++i) v += it[i];
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t w = warp_sums[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w;
    }
    __syncthreads();
    int64_t run = (warp ? warp_sums[warp - 1] : 0) + x - v;
#pragma unroll
    for (int i = 0; i < kScanOneItems; ++i) {
        if (b + i < n) out[b + i] = run;
        run += it[i];
    }
    if (tid == kScanOneThreads - 1) out[n] = warp_sums[kScanOneThreads / 32 - 1];
}

// Up to kScanSelfTiles tiles, each CTA adds up the sums of the tiles before
// its own (a few reads a thread, from L2) instead of a scan of the sums in
// launches between the two.
constexpr int64_t kScanSelfTiles = 2048;

template <class T>
__global__ void __launch_bounds__(kScanThreads) scan_self_kernel(const T* __restrict__ in, int64_t n,
                                                                 const int64_t* __restrict__ sums,
                                                                 int64_t* __restrict__ out)
{
    int64_t before = 0;
    for (int t = threadIdx.x; t < (int)blockIdx.x; t += kScanThreads) before += sums[t];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t v[kScanItems];
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t idx = base + (int64_t)threadIdx.x * kScanItems + i;
        v[i] = idx < n ? (int64_t)in[idx] : 0;
        s += v[i];
    }
    int64_t total, total_before;
    block_exclusive_scan(before, &total_before);
    int64_t run = block_exclusive_scan(s, &total) + total_before;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t idx = base + (int64_t)threadIdx.x * kScanItems + i;
        if (idx < n) out[idx] = run;
        run += v[i];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) out[n] = run;
}

template <class T>
cudaError_t exclusive_scan_impl(const T* in, int64_t* out, int64_t n, cudaStream_t s)
{
    // out[0..n) = exclusive prefix sums, out[n] = total
    if (n == 0) return cudaMemsetAsync(out, 0, sizeof(int64_t), s);
    if (n <= kScanOneMax) {
        { scan_one_kernel<T><<<1, kScanOneThreads, 0, s>>>(in, n, out); note_launch(); }
        return cudaGetLastError();
    }
    const int64_t nb = div_up(n, kScanTile);
    Buf sums, offs;
    MGB_TRY(sums.alloc(sizeof(int64_t) * nb, s));
    { scan_reduce_kernel<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, sums.as<int64_t>()); note_launch(); }
    MGB_TRY(cudaGetLastError());
    if (nb <= kScanSelfTiles) {
        { scan_self_kernel<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, sums.as<int64_t>(), out); note_launch(); }
        return cudaGetLastError();
    }
    MGB_TRY(offs.alloc(sizeof(int64_t) * (nb + 1), s));
    MGB_TRY(exclusive_scan_impl<int64_t>(sums.as<int64_t>(), offs.as<int64_t>(), nb, s));
    { scan_apply_kernel<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, offs.as<int64_t>(), out); note_launch(); }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- radix sort
//
// A key's sort field is bits [lo1, lo1 + w1) above bits [lo0, lo0 + w0) of it
// (w1 = 0: one range), taken in 8-bit digits from the low end.
//
// What bounds these sorts at the sizes of a graph (thousands to a few million
// keys of 8 bytes, all in L2) is launches and serial chains, not bandwidth:
//   n <= kRcMaxKeys   one launch for all digits: a cluster of up to 8 CTAs
//                     holds the keys in registers, the CTAs exchange their
//                     digit counts through distributed shared memory, and the
//                     cluster barrier separates the digits;
//   up to kRsSelfTiles tiles (4.2M keys): two launches a digit (counts per
//                     tile; then every CTA adds up the counts of the tiles
//                     before it, ranks its keys and writes them in runs);
//   more              the counts are scanned by launches in between (every
//                     CTA reading all counts would grow as tiles squared).
// Measured on whole graphs, against count, scan and scatter launches per
// digit (4 to 6 launches of ~10 us each): 13.7k x 37 (22k memberships, one
// cluster launch a sort) 1557 -> 1308 us; 230k x 128 balanced (330k, two
// launches a digit) 3293 -> 2977 us; 1M x 256 (1.25M) 7522 -> 7271 us.
constexpr int kRsBins = 256;

struct SortField {
    int lo0, w0, lo1, w1;
};

__device__ __forceinline__ uint64_t sort_field(uint64_t k, const SortField f)
{
    uint64_t v = k >> f.lo0;
    if (f.w0 < 64) v &= (1ull << f.w0) - 1ull;
    if (f.w1) v |= ((k >> f.lo1) & ((1ull << f.w1) - 1ull)) << f.w0;
    return v;
}

__device__ __forceinline__ int digit_of(uint64_t k, const SortField f, int shift, uint32_t mask)
{
    return (int)((uint32_t)(sort_field(k, f) >> shift) & mask);
}

// Ranks the warp's keys of one digit: warp w of the CTA owns `items` rounds of
// 32 consecutive keys, round by round in lane order, so ranks follow input
// order and the sort is stable. cnt: the warp's own counters (zeroed). at[r]:
// the key's digit, or -1 (no key); on return the digit, and above its 8 bits
// the number of the warp's earlier keys of that digit.
template <int ITEMS>
__device__ __forceinline__ void warp_rank(int (&at)[ITEMS], int items, uint16_t* cnt)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        if (r >= items) break;                                     // uniform
        const int dg = at[r];
        const unsigned peers = __match_any_sync(0xffffffffu, dg);
        const int before = dg >= 0 ? cnt[dg] : 0;
        __syncwarp();
        if (dg >= 0) {
            at[r] = dg | (before + __popc(peers & lt)) << 8;
            if ((peers & lt) == 0) cnt[dg] = (uint16_t)(before + __popc(peers));
        }
        __syncwarp();
    }
}

// Turns wcnt[w][b] (keys of warp w with digit b) into exclusive prefixes over
// the warps, and s_total[b] into their sum. 4 threads a digit, all threads.
template <int WARPS>
__device__ __forceinline__ void warp_prefixes(uint16_t (*wcnt)[kRsBins], int* s_total)
{
    constexpr int kPer = WARPS / 4;
    for (int e = threadIdx.x; e < 4 * kRsBins; e += blockDim.x) {
        const int b = e >> 2, q = e & 3;
        int c[kPer];
        int sum = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            c[i] = wcnt[q * kPer + i][b];
            sum += c[i];
        }
        int x = sum;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o, 4);
            if (q >= o) x += y;
        }
        int run = x - sum;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            wcnt[q * kPer + i][b] = (uint16_t)run;
            run += c[i];
        }
        if (q == 3) s_total[b] = x;
    }
}

// Exclusive scan of 256 values by the CTA's first 256 threads (reached by all
// threads): returns the prefix of thread b's value.
__device__ __forceinline__ int scan256(int v, int* s_warp)
{
    const int tid = threadIdx.x, lane = tid & 31;
    int x = tid < kRsBins ? v : 0;
    if (tid < kRsBins) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[tid >> 5] = x;
    }
    __syncthreads();
    int before = 0;
    if (tid < kRsBins)
        for (int w = 0; w < (tid >> 5); ++w) before += s_warp[w];
    __syncthreads();
    return before + x - v;
}

// ---- one launch: a cluster of CTAs
constexpr int kRcThreads = 1024;
constexpr int kRcWarps = kRcThreads / 32;
constexpr int kRcItems = 16;
constexpr int kRcCluster = 8;                        // the portable cluster size
constexpr int64_t kRcMaxKeys = (int64_t)kRcCluster * kRcThreads * kRcItems;

// CTA c of the cluster holds keys [c per, (c + 1) per), per = 1024 items. Per
// digit: ranks in registers, counts to the other CTAs, then the keys go
// through shared memory (sorted by digit there) so that they are written in
// runs. In place: every key is in registers before the first write.
// n_dev (if set): the number of keys, at most n.
__global__ void __launch_bounds__(kRcThreads) radix_cluster_kernel(uint64_t* __restrict__ keys, int64_t n, SortField f,
                                                                   int items,
                                                                   const unsigned long long* __restrict__ n_dev)
{
    if (n_dev) n = min(n, (int64_t)*n_dev);
    extern __shared__ uint64_t s_keys[];                           // 1024 items keys
    __shared__ __align__(16) uint16_t wcnt[kRcWarps][kRsBins];
    __shared__ int s_total[kRsBins];                               // this CTA's keys of each digit
    __shared__ int s_local[kRsBins];                               // their start in s_keys
    __shared__ int s_out[kRsBins];                                 // their start in the output
    __shared__ int s_warp[8];
    cg::cluster_group cluster = cg::this_cluster();
    const int c = (int)cluster.block_rank(), nc = (int)cluster.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t base = (int64_t)c * kRcThreads * items;
    const int here = (int)max((int64_t)0, min((int64_t)kRcThreads * items, n - base));
    const int w0 = warp * 32 * items;                              // the warp's first key of the CTA's
    const int width = f.w0 + f.w1;
    for (int shift = 0; shift < width; shift += 8) {
        const uint32_t mask = width - shift < 8 ? (1u << (width - shift)) - 1u : 255u;
        uint64_t key[kRcItems];
        int at[kRcItems];
#pragma unroll
        for (int r = 0; r < kRcItems; ++r) {
            if (r >= items) break;
            const int i = w0 + r * 32 + lane;
            key[r] = i < here ? __ldcg(keys + base + i) : 0ull;
            at[r] = i < here ? digit_of(key[r], f, shift, mask) : -1;
        }
        for (int e = lane; e < kRsBins / 2; e += 32) reinterpret_cast<uint32_t*>(wcnt[warp])[e] = 0u;
        __syncwarp();
        warp_rank<kRcItems>(at, items, wcnt[warp]);
        __syncthreads();
        warp_prefixes<kRcWarps>(wcnt, s_total);
        cluster.sync();                                            // counts written, keys read
        int all = 0, before = 0, mine = 0;
        if (tid < kRsBins) {
            mine = s_total[tid];
            for (int o = 0; o < nc; ++o) {
                const int v = cluster.map_shared_rank(s_total, o)[tid];
                all += v;
                if (o < c) before += v;
            }
        }
        const int start = scan256(all, s_warp);
        const int local = scan256(mine, s_warp);
        if (tid < kRsBins) {
            s_local[tid] = local;
            s_out[tid] = start + before - local;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRcItems; ++r) {
            if (r >= items) break;
            const int dg = at[r] & 255;
            if (at[r] >= 0) s_keys[s_local[dg] + wcnt[warp][dg] + (at[r] >> 8)] = key[r];
        }
        __syncthreads();
        for (int i = tid; i < here; i += kRcThreads) {
            const uint64_t k = s_keys[i];
            __stcg(keys + s_out[digit_of(k, f, shift, mask)] + i, k);
        }
        __threadfence();
        cluster.sync();                                            // keys written, counts read
    }
}

// ---- two launches a digit
constexpr int kRsThreads = 1024;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsItems = 8;                          // most rounds per warp
constexpr int64_t kRsSelfTiles = 512;
constexpr int64_t kRsFill = 152;                     // CTAs that fill the chip

// A CTA's tile is kRsThreads * items keys: as few rounds as fill the chip once,
// because a CTA's time is the chain of its rounds (with 16 rounds in 512 threads
// a digit of 330k keys took 13 + 14 us on 41 CTAs, of 1.25M 13 + 19 on 153).
// SELF: hist[block * 256 + digit] (int32); else offs[digit * nblocks + block]
// (int64), the layout that one scan turns into output offsets.
template <bool SELF>
__global__ void __launch_bounds__(kRsThreads) radix_hist_kernel(const uint64_t* __restrict__ keys, int64_t n,
                                                                SortField f, int shift, uint32_t mask, int items,
                                                                void* __restrict__ hist)
{
    __shared__ int cnt[kRsBins];
    if (threadIdx.x < kRsBins) cnt[threadIdx.x] = 0;
    const int64_t base = (int64_t)blockIdx.x * kRsThreads * items;
    const int lane = threadIdx.x & 31;
    uint64_t key[kRsItems];
#pragma unroll
    for (int r = 0; r < kRsItems; ++r) {
        const int64_t idx = base + (int64_t)r * kRsThreads + threadIdx.x;
        key[r] = r < items && idx < n ? keys[idx] : 0ull;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsItems; ++r) {
        if (r >= items) break;                                     // uniform
        const int64_t idx = base + (int64_t)r * kRsThreads + threadIdx.x;
        // one shared-memory atomic per distinct digit of the warp: runs of
        // equal digits (nearly sorted input) would serialise
        const int dg = idx < n ? digit_of(key[r], f, shift, mask) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, dg);
        if (dg >= 0 && (peers & ((1u << lane) - 1u)) == 0) atomicAdd(&cnt[dg], __popc(peers));
    }
    __syncthreads();
    if (threadIdx.x < kRsBins) {
        const int b = threadIdx.x;
        if (SELF) static_cast<int32_t*>(hist)[(int64_t)blockIdx.x * kRsBins + b] = cnt[b];
        else static_cast<int64_t*>(hist)[(int64_t)b * gridDim.x + blockIdx.x] = cnt[b];
    }
}

template <bool SELF>
__global__ void __launch_bounds__(kRsThreads) radix_scatter_kernel(const uint64_t* __restrict__ in,
                                                                   uint64_t* __restrict__ out, int64_t n, SortField f,
                                                                   int shift, uint32_t mask, int items,
                                                                   const void* __restrict__ hist)
{
    extern __shared__ uint64_t s_keys[];                           // the tile's keys
    __shared__ __align__(16) uint16_t wcnt[kRsWarps][kRsBins];
    __shared__ int s_total[kRsBins], s_local[kRsBins];
    __shared__ int64_t s_out[kRsBins];
    __shared__ int s_part[2][4][kRsBins];
    __shared__ int s_warp[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t base = (int64_t)blockIdx.x * kRsThreads * items;
    const int here = (int)min((int64_t)kRsThreads * items, n - base);
    const int w0 = warp * 32 * items;                              // the warp's first key of the tile
    uint64_t key[kRsItems];
    int at[kRsItems];
#pragma unroll
    for (int r = 0; r < kRsItems; ++r) {
        const int i = w0 + r * 32 + lane;
        const bool valid = r < items && i < here;
        key[r] = valid ? in[base + i] : 0ull;
        at[r] = valid ? digit_of(key[r], f, shift, mask) : -1;
    }
    if (SELF) {
        // four threads a digit, each over a quarter of the tiles
        const int32_t* h = static_cast<const int32_t*>(hist);
        const int b = tid & (kRsBins - 1), q = tid >> 8;
        const int nb = (int)gridDim.x, me = (int)blockIdx.x;
        int all = 0, before = 0;
#pragma unroll 8
        for (int t = q; t < nb; t += 4) {
            const int v = __ldg(h + (int64_t)t * kRsBins + b);
            all += v;
            if (t < me) before += v;
        }
        s_part[0][q][b] = all;
        s_part[1][q][b] = before;
    }
    for (int e = lane; e < kRsBins / 2; e += 32) reinterpret_cast<uint32_t*>(wcnt[warp])[e] = 0u;
    __syncwarp();
    warp_rank<kRsItems>(at, items, wcnt[warp]);
    __syncthreads();
    warp_prefixes<kRsWarps>(wcnt, s_total);
    __syncthreads();
    const int mine = tid < kRsBins ? s_total[tid] : 0;
    const int local = scan256(mine, s_warp);
    int start = 0, before = 0;
    if (SELF) {
        int all = 0;
        if (tid < kRsBins) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                all += s_part[0][q][tid];
                before += s_part[1][q][tid];
            }
        }
        start = scan256(all, s_warp);
    }
    if (tid < kRsBins) {
        s_local[tid] = local;
        s_out[tid] = (SELF ? (int64_t)start + before
                           : static_cast<const int64_t*>(hist)[(int64_t)tid * gridDim.x + blockIdx.x]) - local;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsItems; ++r) {
        const int dg = at[r] & 255;
        if (at[r] >= 0) s_keys[s_local[dg] + wcnt[warp][dg] + (at[r] >> 8)] = key[r];
    }
    __syncthreads();
    for (int i = tid; i < here; i += kRsThreads) {
        const uint64_t k = s_keys[i];
        out[s_out[digit_of(k, f, shift, mask)] + i] = k;
    }
}

cudaError_t radix_sort_cluster(uint64_t* keys, int64_t n, const SortField& f, cudaStream_t s,
                               const unsigned long long* n_dev = nullptr)
{
    // the keys spread over the CTAs of the cluster: fewer rounds each
    int nc = 1;
    while (nc < kRcCluster && n > (int64_t)nc * kRcThreads) nc *= 2;
    const int items = (int)((n + (int64_t)nc * kRcThreads - 1) / ((int64_t)nc * kRcThreads));
    const size_t smem = sizeof(uint64_t) * kRcThreads * items;
    MGB_TRY(cudaFuncSetAttribute(radix_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(uint64_t) * kRcThreads * kRcItems)));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nc);
    cfg.blockDim = dim3(kRcThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    note_launch();
    return cudaLaunchKernelEx(&cfg, radix_cluster_kernel, keys, n, f, items, n_dev);
}

cudaError_t radix_sort_field(Buf& keys, Buf& tmp, int64_t n, const SortField& f, cudaStream_t s)
{
    const int width = f.w0 + f.w1;
    if (n <= 1 || width <= 0) return cudaSuccess;
    if (n <= kRcMaxKeys) return radix_sort_cluster(keys.as<uint64_t>(), n, f, s);
    const int items = (int)std::min<int64_t>(kRsItems, div_up(n, (int64_t)kRsThreads * kRsFill));
    const int tile = kRsThreads * items;
    const int64_t nb = div_up(n, tile);
    const bool self = nb <= kRsSelfTiles;
    Buf hist, offs;
    MGB_TRY(hist.alloc((self ? sizeof(int32_t) : sizeof(int64_t)) * kRsBins * nb, s));
    if (!self) MGB_TRY(offs.alloc(sizeof(int64_t) * (kRsBins * nb + 1), s));
    const size_t smem = sizeof(uint64_t) * tile, most = sizeof(uint64_t) * kRsThreads * kRsItems;
    if (self) MGB_TRY(cudaFuncSetAttribute(radix_scatter_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
    else MGB_TRY(cudaFuncSetAttribute(radix_scatter_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
    for (int shift = 0; shift < width; shift += 8) {
        const uint32_t mask = width - shift < 8 ? (1u << (width - shift)) - 1u : 255u;
        const uint64_t* src = keys.as<uint64_t>();
        uint64_t* dst = tmp.as<uint64_t>();
        const unsigned g = (unsigned)nb;
        if (self) {
            radix_hist_kernel<true><<<g, kRsThreads, 0, s>>>(src, n, f, shift, mask, items, hist.p);
            MGB_TRY(cudaGetLastError());
            radix_scatter_kernel<true><<<g, kRsThreads, smem, s>>>(src, dst, n, f, shift, mask, items, hist.p);
        } else {
            radix_hist_kernel<false><<<g, kRsThreads, 0, s>>>(src, n, f, shift, mask, items, hist.p);
            MGB_TRY(cudaGetLastError());
            MGB_TRY(exclusive_scan_i64(hist.as<int64_t>(), offs.as<int64_t>(), kRsBins * nb, s));
            radix_scatter_kernel<false><<<g, kRsThreads, smem, s>>>(src, dst, n, f, shift, mask, items, offs.p);
        }
        note_launch(2);
        MGB_TRY(cudaGetLastError());
        std::swap(keys, tmp);
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t exclusive_scan_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, cudaStream_t s)
{
    return exclusive_scan_impl<int32_t>(in, out, n, s);
}

cudaError_t exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t s)
{
    return exclusive_scan_impl<int64_t>(in, out, n, s);
}

cudaError_t exclusive_scan_slot_flags(const uint8_t* in, int64_t* out, int64_t n, cudaStream_t s)
{
    return exclusive_scan_impl<SlotFlag>(reinterpret_cast<const SlotFlag*>(in), out, n, s);
}

cudaError_t radix_sort_u64(Buf& keys, Buf& tmp, int64_t n, int lo_bit, int hi_bit, cudaStream_t s)
{
    return radix_sort_field(keys, tmp, n, SortField{lo_bit, hi_bit - lo_bit, 0, 0}, s);
}

cudaError_t radix_sort_u64_two_dev(uint64_t* keys, int64_t n_max, const unsigned long long* n_dev, int lo0, int lo1,
                                   int bits, cudaStream_t s)
{
    if (n_max > kRcMaxKeys) return cudaErrorInvalidValue;
    return radix_sort_cluster(keys, n_max, SortField{lo0, bits, lo1, bits}, s, n_dev);
}

cudaError_t radix_sort_u64_two(Buf& keys, Buf& tmp, int64_t n, int lo0, int lo1, int bits, cudaStream_t s)
{
    return radix_sort_field(keys, tmp, n, SortField{lo0, bits, lo1, bits}, s);
}

}  // namespace mgb
