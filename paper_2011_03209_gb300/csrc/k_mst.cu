// k_mst.cu -- single-linkage forest of every cover element.
//
// "Mapper Interactive" §5: Lum et al. cluster each cover element by single
// linkage, where the tool uses DBSCAN. Single linkage cut at a height h gives
// the connected components of the h-graph; the whole dendrogram up to eps is
// the minimum spanning forest of the element's eps-graph (pairs with d2 <=
// eps^2, the DBSCAN distance). Edges are ordered by the key (d2, smaller
// point, larger point), so the forest is unique when distances tie.
//
// Borůvka rounds over the tile pairs of the element (those not certified
// all-out at eps by the tile layout's bounding spheres), every round on CUDA
// cores:
//   1. the FP32 sum of squared differences s of every pair whose rows lie in
//      two components and which may be within eps (s <= the FP32 screen's
//      upper limit): the smallest s of each component (atomicMin), and in the
//      same pass a queue of the pairs whose s lies within the FP32 error of
//      the smallest seen so far (|s - d2| <= eta d2 + tiny; the limits only
//      fall, so the pairs within the final limit are all in the queue);
//   2. the queued pairs still within their component's final limit (the
//      lightest edge is among them) get their FP64 d2 by the defining
//      expression, one a thread, and, when d2 <= eps^2, their key competes for
//      the component's lightest edge (a 128-bit atomic minimum of (d2, slots));
//      a round whose queue overflows screens its pairs again instead;
//   3. every component adds its lightest edge to the forest (once for an
//      edge two components chose) and joins the other component
//      (lock-free union-find whose roots are the smallest point index).
// One screen a round (two before, the second with its FP64 sums inside the
// tile loop, a warp's slot for every pair): 19.1 -> 4.0 ms of screens and 0.47
// of FP64 on the 100k x 64 cover of 50 elements (5 rounds).
// Within an element the cover slots are in ascending point order, so slot
// indices order the ties as point indices do. Tile pairs whose rows all share
// one component drop out of later rounds.
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstring>
#include <string>
#include <utility>

#include "../../include/mapper.h"
#include "dbscan.cuh"

namespace mgb {

namespace {

constexpr int kT = kTile;

__device__ __forceinline__ int mfind(int32_t* parent, int x)
{
    volatile int32_t* par = parent;
    int p = par[x];
    while (p != x) {
        const int gp = par[p];
        if (gp != p) par[x] = gp;
        x = p;
        p = par[x];
    }
    return x;
}

// Joins two components; the root of larger point index goes under the other.
__device__ __forceinline__ void munion(int32_t* parent, const int32_t* row_pt, int a, int b)
{
    while (true) {
        a = mfind(parent, a);
        b = mfind(parent, b);
        if (a == b) return;
        if (row_pt[a] < row_pt[b]) { const int t = a; a = b; b = t; }
        if (atomicCAS(&parent[a], a, b) == a) return;
    }
}

__device__ __forceinline__ double msf_sqdist(const float* __restrict__ x, const float* __restrict__ y, int d)
{
    double s = 0.0;
    for (int k = 0; k < d; ++k) {
        const double t = __dsub_rn((double)x[k], (double)y[k]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// 128-bit keys: y = bits of d2 (non-negative doubles order as their bits),
// x = (smaller slot << 32) | larger slot; the minimum is lexicographic in (y, x).
__device__ __forceinline__ bool key_less(ulonglong2 a, ulonglong2 b)
{
    return a.y < b.y || (a.y == b.y && a.x < b.x);
}

__device__ __forceinline__ ulonglong2 cas128(ulonglong2* addr, ulonglong2 cmp, ulonglong2 val)
{
    unsigned long long lo, hi;
    asm volatile(
        "{\n .reg .b128 c, v, o;\n mov.b128 c, {%2, %3};\n mov.b128 v, {%4, %5};\n"
        " atom.relaxed.gpu.global.cas.b128 o, [%6], c, v;\n mov.b128 {%0, %1}, o;\n}"
        : "=l"(lo), "=l"(hi)
        : "l"(cmp.x), "l"(cmp.y), "l"(val.x), "l"(val.y), "l"(addr)
        : "memory");
    return make_ulonglong2(lo, hi);
}

__device__ __forceinline__ void key_min(ulonglong2* addr, ulonglong2 k)
{
    const volatile unsigned long long* va = reinterpret_cast<const volatile unsigned long long*>(addr);
    ulonglong2 cur = make_ulonglong2(va[0], va[1]);       // may be torn: the CAS returns the true value
    while (key_less(k, cur)) {
        const ulonglong2 old = cas128(addr, cur, k);
        if (old.x == cur.x && old.y == cur.y) return;
        cur = old;
    }
}

struct MsfArgs {
    PassArgs A;                     // rows (G or X via row_pt), dp, d, pairs, tile_n, eps2, hi_thr
    const int32_t* root;            // component root row of every row (this round)
    const int32_t* row_slot;
    unsigned* cmin;                 // per root row: the smallest FP32 s of its candidate pairs (as bits)
    ulonglong2* ckey;               // per root row: the lightest candidate edge's key
    float eta, tiny;                // |s - d2| <= eta d2 + tiny
    int4* queue;                    // candidate pairs: (row a, row b, bits of s, 0)
    unsigned long long* queue_n;    // their number (may pass the capacity: then they are not used)
    unsigned long long queue_cap;
    unsigned long long* oob;        // checked build: indices found out of range
};

// s of a component's lightest edge is at most m (1 + eta)^2 / (1 - eta) +
// 2 tiny, m the component's smallest s
__device__ __forceinline__ float key_limit(const MsfArgs& M, float m)
{
    return __fmaf_ru(m, 4.f * M.eta, __fadd_ru(m, 2.f * M.tiny));
}

// The FP64 key of a pair, against the lightest edges of its components.
__device__ __forceinline__ void key_pair(const MsfArgs& M, int64_t ra, int64_t rb, int root_a, int root_b, bool ca,
                                         bool cb)
{
    const PassArgs& A = M.A;
    const double d2 = msf_sqdist(pass_row(A, ra), pass_row(A, rb), A.d);
    if (!(d2 <= A.eps2)) return;
    const unsigned s1 = (unsigned)M.row_slot[ra], s2 = (unsigned)M.row_slot[rb];
    const ulonglong2 key = make_ulonglong2(((unsigned long long)min(s1, s2) << 32) | (unsigned long long)max(s1, s2),
                                           (unsigned long long)__double_as_longlong(d2));
    if (ca) key_min(&M.ckey[root_a], key);
    if (cb) key_min(&M.ckey[root_b], key);
}

// STAGE 1: component minima of s, and the queue of the pairs near them. STAGE
// 2 (after a queue that overflowed): the exact keys of the pairs near the final
// minima. Bound by the FP32 pipe (simt_tile_sums); per tile pair one atomic for
// each row and column.
template <int STAGE>
__global__ void __launch_bounds__(256, 2) msf_screen_kernel(const MsfArgs M)
{
    __shared__ __align__(16) float As[kSimtK][kSimtPad];
    __shared__ __align__(16) float Bs[kSimtK][kSimtPad];
    __shared__ int s_root[2 * kT];
    __shared__ unsigned s_min[2 * kT];                         // smallest s of each row and column
    __shared__ float s_lim[2 * kT];
    __shared__ unsigned s_n;
    __shared__ unsigned long long s_base;
    const PassArgs& A = M.A;
    const int tid = threadIdx.x;
    if (A.n_dev && (unsigned long long)blockIdx.x >= *A.n_dev) return;
    const int2 p = A.pairs[blockIdx.x];
    int ta = p.x, tb = p.y & kPairTileMask;
    bool ok = true;
    if (!MGB_IN_RANGE(ta, A.n_tiles, M.oob) || !MGB_IN_RANGE(tb, A.n_tiles, M.oob)) {
        ta = tb = 0;                                       // checked build: counted, then skipped
        ok = false;
    }
    const int64_t sa = (int64_t)ta * kT, sb = (int64_t)tb * kT;
    const int na = ok ? A.tile_n[ta] : 0, nb = ok ? A.tile_n[tb] : 0;
    const bool diag = ta == tb;
    s_root[tid] = tid < kT ? (tid < na ? M.root[sa + tid] : -1) : (tid - kT < nb ? M.root[sb + tid - kT] : -2);
    s_min[tid] = 0x7f800000u;
    if (tid == 0) s_n = 0u;

    const int tx = tid & 15, ty = tid >> 4;
    float acc[8][8];
    simt_tile_sums(A, sa, sb, na, nb, As, Bs, acc);

    auto row_of = [&](int i) { return i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4; };
    auto col_of = [&](int j) { return j < 4 ? tx * 4 + j : 64 + tx * 4 + j - 4; };
    // a pair of rows in two components that may lie within eps (diagonal:
    // once); other pairs get s = inf
    float rmin[8], cmin[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { rmin[i] = INFINITY; cmin[i] = INFINITY; }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = row_of(i), ra = s_root[r];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = col_of(j);
            if (r >= na || c >= nb || (diag && c <= r) || ra == s_root[kT + c] || !(acc[i][j] <= A.hi_thr))
                acc[i][j] = INFINITY;
            rmin[i] = fminf(rmin[i], acc[i][j]);
            cmin[j] = fminf(cmin[j], acc[i][j]);
        }
    }
    if (STAGE == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) rmin[i] = fminf(rmin[i], __shfl_xor_sync(0xffffffffu, rmin[i], o));
            cmin[i] = fminf(cmin[i], __shfl_xor_sync(0xffffffffu, cmin[i], 16));
            if (tx == 0) s_min[row_of(i)] = __float_as_uint(rmin[i]);          // (non-negative floats order as bits)
            if ((tid & 16) == 0 && cmin[i] < INFINITY) atomicMin(&s_min[kT + col_of(i)], __float_as_uint(cmin[i]));
        }
        __syncthreads();
        const unsigned mine = s_min[tid];
        if (mine < 0x7f800000u) atomicMin(&M.cmin[s_root[tid]], mine);
        __syncthreads();
    }
    // limits of the rows' and columns' components (stage 1: so far)
    const bool live = STAGE == 1 ? s_min[tid] < 0x7f800000u : s_root[tid] >= 0;
    s_lim[tid] = live ? key_limit(M, __uint_as_float(__ldcg(M.cmin + s_root[tid]))) : -1.f;
    __syncthreads();
    unsigned long long near = 0ull;                            // bit 8 i + j: a candidate
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float lr = s_lim[row_of(i)];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (acc[i][j] <= fmaxf(lr, s_lim[kT + col_of(j)]) && acc[i][j] < INFINITY) near |= 1ull << (8 * i + j);
    }
    if (STAGE == 1) {
        unsigned at = 0u;
        if (near) at = atomicAdd(&s_n, (unsigned)__popcll(near));
        __syncthreads();
        if (tid == 0) s_base = s_n ? atomicAdd(M.queue_n, (unsigned long long)s_n) : 0ull;
        __syncthreads();
        unsigned long long pos = s_base + at;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if ((near >> (8 * i + j)) & 1ull) {
                    if (pos < M.queue_cap)
                        M.queue[pos] = make_int4((int)(sa + row_of(i)), (int)(sb + col_of(j)),
                                                 __float_as_int(acc[i][j]), 0);
                    ++pos;
                }
    } else if (near) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if ((near >> (8 * i + j)) & 1ull) {
                    const int r = row_of(i), c = col_of(j);
                    key_pair(M, sa + r, sb + c, s_root[r], s_root[kT + c], acc[i][j] <= s_lim[r],
                             acc[i][j] <= s_lim[kT + c]);
                }
    }
}

// The queued pairs within a final limit: compacted per block first, because a
// warp's FP64 instruction costs the same however few lanes take part.
constexpr int kEvalPer = 8;

__global__ void __launch_bounds__(256) msf_eval_kernel(const MsfArgs M)
{
    __shared__ int2 s_row[256 * kEvalPer];
    __shared__ uint8_t s_side[256 * kEvalPer];
    __shared__ unsigned s_n;
    const unsigned long long n = *M.queue_n;
    if (n > M.queue_cap) return;                               // the pairs are screened again
    for (unsigned long long b = (unsigned long long)blockIdx.x * (256 * kEvalPer); b < n;
         b += (unsigned long long)gridDim.x * (256 * kEvalPer)) {
        if (threadIdx.x == 0) s_n = 0u;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kEvalPer; ++k) {
            const unsigned long long i = b + (unsigned long long)(k * 256 + (int)threadIdx.x);
            if (i >= n) continue;
            const int4 e = M.queue[i];
            const float s = __int_as_float(e.z);
            const bool ca = s <= key_limit(M, __uint_as_float(M.cmin[M.root[e.x]]));
            const bool cb = s <= key_limit(M, __uint_as_float(M.cmin[M.root[e.y]]));
            if (!ca && !cb) continue;
            const unsigned at = atomicAdd(&s_n, 1u);
            s_row[at] = make_int2(e.x, e.y);
            s_side[at] = (uint8_t)((ca ? 1 : 0) | (cb ? 2 : 0));
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < s_n; i += blockDim.x) {
            const int2 r = s_row[i];
            key_pair(M, r.x, r.y, M.root[r.x], M.root[r.y], s_side[i] & 1, s_side[i] & 2);
        }
        __syncthreads();
    }
}

// Each component root with a candidate adds its lightest edge (once when
// both components chose the same edge) and joins the other component.
__global__ void msf_pick_kernel(const int32_t* __restrict__ root, const ulonglong2* __restrict__ ckey,
                                const int32_t* __restrict__ slot_row, const int32_t* __restrict__ slot_point,
                                const int32_t* __restrict__ slot_elem, const int32_t* __restrict__ row_pt, int64_t R,
                                int32_t* parent, int32_t* __restrict__ e_u, int32_t* __restrict__ e_v,
                                int32_t* __restrict__ e_elem, int32_t* __restrict__ e_su, int32_t* __restrict__ e_sv,
                                double* __restrict__ e_d2, unsigned long long* n_edges, unsigned long long* picks,
                                const unsigned long long* queue_n, unsigned long long queue_cap)
{
    if (*queue_n > queue_cap) return;                          // the keys are not there yet
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= R || root[x] != (int32_t)x) return;
    const ulonglong2 k = ckey[x];
    if (k.y == ~0ull) return;
    const int s1 = (int)(k.x >> 32), s2 = (int)(k.x & 0xffffffffull);
    const int r1 = slot_row[s1], r2 = slot_row[s2];
    const int other = root[r1] == (int32_t)x ? root[r2] : root[r1];
    atomicAdd(picks, 1ull);
    const ulonglong2 ko = ckey[other];
    if (!(ko.x == k.x && ko.y == k.y) || x < other) {
        const unsigned long long at = atomicAdd(n_edges, 1ull);
        e_u[at] = slot_point[s1];
        e_v[at] = slot_point[s2];
        e_elem[at] = slot_elem[s1];
        e_su[at] = s1;
        e_sv[at] = s2;
        e_d2[at] = __longlong_as_double((long long)k.y);
    }
    munion(parent, row_pt, (int)x, other);
}

__global__ void msf_flatten_kernel(int32_t* parent, const int32_t* __restrict__ row_slot, int64_t R,
                                   int32_t* __restrict__ root, unsigned* __restrict__ cmin,
                                   ulonglong2* __restrict__ ckey)
{
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= R) return;
    root[x] = row_slot[x] >= 0 ? mfind(parent, (int)x) : (int32_t)x;
    cmin[x] = 0x7f800000u;                                 // +inf
    ckey[x] = make_ulonglong2(~0ull, ~0ull);
}

__global__ void msf_init_kernel(const int32_t* __restrict__ row_slot, int64_t R, int32_t* __restrict__ parent,
                                int32_t* __restrict__ slot_row)
{
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= R) return;
    parent[x] = (int32_t)x;
    if (row_slot[x] >= 0) slot_row[row_slot[x]] = (int32_t)x;
}

// Per tile: the smallest and largest root of its valid rows.
__global__ void msf_tile_roots_kernel(const int32_t* __restrict__ root, const int32_t* __restrict__ tile_n,
                                      int64_t T, int2* __restrict__ tr)
{
    const int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (t >= T) return;
    int lo = INT_MAX, hi = INT_MIN;
    for (int r = lane; r < tile_n[t]; r += 32) {
        const int v = root[t * kT + r];
        lo = min(lo, v);
        hi = max(hi, v);
    }
    for (int o = 16; o; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) tr[t] = make_int2(lo, hi);
}

// Keeps the tile pairs whose rows are not all in one component.
__global__ void msf_filter_kernel(const int2* __restrict__ pairs, int64_t n, const unsigned long long* __restrict__ n_in,
                                  const int2* __restrict__ tr, int2* __restrict__ out, unsigned long long* n_out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || (n_in && (unsigned long long)i >= *n_in)) return;
    const int2 p = pairs[i];
    const int2 a = tr[p.x], b = tr[p.y & kPairTileMask];
    if (a.x == a.y && b.x == b.y && a.x == b.x) return;
    out[atomicAdd(n_out, 1ull)] = p;
}

// Single-linkage cut in cover-slot space: slots of one component (edges
// with d2 <= h^2) take the smallest slot as root (slot order = point order
// within an element).
__global__ void cut_init_kernel(int64_t M, int32_t* __restrict__ parent)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < M) parent[i] = (int32_t)i;
}

__device__ __forceinline__ void slot_union(int32_t* parent, int a, int b)
{
    while (true) {
        a = mfind(parent, a);
        b = mfind(parent, b);
        if (a == b) return;
        if (a < b) { const int t = a; a = b; b = t; }
        if (atomicCAS(&parent[a], a, b) == a) return;
    }
}

__global__ void cut_union_kernel(const int32_t* __restrict__ e_su, const int32_t* __restrict__ e_sv,
                                 const double* __restrict__ e_d2, int64_t n, double h2, int32_t* parent)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && e_d2[i] <= h2) slot_union(parent, e_su[i], e_sv[i]);
}

__global__ void cut_labels_kernel(int32_t* parent, const int32_t* __restrict__ slot_point, int64_t M,
                                  int32_t* __restrict__ lab, uint8_t* __restrict__ flags,
                                  int64_t* __restrict__ slot_label,
                                  uint8_t* __restrict__ core)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    const int r = mfind(parent, (int)i);
    lab[i] = r;
    slot_label[i] = slot_point[r];
    flags[i] = r == (int)i ? 3 : 1;
    core[i] = 1;
}

// Sort keys of the edges: word `which` (0 sv, 1 su, 2 and 3 the halves of d2's
// bits, 4 the element) of edge order[i] (order null: edge i) above the edge.
__global__ void edge_word_kernel(const int32_t* __restrict__ su, const int32_t* __restrict__ sv,
                                 const double* __restrict__ d2, const int32_t* __restrict__ elem, int64_t n, int which,
                                 const uint64_t* __restrict__ order, uint64_t* __restrict__ keys)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t e = order ? (uint32_t)order[i] : (uint32_t)i;
    const unsigned long long bits = (unsigned long long)__double_as_longlong(d2[e]);
    const uint32_t w = which == 0 ? (uint32_t)sv[e] : which == 1 ? (uint32_t)su[e] : which == 2 ? (uint32_t)bits
                     : which == 3 ? (uint32_t)(bits >> 32) : (uint32_t)elem[e];
    keys[i] = ((uint64_t)w << 32) | e;
}

__global__ void edge_gather_kernel(const uint64_t* __restrict__ order, int64_t n, const int32_t* __restrict__ u,
                                   const int32_t* __restrict__ v, const int32_t* __restrict__ elem,
                                   const int32_t* __restrict__ su, const int32_t* __restrict__ sv,
                                   const double* __restrict__ d2, int32_t* __restrict__ ou, int32_t* __restrict__ ov,
                                   int32_t* __restrict__ oelem, int32_t* __restrict__ osu, int32_t* __restrict__ osv,
                                   double* __restrict__ od2)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t e = (uint32_t)order[i];
    ou[i] = u[e];
    ov[i] = v[e];
    oelem[i] = elem[e];
    osu[i] = su[e];
    osv[i] = sv[e];
    od2[i] = d2[e];
}

int word_bits(uint32_t most)          // bits of the values 0 .. most, at least 1
{
    int b = 1;
    while (b < 32 && (most >> b)) ++b;
    return b;
}

// Orders the edges by (element, d2, u, v): stable sorts of words from the last
// to the first (non-negative doubles order as their bits; slots order as
// points within an element). At 130k edges a fraction of a millisecond;
// sorting the copied arrays on the host takes tens.
cudaError_t sort_forest(ForestOut* out, int64_t M, int64_t E, double eps2, cudaStream_t s)
{
    const int64_t n = out->n;
    if (n <= 1) return cudaSuccess;
    Buf order, tmp, ou, ov, oelem, osu, osv, od2;
    MGB_TRY(order.alloc(sizeof(uint64_t) * n, s));
    MGB_TRY(tmp.alloc(sizeof(uint64_t) * n, s));
    const unsigned g = (unsigned)div_up(n, 256);
    unsigned long long e2 = 0;
    std::memcpy(&e2, &eps2, sizeof(e2));
    const int bits[5] = {word_bits((uint32_t)M), word_bits((uint32_t)M), 32, word_bits((uint32_t)(e2 >> 32)),
                         word_bits((uint32_t)E)};
    for (int w = 0; w < 5; ++w) {
        edge_word_kernel<<<g, 256, 0, s>>>(out->su.as<int32_t>(), out->sv.as<int32_t>(), out->d2.as<double>(),
                                           out->elem.as<int32_t>(), n, w, w ? order.as<uint64_t>() : nullptr,
                                           tmp.as<uint64_t>());
        note_launch();
        MGB_TRY(cudaGetLastError());
        std::swap(order, tmp);
        MGB_TRY(radix_sort_u64(order, tmp, n, 32, 32 + bits[w], s));
    }
    MGB_TRY(ou.alloc(sizeof(int32_t) * M, s));
    MGB_TRY(ov.alloc(sizeof(int32_t) * M, s));
    MGB_TRY(oelem.alloc(sizeof(int32_t) * M, s));
    MGB_TRY(osu.alloc(sizeof(int32_t) * M, s));
    MGB_TRY(osv.alloc(sizeof(int32_t) * M, s));
    MGB_TRY(od2.alloc(sizeof(double) * M, s));
    edge_gather_kernel<<<g, 256, 0, s>>>(order.as<uint64_t>(), n, out->u.as<int32_t>(), out->v.as<int32_t>(),
                                         out->elem.as<int32_t>(), out->su.as<int32_t>(), out->sv.as<int32_t>(),
                                         out->d2.as<double>(), ou.as<int32_t>(), ov.as<int32_t>(), oelem.as<int32_t>(),
                                         osu.as<int32_t>(), osv.as<int32_t>(), od2.as<double>());
    note_launch();
    MGB_TRY(cudaGetLastError());
    out->u = std::move(ou);
    out->v = std::move(ov);
    out->elem = std::move(oelem);
    out->su = std::move(osu);
    out->sv = std::move(osv);
    out->d2 = std::move(od2);
    return cudaSuccess;
}

}  // namespace

int msf_forest(const PassArgs& a, const int32_t* row_slot, const int32_t* slot_point, const int32_t* slot_elem,
               int64_t M, int64_t E, int64_t R, int64_t T, int64_t n_pairs, size_t queue_bytes,
               ForestOut* out, cudaStream_t s)
{
#define MK(expr)                                                                   \
    do {                                                                           \
        cudaError_t e_ = (expr);                                                   \
        if (e_ != cudaSuccess) {                                                   \
            set_error(std::string("single linkage: ") + cudaGetErrorString(e_));   \
            return e_ == cudaErrorMemoryAllocation ? MAPPER_ENOMEM : MAPPER_ECUDA;  \
        }                                                                          \
    } while (0)
    out->n = 0;
    const int64_t cap = std::max<int64_t>(M, 1);
    MK(out->u.alloc(sizeof(int32_t) * cap, s));
    MK(out->v.alloc(sizeof(int32_t) * cap, s));
    MK(out->elem.alloc(sizeof(int32_t) * cap, s));
    MK(out->su.alloc(sizeof(int32_t) * cap, s));
    MK(out->sv.alloc(sizeof(int32_t) * cap, s));
    MK(out->d2.alloc(sizeof(double) * cap, s));
    if (R == 0 || n_pairs == 0) return MAPPER_OK;           // no pair can lie within eps
    Buf parent, root, slot_row, cmin, ckey, tr, lists[2], counts, queue;
    MK(parent.alloc(sizeof(int32_t) * R, s));
    MK(root.alloc(sizeof(int32_t) * R, s));
    MK(slot_row.alloc(sizeof(int32_t) * cap, s));
    MK(cmin.alloc(sizeof(unsigned) * R, s));
    MK(ckey.alloc(sizeof(ulonglong2) * R, s));
    MK(tr.alloc(sizeof(int2) * std::max<int64_t>(T, 1), s));
    MK(lists[0].alloc(sizeof(int2) * std::max<int64_t>(n_pairs, 1), s));
    MK(lists[1].alloc(sizeof(int2) * std::max<int64_t>(n_pairs, 1), s));
    MK(counts.alloc(sizeof(unsigned long long) * 6, s));       // n_edges, picks, queue, list lengths, index checks
    unsigned long long* n_edges = counts.as<unsigned long long>();
    unsigned long long* picks = n_edges + 1;
    unsigned long long* queue_n = n_edges + 2;
    unsigned long long* len = n_edges + 3;
    unsigned long long* oob = n_edges + 5;
    MK(cudaMemsetAsync(counts.p, 0, sizeof(unsigned long long) * 6, s));
    // every row queues its nearest so far, a few times over (about log(tile
    // pairs of its element) each). That is 128 bytes a row, so the queue keeps to
    // queue_bytes and takes what can be had: a round that overflows it (at worst
    // all of them) is screened twice.
    unsigned long long queue_cap = 8ull * (unsigned long long)R;
    if (queue_bytes) queue_cap = std::min<unsigned long long>(queue_cap, queue_bytes / sizeof(int4));
    for (;; queue_cap /= 2) {
        const cudaError_t e = queue.alloc(sizeof(int4) * queue_cap, s);
        if (e == cudaSuccess) break;
        if (e != cudaErrorMemoryAllocation || queue_cap == 0) MK(e);
        cudaGetLastError();
    }
    const unsigned gR = (unsigned)div_up(R, 256);
    msf_init_kernel<<<gR, 256, 0, s>>>(row_slot, R, parent.as<int32_t>(), slot_row.as<int32_t>());
    MK(cudaGetLastError());
    MK(cudaMemcpyAsync(lists[0].p, a.pairs, sizeof(int2) * n_pairs, cudaMemcpyDeviceToDevice, s));
    MK(cudaMemcpyAsync(len, &n_pairs, sizeof(unsigned long long), cudaMemcpyHostToDevice, s));
    MsfArgs m{};
    m.A = a;
    m.root = root.as<int32_t>();
    m.row_slot = row_slot;
    m.cmin = cmin.as<unsigned>();
    m.ckey = ckey.as<ulonglong2>();
    m.eta = (float)(1.5 * (a.d + 4) * std::ldexp(1.0, -24));
    m.oob = oob;
    m.tiny = (float)(3.0 * (a.d + 2) * std::ldexp(1.0, -149));
    if (m.tiny == 0.f) m.tiny = std::ldexp(1.0f, -149);
    m.queue = queue.as<int4>();
    m.queue_n = queue_n;
    m.queue_cap = queue_cap;
    const unsigned g_eval = (unsigned)std::min<int64_t>(div_up(R, 256), 152 * 4);
    int cur = 0;
    for (int round = 0; round < 64; ++round) {
        msf_flatten_kernel<<<gR, 256, 0, s>>>(parent.as<int32_t>(), row_slot, R, root.as<int32_t>(), cmin.as<unsigned>(),
                                             ckey.as<ulonglong2>());
        // drop the tile pairs whose rows are all in one component
        msf_tile_roots_kernel<<<(unsigned)div_up(T, 8), 256, 0, s>>>(root.as<int32_t>(), a.tile_n, T, tr.as<int2>());
        MK(cudaMemsetAsync(len + 1 - cur, 0, sizeof(unsigned long long), s));
        msf_filter_kernel<<<(unsigned)div_up(n_pairs, 256), 256, 0, s>>>(lists[cur].as<int2>(), n_pairs, len + cur,
                                                                           tr.as<int2>(), lists[1 - cur].as<int2>(),
                                                                           len + 1 - cur);
        cur = 1 - cur;
        MK(cudaMemsetAsync(picks, 0, sizeof(unsigned long long) * 2, s));          // and queue_n
        note_launch(3);
        m.A.pairs = lists[cur].as<int2>();
        m.A.n_dev = len + cur;
        auto pick = [&]() {
            msf_pick_kernel<<<gR, 256, 0, s>>>(root.as<int32_t>(), ckey.as<ulonglong2>(), slot_row.as<int32_t>(),
                                               slot_point, slot_elem, a.row_pt, R, parent.as<int32_t>(),
                                               out->u.as<int32_t>(), out->v.as<int32_t>(), out->elem.as<int32_t>(),
                                               out->su.as<int32_t>(), out->sv.as<int32_t>(), out->d2.as<double>(),
                                               n_edges, picks, queue_n, queue_cap);
        };
        msf_screen_kernel<1><<<(unsigned)n_pairs, 256, 0, s>>>(m);
        msf_eval_kernel<<<g_eval, 256, 0, s>>>(m);
        pick();
        note_launch(3);
        MK(cudaGetLastError());
        unsigned long long h[2] = {0, 0};
        MK(cudaMemcpyAsync(h, picks, sizeof(h), cudaMemcpyDeviceToHost, s));
        MK(cudaStreamSynchronize(s));
        if (h[1] > queue_cap) {
            MK(cudaMemsetAsync(queue_n, 0, sizeof(unsigned long long), s));
            msf_screen_kernel<2><<<(unsigned)n_pairs, 256, 0, s>>>(m);
            pick();
            note_launch(2);
            MK(cudaGetLastError());
            MK(cudaMemcpyAsync(h, picks, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
            MK(cudaStreamSynchronize(s));
        }
        if (h[0] == 0) break;
    }
    unsigned long long ne = 0, h_oob = 0;
    MK(cudaMemcpyAsync(&ne, n_edges, sizeof(ne), cudaMemcpyDeviceToHost, s));
    MK(cudaMemcpyAsync(&h_oob, oob, sizeof(h_oob), cudaMemcpyDeviceToHost, s));
    MK(cudaStreamSynchronize(s));
    out->n = (int64_t)ne;
    if (h_oob) {
        set_error("single linkage: a device-side index check failed");
        return MAPPER_EINTERNAL;
    }
    MK(sort_forest(out, M, E, a.eps2, s));
#undef MK
    return MAPPER_OK;
}

int msf_cut(const ForestOut& f, const int32_t* slot_point, int64_t M, double h, int32_t* lab, uint8_t* flags,
            int64_t* slot_label, uint8_t* core, cudaStream_t s)
{
    if (M == 0) return MAPPER_OK;
    Buf parent;
    cudaError_t e = parent.alloc(sizeof(int32_t) * M, s);
    if (e == cudaSuccess) {
        cut_init_kernel<<<(unsigned)div_up(M, 256), 256, 0, s>>>(M, parent.as<int32_t>());
        if (f.n > 0)
            cut_union_kernel<<<(unsigned)div_up(f.n, 256), 256, 0, s>>>(f.su.as<int32_t>(), f.sv.as<int32_t>(),
                                                                         f.d2.as<double>(), f.n, h * h,
                                                                         parent.as<int32_t>());
        cut_labels_kernel<<<(unsigned)div_up(M, 256), 256, 0, s>>>(parent.as<int32_t>(), slot_point, M, lab, flags,
                                                                     slot_label, core);
        note_launch(3);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error(std::string("single-linkage cut: ") + cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? MAPPER_ENOMEM : MAPPER_ECUDA;
    }
    return MAPPER_OK;
}

}  // namespace mgb
