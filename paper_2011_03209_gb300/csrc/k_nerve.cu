// k_nerve.cu -- nodes and the 1D nerve ("Mapper Interactive" §3: the clusters
// of every cover element are the nodes; an edge joins two nodes whose point
// sets intersect).
//
// Nodes are numbered by the cover slot of their root (slots are ordered by
// element, then point), i.e. by (element, canonical id). Memberships become
// (node << 32 | point) keys, sorted into per-node member lists; the same
// memberships in point order (kept by the cover) give the nodes of each point,
// whose pairs go through a hash set of the distinct edges, sorted at the end.
// Without that order (given nodes, cover subsets), or with more edges than the
// set takes, the memberships re-keyed as (point << 32 | node) and sorted group
// the nodes of each point, every pair of them is emitted as (u << 32 | v), u < v,
// and a sort-unique of those keys gives the edge list in lexicographic order.
#include "dbscan.cuh"

namespace mgb {

namespace {

__global__ void member_keys_kernel(const int32_t* __restrict__ lab, const int64_t* __restrict__ pos,
                                   const int32_t* __restrict__ slot_point,
                                   const int32_t* __restrict__ slot_elem, const int32_t* __restrict__ slot_o, int64_t M,
                                   uint64_t* __restrict__ keys, int32_t* __restrict__ node_elem,
                                   int32_t* __restrict__ node_o)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= M) return;
    const int l = lab[s];
    const int node = l < 0 ? -1 : (int)(pos[l] >> 32);
    if (node_o) node_o[slot_o[s]] = node;
    if (l < 0) return;
    keys[(uint32_t)pos[s]] = ((uint64_t)(uint32_t)node << 32) | (uint64_t)(uint32_t)slot_point[s];
    if (l == (int)s) node_elem[node] = slot_elem[s];
}

// keys2 (if set): the same memberships as (point << 32 | node)
__global__ void node_offsets_kernel(const uint64_t* __restrict__ keys, int64_t G, int64_t N,
                                    int64_t* __restrict__ node_off, int32_t* __restrict__ members,
                                    uint64_t* __restrict__ keys2)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G) return;
    const uint64_t k = keys[i];
    const int64_t node = (int64_t)(k >> 32);
    members[i] = (int32_t)(uint32_t)k;
    if (keys2) keys2[i] = ((k & 0xffffffffull) << 32) | (uint64_t)node;
    if (i == 0 || (int64_t)(keys[i - 1] >> 32) != node) node_off[node] = i;
    if (i == G - 1) node_off[N] = G;
}

// Nerve edges from the nodes of every membership in point order (node_o, -1:
// none; pt: the memberships' points): each pair of a point's nodes goes through a
// hash set of the distinct edges, and the thread that adds one to the set
// appends it to the list. A thread takes a membership against the later ones of
// its point (a thread a point walked all k (k - 1) / 2 pairs of a point in k
// elements by itself: 2000 points in 255 elements with 0.996 overlap 24 ms of
// nerve, now 0.5). Memberships of a point ascend in element, and nodes in
// (element, root), so u < v. A pair seen before is one read of the set (in L2);
// the edges are few (hundreds) beside the points, so sorting all pairs, or the
// memberships by point, would move far more. counts[0]: edges, counts[1]: set when
// the list or a probe run is full. A CTA's threads stop at the first pair that it
// has no place for, and a CTA that starts later at once (a read of the flag at
// every membership, all of one address, cost more than it saved: nerve of 868k
// memberships and 1.0 M edges 0.85 -> 1.35 ms).
constexpr int kEdgeProbes = 64;

__global__ void __launch_bounds__(256) edge_set_kernel(const int32_t* __restrict__ pt, int64_t M,
                                                       const int32_t* __restrict__ node_o,
                                                       unsigned long long* set, uint32_t mask,
                                                       uint64_t* __restrict__ list, uint32_t cap,
                                                       unsigned long long* counts)
{
    __shared__ volatile int s_full;                  // counts[1] as the CTA knows it
    if (threadIdx.x == 0) s_full = __ldcg(counts + 1) != 0ull;
    __syncthreads();
    const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= M || s_full) return;
    const int u = node_o[a], p = pt[a];
    if (u < 0) return;
    for (int64_t b = a + 1; b < M && pt[b] == p; ++b) {
        const int v = node_o[b];
        if (v < 0) continue;
        // (v in the high half: the sorted list is then the int32 pairs (u, v))
        const unsigned long long key = ((unsigned long long)(unsigned)v << 32) | (unsigned)u;
        unsigned long long x = key * 0x9E3779B97F4A7C15ull;
        uint32_t h = (uint32_t)(x >> 40) & mask;
        int tries = 0;
        for (; tries < kEdgeProbes; ++tries, h = (h + 1) & mask) {
            unsigned long long cur = __ldcg(set + h);
            if (cur == key) break;
            if (cur != ~0ull) continue;
            if (s_full) return;
            cur = atomicCAS(set + h, ~0ull, key);
            if (cur == key) break;
            if (cur != ~0ull) continue;
            const unsigned long long at = atomicAdd(&counts[0], 1ull);
            if (at >= cap) {
                s_full = 1;
                counts[1] = 1ull;
                return;
            }
            list[at] = key;
            break;
        }
        if (tries == kEdgeProbes) {
            s_full = 1;
            counts[1] = 1ull;
            return;
        }
    }
}

// Nerve keys (point << 32 | node) of given nodes: member i belongs to the
// node u with node_off[u] <= i < node_off[u + 1].
__global__ void node_member_keys_kernel(const int64_t* __restrict__ node_off, int64_t N, int64_t G,
                                        const int32_t* __restrict__ members, uint64_t* __restrict__ keys2)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G) return;
    int64_t lo = 0, hi = N;                    // last u with node_off[u] <= i
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (node_off[mid] <= i) lo = mid; else hi = mid;
    }
    keys2[i] = ((uint64_t)(uint32_t)members[i] << 32) | (uint64_t)lo;
}

// Slot -> element index of a cover whose element offsets are elem_off[0..k].
__global__ void fill_slot_elem_kernel(const int64_t* __restrict__ elem_off, int32_t k, int64_t M,
                                      int32_t* __restrict__ slot_elem)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    int32_t lo = 0, hi = k;                    // last e with elem_off[e] <= i
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (elem_off[mid] <= i) lo = mid; else hi = mid;
    }
    slot_elem[i] = lo;
}

__global__ void run_pairs_kernel(const uint64_t* __restrict__ keys2, int64_t G,
                                 int64_t* __restrict__ cnt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G) return;
    const uint64_t pt = keys2[i] >> 32;
    int64_t c = 0;
    if (i == 0 || (keys2[i - 1] >> 32) != pt) {
        int64_t len = 1;
        while (i + len < G && (keys2[i + len] >> 32) == pt) ++len;
        c = len * (len - 1) / 2;
    }
    cnt[i] = c;
}

__global__ void emit_pairs_kernel(const uint64_t* __restrict__ keys2, int64_t G,
                                  const int64_t* __restrict__ pos, uint64_t* __restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G) return;
    const uint64_t pt = keys2[i] >> 32;
    if (!(i == 0 || (keys2[i - 1] >> 32) != pt)) return;
    int64_t len = 1;
    while (i + len < G && (keys2[i + len] >> 32) == pt) ++len;
    int64_t o = pos[i];
    for (int64_t a = 0; a < len; ++a)
        for (int64_t b = a + 1; b < len; ++b)
            out[o++] = ((keys2[i + a] & 0xffffffffull) << 32) | (keys2[i + b] & 0xffffffffull);
}

__global__ void unique_flags_kernel(const uint64_t* __restrict__ k, int64_t P,
                                    int32_t* __restrict__ flag)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P) return;
    flag[i] = (i == 0 || k[i] != k[i - 1]);
}

__global__ void unique_emit_kernel(const uint64_t* __restrict__ k, const int32_t* __restrict__ flag,
                                   const int64_t* __restrict__ pos, int64_t P,
                                   int32_t* __restrict__ edges)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P || !flag[i]) return;
    const int64_t o = pos[i];
    edges[2 * o] = (int32_t)(k[i] >> 32);
    edges[2 * o + 1] = (int32_t)(uint32_t)k[i];
}

inline unsigned grid_for(int64_t n, int t = 256) { return (unsigned)std::max<int64_t>(1, div_up(n, t)); }

}  // namespace

cudaError_t member_keys(const int32_t* lab, const int64_t* pos, const int32_t* slot_point, const int32_t* slot_elem,
                        const int32_t* slot_o, int64_t M, uint64_t* keys, int32_t* node_elem, int32_t* node_o,
                        cudaStream_t s)
{
    if (M == 0) return cudaSuccess;
    { member_keys_kernel<<<grid_for(M), 256, 0, s>>>(lab, pos, slot_point, slot_elem, slot_o, M, keys, node_elem,
                                                   node_o); note_launch(); }
    return cudaGetLastError();
}

cudaError_t node_offsets(const uint64_t* keys, int64_t G, int64_t N, int64_t* node_off, int32_t* members,
                         uint64_t* keys2, cudaStream_t s)
{
    if (G == 0) return cudaMemsetAsync(node_off, 0, sizeof(int64_t) * (N + 1), s);
    { node_offsets_kernel<<<grid_for(G), 256, 0, s>>>(keys, G, N, node_off, members, keys2); note_launch(); }
    return cudaGetLastError();
}

cudaError_t edge_set(const int32_t* pt, int64_t M, const int32_t* node_o, int64_t cap, Buf* list,
                     unsigned long long* counts, cudaStream_t s)
{
    if (cap > kEdgeListMax) return cudaErrorInvalidValue;
    constexpr uint32_t kSlots = 4 * kEdgeListMax;
    Buf set;
    MGB_TRY(set.alloc(sizeof(uint64_t) * kSlots, s));
    MGB_TRY(list->alloc(sizeof(uint64_t) * cap, s));
    MGB_TRY(cudaMemsetAsync(set.p, 0xff, sizeof(uint64_t) * kSlots, s));
    MGB_TRY(cudaMemsetAsync(counts, 0, 2 * sizeof(unsigned long long), s));
    edge_set_kernel<<<grid_for(M), 256, 0, s>>>(pt, M, node_o, set.as<unsigned long long>(), kSlots - 1,
                                                list->as<uint64_t>(), (uint32_t)cap, counts);
    note_launch();
    return cudaGetLastError();
}

cudaError_t node_member_keys(const int64_t* node_off, int64_t N, int64_t G, const int32_t* members,
                             uint64_t* keys2, cudaStream_t s)
{
    if (G == 0 || N == 0) return cudaSuccess;
    { node_member_keys_kernel<<<grid_for(G), 256, 0, s>>>(node_off, N, G, members, keys2); note_launch(); }
    return cudaGetLastError();
}

cudaError_t fill_slot_elem(const int64_t* elem_off, int32_t k, int64_t M, int32_t* slot_elem, cudaStream_t s)
{
    if (M == 0 || k == 0) return cudaSuccess;
    { fill_slot_elem_kernel<<<grid_for(M), 256, 0, s>>>(elem_off, k, M, slot_elem); note_launch(); }
    return cudaGetLastError();
}

cudaError_t run_pairs(const uint64_t* keys2, int64_t G, int64_t* cnt, cudaStream_t s)
{
    if (G == 0) return cudaSuccess;
    { run_pairs_kernel<<<grid_for(G), 256, 0, s>>>(keys2, G, cnt); note_launch(); }
    return cudaGetLastError();
}

cudaError_t emit_pairs(const uint64_t* keys2, int64_t G, const int64_t* pos, uint64_t* out,
                       cudaStream_t s)
{
    if (G == 0) return cudaSuccess;
    { emit_pairs_kernel<<<grid_for(G), 256, 0, s>>>(keys2, G, pos, out); note_launch(); }
    return cudaGetLastError();
}

cudaError_t unique_flags(const uint64_t* k, int64_t P, int32_t* flag, cudaStream_t s)
{
    if (P == 0) return cudaSuccess;
    { unique_flags_kernel<<<grid_for(P), 256, 0, s>>>(k, P, flag); note_launch(); }
    return cudaGetLastError();
}

cudaError_t unique_emit(const uint64_t* k, const int32_t* flag, const int64_t* pos, int64_t P,
                        int32_t* edges, cudaStream_t s)
{
    if (P == 0) return cudaSuccess;
    { unique_emit_kernel<<<grid_for(P), 256, 0, s>>>(k, flag, pos, P, edges); note_launch(); }
    return cudaGetLastError();
}

}  // namespace mgb
