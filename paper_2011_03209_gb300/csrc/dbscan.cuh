// dbscan.cuh -- internal interface of the per-element DBSCAN stage: tile
// layout (k_tiles.cu), screening passes (k_dbscan.cu, k_tc.cu) and graph
// assembly (k_nerve.cu).
#pragma once

#include "common.cuh"

namespace mgb {

constexpr int kTile = 128;          // rows per tile (one tcgen05 M block)

// A union-pass list entry may carry a flag in bit 30 of its second tile:
// the A-tile cores already share one root and the B-tile cores another, so
// one neighbour pair between them is enough (no per-pair unions).
constexpr int kPairOneEach = 1 << 30;
constexpr int kPairTileMask = kPairOneEach - 1;

enum : int { kStatBand = 0, kStatTies = 1, kStatScreened = 2, kStatCore = 3, kStatTileOut = 4,
             kStatTileIn = 5, kStatSkipped = 6, kStatTcPairs = 7, kStatSimtPairs = 8, kStatFp64 = 9,
             kStatUnion = 10, kStatRedo = 11, kStatOob = 12, kStatRedoBlocks = 13, kStatRedoParts = 14,
             kStatCount = 15 };

// Work lists of tile pairs, classified by bounding spheres.
enum : int { kListAllIn = 0, kListTC = 1, kListSimt = 2, kListCount = 3 };

// Arguments of one screening pass. Rows are points of one element laid out
// in tiles of kTile rows; a tile pair (a, b), a <= b, belongs to one element.
//   explicit mode (pairs != nullptr): tile pair q is pairs[q] (tile indices),
//     tile t spans rows [t*kTile, t*kTile + tile_n[t]);
//   implicit mode: every tile pair of every element, elements given by
//     elem_off (rows) and pair_off (tile pairs), rows = cover slots.
struct PassArgs {
    const float* G;              // FP32 rows, pitch dp floats (zero padded), or nullptr:
    const float* X;              //   then row r is X + row_pt[r] * ld (d columns)
    int64_t ld;
    bool xvec;                   //   X rows 16-byte aligned (float4 loads)
    int dp;                      // row pitch (multiple of 32)
    int d;                       // true dimension
    const int2* pairs;           // explicit list, or nullptr
    const unsigned long long* n_dev;   // explicit list: its length on the device, if set
                                       //   (launches cover an upper bound; the rest exit)
    const int32_t* tile_n;       // valid rows per tile (explicit mode)
    const int64_t* elem_off;     // implicit mode: [E+1] row offsets of the elements
    const int64_t* pair_off;     // implicit mode: [E+1] tile-pair offsets
    int E;
    float lo_thr, hi_thr;        // FP32 screen: in if s <= lo_thr, out if s > hi_thr
    double eps2;                 // eps * eps in double
    double tie_thr;              // 1e-12 * eps2
    const int32_t* row_pt;       // point index of each row (nullptr: the row index)
    int32_t* count;              // pass 1 output, per row
    int32_t* nbr;                // pass 1: first `cap` neighbour rows of each row
    int cap;                     //   (0: no lists)
    int need = INT_MAX;          // pass 1: a count of at least this many is not needed exactly (more
                                 //   may stay uncounted): minPts, which decides the core flag and
                                 //   is above every list; INT_MAX: exact counts
    uint8_t* pair_hit;           // pass 1 (explicit mode, optional): set to 1 for each tile
                                 //   pair with a neighbour pair, or one left to the recheck
    const uint8_t* core;         // passes 2, 3
    int32_t* parent;             // pass 2 union-find over rows
    const int32_t* root;         // pass 3 (flattened)
    unsigned long long* border;  // pass 3 output: (canonical point << 32 | root row), min
    unsigned long long* stats;   // kStat* counters
    int64_t n_rows, n_tiles;     // rows and tiles of the layout (index checks of the checked build)
};

// Row `row` of a pass (the tile layout's FP32 rows, or the input rows).
__device__ __forceinline__ const float* pass_row(const PassArgs& A, int64_t row)
{
    return A.G ? A.G + row * A.dp : A.X + (int64_t)A.row_pt[row] * A.ld;
}

// Columns 4 k4 .. 4 k4 + 3 of a row from pass_row (zero from column d on).
__device__ __forceinline__ float4 pass_ld4(const PassArgs& A, const float* p, int k4)
{
    if (A.G) return reinterpret_cast<const float4*>(p)[k4];
    const int k = 4 * k4;
    if (A.xvec && k + 3 < A.d) return *reinterpret_cast<const float4*>(p + k);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < A.d) v.x = p[k];
    if (k + 1 < A.d) v.y = p[k + 1];
    if (k + 2 < A.d) v.z = p[k + 2];
    if (k + 3 < A.d) v.w = p[k + 3];
    return v;
}

// Packed FP32 pairs (each half rounded as the scalar instruction).
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void f2_unpack(unsigned long long v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// acc += (a + b)^2 per half, one rounding each for the sum and the FMA
__device__ __forceinline__ void f2_sq_acc(unsigned long long& acc, unsigned long long a, unsigned long long b)
{
    unsigned long long t;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(a), "l"(b));
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(acc) : "l"(t));
}

constexpr int kSimtK = 32;      // columns staged per step
constexpr int kSimtPad = 132;   // shared-memory row pitch (floats)

// FP32 sums of squared differences of the rows sa .. sa + 127 and sb .. sb +
// 127 (rows past na, nb count as zeros) by 256 threads: thread (ty, tx) =
// (tid / 16, tid % 16) gets rows 4 ty + i, 64 + 4 ty + i - 4 and columns 4 tx
// + j, 64 + 4 tx + j - 4; columns of a row in order, an FMA each. B is staged
// negated, so that a difference is a packed add. Bound by the FP32 pipe, which
// retires a packed instruction at half the rate of a scalar one, so packing
// saves issue slots, not the pipe (count pass of the 65k x 64 FP32 graph 341 ->
// 297 us, pivot assignment 102 -> 93).
__device__ __forceinline__ void simt_tile_sums(const PassArgs& A, int64_t sa, int64_t sb, int na, int nb,
                                               float (*As)[kSimtPad], float (*Bs)[kSimtPad], float (&acc)[8][8])
{
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    unsigned long long s[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = 0ull;
    for (int k0 = 0; k0 < A.dp; k0 += kSimtK) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int idx = tid + 256 * v;       // float4 index in the 128 x 32 chunk
            const int r = idx >> 3, k4 = (idx & 7) * 4;
            float4 xa = make_float4(0.f, 0.f, 0.f, 0.f), xb = xa;
            if (r < na) xa = pass_ld4(A, pass_row(A, sa + r), (k0 + k4) >> 2);
            if (r < nb) xb = pass_ld4(A, pass_row(A, sb + r), (k0 + k4) >> 2);
            As[k4 + 0][r] = xa.x; As[k4 + 1][r] = xa.y; As[k4 + 2][r] = xa.z; As[k4 + 3][r] = xa.w;
            Bs[k4 + 0][r] = -xb.x; Bs[k4 + 1][r] = -xb.y; Bs[k4 + 2][r] = -xb.z; Bs[k4 + 3][r] = -xb.w;
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < kSimtK; ++k) {
            const float4 a0 = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[k][64 + ty * 4]);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[k][tx * 4]);
            const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[k][64 + tx * 4]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const unsigned long long b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned long long aa = f2_pack(a[i], a[i]);
#pragma unroll
                for (int j = 0; j < 4; ++j) f2_sq_acc(s[i][j], aa, b[j]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) f2_unpack(s[i][j], acc[i][2 * j], acc[i][2 * j + 1]);
}

// FP32 screen thresholds for eps2 at dimension d: a pair is certainly a
// neighbour when the FP32 screen value is <= *lo, certainly not when > *hi.
void fp32_thresholds(double eps2, int d, float* lo, float* hi);

// --- screening passes (k_dbscan.cu)
cudaError_t simt_pass(int mode, const PassArgs& a, int64_t n_pairs, cudaStream_t s);
cudaError_t allin_pass(int mode, const PassArgs& a, int64_t n_pairs, cudaStream_t s);
// mode 2 once the neighbour lists have joined most rows (tile_roots: scratch, [T])
cudaError_t allin_unions(const PassArgs& a, int64_t n_pairs, int64_t T, int2* tile_roots, cudaStream_t s);
cudaError_t core_flags(const int32_t* count, int64_t R, int32_t min_pts, uint8_t* core,
                       int32_t* parent, unsigned long long* border, unsigned long long* stats,
                       cudaStream_t s);
cudaError_t flatten(const int32_t* parent, const uint8_t* core, int64_t R, int32_t* root,
                    cudaStream_t s);
cudaError_t border_from_lists(const int32_t* count, const int32_t* nbr, int cap,
                              const uint8_t* core, const int32_t* root, const int32_t* row_pt,
                              int64_t R, unsigned long long* border, cudaStream_t s,
                              unsigned long long* oob = nullptr);
// Row space -> cover-slot space: per slot the root slot of its node (or -1),
// canonical point id (or -1), the flags of exclusive_scan_slot_flags and the
// core flag.
// Unions of each core row with the core rows of its pass-1 neighbour list.
// root: scratch of R entries.
cudaError_t list_unions(const int32_t* count, const int32_t* nbr, int cap, const uint8_t* core, int32_t* parent,
                        int32_t* root, const int32_t* row_pt, int64_t R, cudaStream_t s,
                        unsigned long long* oob = nullptr);
cudaError_t rows_to_slots(const int32_t* row_slot, const int32_t* row_pt, const uint8_t* core,
                          const int32_t* root, const unsigned long long* border, int64_t R,
                          int32_t* lab, uint8_t* flags,
                          int64_t* slot_label, uint8_t* slot_core, cudaStream_t s);
cudaError_t element_offsets(const uint64_t* keys, int64_t M, int64_t E, int64_t* elem_off,
                            cudaStream_t s);
// f[row_pt[row] * m + j] = count[row] for every non-padding row (the rows of
// a one-element cover of the whole cloud: the density filter).
cudaError_t counts_to_lens(const int32_t* row_slot, const int32_t* row_pt, const int32_t* count, int64_t R,
                           double* f, int m, int j, cudaStream_t s);
// The tile pairs of a union round: appends to `out` the pairs of a.pairs[0 .. n)
// flagged in a.pair_hit with lo < b - a <= hi and (filter) core rows that do not
// all share one root yet (flagging kPairOneEach pairs); *count (zeroed by the
// caller) receives their number. first: also adds the flagged pairs to
// kStatUnion. tile_roots: scratch of T entries (the root range of each tile).
cudaError_t select_round(const PassArgs& a, int64_t T, int2* tile_roots, int64_t n, int lo, int hi, bool filter,
                         bool first, int2* out, unsigned long long* count, cudaStream_t s);

// --- single-linkage forest (k_mst.cu)
// Edges of the minimum spanning forests of the eps-graphs of all elements:
// points u < v, element, the two cover slots (su < sv) and the FP64 d2; n
// edges (capacity M), sorted by (element, d2, u, v).
struct ForestOut {
    Buf u, v, elem, su, sv, d2;
    int64_t n = 0;
};
// a: the rows of a tile layout (G or X via row_pt, dp, d, tile_n, row_pt,
// eps2, hi_thr of fp32_thresholds) and a.pairs[0 .. n_pairs) the element tile
// pairs not certified all-out at eps. queue_bytes: the most that the queue of
// candidate pairs may take (0: no limit). Returns a mapper_status.
int msf_forest(const PassArgs& a, const int32_t* row_slot, const int32_t* slot_point, const int32_t* slot_elem,
               int64_t M, int64_t E, int64_t R, int64_t T, int64_t n_pairs, size_t queue_bytes, ForestOut* out,
               cudaStream_t s);
// Single-linkage clusters at height h (edges with d2 <= h^2) in cover-slot
// space, in the layout of rows_to_slots (every slot a member and core).
int msf_cut(const ForestOut& f, const int32_t* slot_point, int64_t M, double h, int32_t* lab, uint8_t* flags,
            int64_t* slot_label, uint8_t* core, cudaStream_t s);

// --- nodes and nerve (k_nerve.cu)
// Nerve keys (point << 32 | node) of the members of nodes given by offsets.
cudaError_t node_member_keys(const int64_t* node_off, int64_t N, int64_t G, const int32_t* members,
                             uint64_t* keys2, cudaStream_t s);
// slot_elem[i] = the element e with elem_off[e] <= i < elem_off[e + 1].
cudaError_t fill_slot_elem(const int64_t* elem_off, int32_t k, int64_t M, int32_t* slot_elem, cudaStream_t s);
// pos: the scan of the slots' flags. keys: (node << 32 | point) of the member
// slots; node_elem; node_o (if set): the node of every membership in point order
// (slot_o of split_keys), -1 for none.
cudaError_t member_keys(const int32_t* lab, const int64_t* pos, const int32_t* slot_point, const int32_t* slot_elem,
                        const int32_t* slot_o, int64_t M, uint64_t* keys, int32_t* node_elem, int32_t* node_o,
                        cudaStream_t s);
cudaError_t node_offsets(const uint64_t* keys, int64_t G, int64_t N, int64_t* node_off, int32_t* members,
                         uint64_t* keys2, cudaStream_t s);
// From the points pt (ascending) and nodes node_o of M memberships in point order:
// the distinct node pairs (v << 32 | u) sharing a point, unsorted, into *list (at
// most cap <= kEdgeListMax); counts[0]: their number, counts[1]: nonzero if the list
// does not hold them all.
// kEdgeListMax: what one cluster launch sorts in 4 rounds, with a set of four slots
// an entry (1 MB, cleared on each call). Nerves with the list and with the sort of
// all pairs: 3k edges 97 and 193 us, 13k 120 and 228, 30k 129 and 260, 7k edges of
// points in 30 elements each 216 and 977; with more edges than it holds, and so
// both, 40k 292 and 280, 101k 432 and 429. A list of 2^17 took 110, 173, 207 and
// 163 us for the first four and 207 and 267 for the last two.
constexpr uint32_t kEdgeListMax = 1u << 15;
cudaError_t edge_set(const int32_t* pt, int64_t M, const int32_t* node_o, int64_t cap, Buf* list,
                     unsigned long long* counts, cudaStream_t s);
cudaError_t run_pairs(const uint64_t* keys2, int64_t G, int64_t* cnt, cudaStream_t s);
cudaError_t emit_pairs(const uint64_t* keys2, int64_t G, const int64_t* pos, uint64_t* out,
                       cudaStream_t s);
cudaError_t unique_flags(const uint64_t* k, int64_t P, int32_t* flag, cudaStream_t s);
cudaError_t unique_emit(const uint64_t* k, const int32_t* flag, const int64_t* pos, int64_t P,
                        int32_t* edges, cudaStream_t s);

// --- tile layout (k_tiles.cu)
struct TileLayout {
    int64_t R = 0;               // rows (multiple of kTile)
    int64_t T = 0;               // tiles
    int64_t n_seg = 0;           // (element, group) segments
    int n_groups = 0;            // pivot groups (outliers form group n_groups)
    Buf row_slot;                // [R] int32 cover slot, -1 for padding
    Buf row_pt;                  // [R] int32 point, INT32_MAX for padding
    Buf G;                       // [R x dp] FP32 rows (unset on the tensor-core path for dp <= 256)
    Buf tile_n, tile_seg, tile_elem;      // [T] int32
    Buf tile_cent;               // [T x dp] FP32 centre
    Buf tile_rad;                // [T] FP64 upper bound of the rows' distance to it
    Buf seg_cent;                // [n_seg x dp] FP32 centre of each segment
    Buf seg_outlier;             // [n_seg] int32: 1 if the segment holds outliers
    Buf seg_elem;                // [n_seg] int32 element of each segment
    Buf seg_toff;                // [n_seg + 1] int64 first tile of each segment
    Buf eseg_off;                // [E + 1] int64 first segment of each element
    Buf blk_off;                 // [n_seg + 1] int64 blocks of tiles before each segment (classification)
    int64_t n_cand = 0;          // tile pairs of all elements
    Buf seg_rad;                 // [n_seg] FP64 upper bound of its rows' distance to its centre
    Buf Ah, Al;                  // [R x dp] BF16 centred rows (hi and lo parts)
    Buf rn2, rn;                 // [R] FP32 |a|^2 and |a| (rounded up)
    Buf rl;                      // [R] FP32 |a - hi| (rounded up): the residual of the hi part
    Buf tmax;                    // [T] float4: largest |a|^2, |a|, |a - hi| of each tile's rows
    Buf tn2min;                  // [T] smallest |a|^2 of each tile's valid rows
    Buf Fh, Fl;                  // [R x dp] FP8 E4M3 parts of a / s (s: the tile's scale), if built
    Buf frl;                     // [R] |a - s hi| (FP8 hi part), rounded up
    Buf ftmax;                   // [T] float4: largest |a|^2, |a|, frl of each tile, and its scale s
};

struct PairLists {
    Buf list[kListCount];        // int2 tile pairs
    int64_t n[kListCount] = {0, 0, 0};
    int64_t n_candidates = 0, n_out = 0;
};

// The pivots of the tile layout and every point's nearest one: K pivots
// (points floor(k n / K)), Pv their FP32 rows (K x dp), piv[n] the nearest
// pivot and pd2[n] an FP32 squared distance to it. They depend on X only, so
// one set serves every layout of the cloud.
struct PivotSet {
    int K = 0;
    Buf Pv, piv, pd2;
    Buf err;                     // int: set if the tensor-core assignment gave up waiting (read by build_tiles)
    // set by pivot_prepare: the pivots' centre c and the points' split for
    // the tensor-core assignment (written by the lens pass, lens_l2_split)
    bool split = false;
    Buf c, xh, xn2;
};
// Allocates the set on stream `alloc_s` (where it is later freed) and
// computes it on stream `s` (which must wait for alloc_s).
cudaError_t pivot_alloc(int64_t n, int dp, PivotSet* P, cudaStream_t alloc_s);
int pivot_assign(const float* X, int64_t n, int32_t d, int64_t ld, int dp, bool bf16, int num_sms, PivotSet* P,
                 cudaStream_t s);
// Before the lens pass (P from pivot_alloc): the pivot rows (X's rows
// k n / K; X in host memory when `host`), their FP32 centre c, and room for the
// points' BF16 split (rows past n zeroed), which lens_l2_split then writes;
// pivot_assign afterwards skips its own split. A mapper_status.
int pivot_prepare(const float* X, int64_t n, int32_t d, int64_t ld, int dp, bool host, PivotSet* P, cudaStream_t s);

// Orders every element's points by pivot group, lays them out in tiles
// (a tile never mixes groups) and gathers rows. tau: distance under which two
// pivots join a group and beyond which a point is an outlier. bf16: also
// build the tensor-core operands (and assign pivots on tensor cores).
// pre: the pivot set, computed beforehand (stream-ordered before s), or null.
int build_tiles(const float* X, int64_t n, int32_t d, int64_t ld, int dp, const int32_t* slot_point,
                const int32_t* slot_elem, int64_t M, int64_t E, double tau, bool bf16, int num_sms,
                TileLayout* L, int* nonfinite, cudaStream_t s, const PivotSet* pre = nullptr);
// Classifies every tile pair of every element by bounding spheres: out (no
// pair within eps), all-in, or mixed (to the tensor-core list when both tiles
// are one non-outlier segment and use_tc, else to the CUDA-core list).
// X, ld, d: the rows (read for the outlier tiles' distance bounds when G is
// not gathered). eps_all_in (if > 0, <= eps): the radius a pair must be all in
// at to go to the all-in list (the smallest of several radii sharing the
// lists; out stays decided at eps, the largest).
int classify_pairs(const TileLayout& L, const float* X, int64_t ld, int d, int dp, int64_t E, double eps,
                   bool use_tc, PairLists* P, cudaStream_t s, double eps_all_in = 0.0);
// Count-pass phase choice per tile pair: bin[q] (< kPairBins) of the pair's
// statistic (|c_a - c_b|^2 + r_a^2 + r_b^2) / eps^2 from the layout's tile
// spheres, on a log2 scale of 8 bins per octave from 2^-4.
constexpr int kPairBins = 64;
cudaError_t pair_bins(const TileLayout& L, const int2* pairs, int64_t n, int dp, double eps, uint8_t* bin,
                      cudaStream_t s);
// Tally of sampled pairs (mask[j] pair j's first phase's deferred blocks, bin[j]
// its bin): cnt[2 b] sampled pairs of bin b, cnt[2 b + 1] of them that deferred a
// block (2 kPairBins counters, zeroed here).
cudaError_t sample_bins(const uint32_t* mask, int64_t n_s, const uint8_t* bin, unsigned long long* cnt,
                        cudaStream_t s);
// Stable partition of pairs[0 .. n): those whose bin is chosen (chosen: kPairBins
// bytes on the device) first, then the rest, into out; *pos receives [n + 1]
// int64 with their number at pos[n].
cudaError_t partition_pairs(const int2* pairs, const uint8_t* bin, const uint8_t* chosen, int64_t n, int2* out,
                            Buf* pos, cudaStream_t s);
// FP8 E4M3 operands of a tile layout built with BF16 operands (needs its
// centres and tmax): per tile a power-of-two scale s, hi and lo parts of a / s
// (Fh, Fl), frl and ftmax. A no-op when already built. Returns a mapper_status.
int fp8_operands(TileLayout* L, const float* X, int64_t ld, int d, int dp, cudaStream_t s);
// BF16 hi + lo operands of rows row_pt[.] of X (T tiles of 128 rows, the
// first tile_n[t] of tile t valid, the rest zero), centred on cents[tile_cent[t]]
// (dp floats each), with FP32 |a|^2 and |a| rounded up. nonfinite (nullable):
// set to 1 when a valid row's |a|^2 is not finite (a NaN or Inf in the row, or
// a norm beyond FP32).
cudaError_t centred_operands(const float* X, int64_t ld, int d, int dp, const int32_t* row_pt, const int32_t* tile_n,
                             const int32_t* tile_cent, const float* cents, int64_t T, void* Ah, void* Al, float* rn2,
                             float* rn, cudaStream_t s, int* nonfinite = nullptr);
// Tensor-core operands for the CUDA-core list (tile pairs of one element, two
// segments): every row centred on its element's centre, BF16 hi + lo, with
// FP32 |a|^2, and |a| and |a - hi| rounded up (R rows each), their largest
// values per tile (T float4) and the smallest |a|^2 per tile.
int cross_operands(const TileLayout& L, const float* X, int64_t ld, int d, int dp, int64_t E, Buf* Ah, Buf* Al,
                   Buf* rn2, Buf* rn, Buf* rl, Buf* tmax, Buf* tn2min, cudaStream_t s);

}  // namespace mgb
