// Internal declarations shared by the library's translation units.
// Nothing here is part of the public ABI (include/akashic_mem.h is).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/akashic_mem.h"
#include "ak_sizes.h"

namespace ak {

// ------------------------------------------------------------------ status word
// Device-side faults are recorded with atomicCAS(status, 0, code) so that the
// first one wins; the host reads and clears the word in akashic_mem_sync.
__device__ __forceinline__ void set_status(int *status, int code) {
    if (status) atomicCAS(status, 0, code);
}

// ------------------------------------------------------------------ dependent launches
// The kernels of a retrieval and of the graph's and the pages' upkeep are
// launched with programmatic stream serialisation (launch_pdl): each may be
// scheduled while the kernel before it in the stream drains, and waits here,
// before it touches global memory, until that kernel has completed and its
// writes are visible (a kernel launched without the attribute returns from the
// wait at once).  Every thread waits before anything else, so that a kernel's
// end says that all before it have ended.  An upkeep call is a chain of 10 to 45
// short kernels: 40 chunks added to 262,144 712 -> 640 us, 200 deleted from
// 524,288 575 -> 547.
__device__ __forceinline__ void griddep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// ------------------------------------------------------------------ ordered tiles
// Ordered compaction in two passes: the first tests the items and counts every
// tile's survivors, in the second a CTA a tile adds up the counts before its
// own and writes.  (One pass in which a tile waits for the totals before it
// was slower wherever all tiles start together, as the wait runs through them
// 32 at a time: a deletion's 16.8M edges 114 us against 88, a directory of
// 1,048,576 chunks 25 against 13.)
// The sum of counts[first .. tile), on every thread; 256 threads, a grid of one CTA
// a tile.  Past TILE_FLAT tiles, where every CTA's reading of all counts before its
// own would grow with their square, the sums of 1024 tiles each stand behind the
// counts (launch_tile_groups between the passes) and a CTA reads those before its
// group and the counts within it (200 chunks deleted from 128M edges, 31,250 tiles:
// 2.73 -> 2.59 ms, from 256M 7.9 -> 7.3).  TILE_FLAT: up to there (a deletion's 16.8M
// edges) the flat sum costs no launch.
constexpr int TILE_GROUP = 1024;
constexpr int64_t TILE_FLAT = 4096;
// Words of counts for so many tiles, and the sums of their groups.
__host__ __device__ __forceinline__ int64_t tile_words(int64_t tiles) {
    return tiles + (tiles > TILE_FLAT ? (tiles + TILE_GROUP - 1) / TILE_GROUP : 0);
}
cudaError_t launch_tile_groups(int32_t *counts, int64_t tiles, cudaStream_t st,
                               int *launches = nullptr);
__device__ __forceinline__ int64_t tile_base(const int32_t *__restrict__ counts, int64_t first,
                                             int64_t tile) {
    __shared__ int64_t part[8];
    int64_t s = 0, g0 = (first + TILE_GROUP - 1) / TILE_GROUP, g1 = tile / TILE_GROUP;
    if ((int64_t)gridDim.x > TILE_FLAT && g0 < g1) {
        const int32_t *groups = counts + gridDim.x;
        for (int64_t i = first + threadIdx.x; i < g0 * TILE_GROUP; i += 256) s += counts[i];
        for (int64_t g = g0 + threadIdx.x; g < g1; g += 256) s += groups[g];
        first = g1 * TILE_GROUP;
    }
    for (int64_t i = first + threadIdx.x; i < tile; i += 256) s += counts[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    s = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += part[w];
    return s;
}
// A tile of 1024 items, 256 threads, item q * 256 + thread survives where bit
// `lane` of bal[q] is set (the warp's ballot): places[q] = the item's place among
// the tile's survivors; returns their number.
__device__ __forceinline__ int tile_places(const unsigned (&bal)[4], int (&places)[4]) {
    __shared__ int wcnt[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) wcnt[q * 8 + warp] = __popc(bal[q]);
    __syncthreads();
    const int c = wcnt[lane];
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    const int excl = incl - c, total = __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
    for (int q = 0; q < 4; ++q)
        places[q] = __shfl_sync(0xffffffffu, excl, q * 8 + warp) +
                    __popc(bal[q] & ((1u << lane) - 1u));
    return total;
}

// ------------------------------------------------------------------ small helpers
__device__ __forceinline__ float bf16_to_f32(uint16_t h) {
    return __uint_as_float(((uint32_t)h) << 16);
}

template <typename T>
__host__ __device__ __forceinline__ T ceil_div(T a, T b) { return (a + b - 1) / b; }

// Selection key: larger key = better.  High word: the score's fp32 bit
// pattern (scores are >= 0, where the bit pattern is monotone in value);
// low word: ~id, so that on equal scores the lower chunk ID wins.
__device__ __forceinline__ unsigned long long make_key(float score, uint32_t id) {
    return ((unsigned long long)__float_as_uint(score) << 32) | (unsigned long long)(~id);
}
__device__ __forceinline__ float key_score(unsigned long long key) {
    return __uint_as_float((uint32_t)(key >> 32));
}
__device__ __forceinline__ uint32_t key_id(unsigned long long key) {
    return ~(uint32_t)(key & 0xffffffffull);
}

// Candidate scope of a selection.  Namespaces (§4.1: the candidates of a
// query are the chunks of the caller's (user_id, session_id) table): row j
// is a candidate for query column c only if ns_row[j] == q_ns[c]
// (q_ns == NULL: no namespace scope).  Deletions (tombstones): a row with
// dead[j] != 0 is never a candidate (dead == NULL: none deleted).
struct NsScope {
    const int32_t *ns_row;   // [rows] tag of the chunk in each row (or sample row)
    const int32_t *q_ns;     // [bp] tag of each query column
    const int32_t *dead;     // [rows] 1 where the chunk was deleted
};
__device__ __forceinline__ bool in_scope(const NsScope &s, int64_t row, int col) {
    return (!s.dead || !s.dead[row]) && (!s.q_ns || s.ns_row[row] == s.q_ns[col]);
}
__host__ __device__ __forceinline__ bool scope_active(const NsScope &s) {
    return s.q_ns != nullptr || s.dead != nullptr;
}

// Split-bf16 of two fp32 values: hi = bf16(x) (round to nearest), lo =
// bf16(x - hi) (x - hi is exact in fp32), packed two to a word (x in the low
// half); x = hi + lo to within 2^-17 relative.
__device__ __forceinline__ uint32_t split_bf16_pair(float x, float y, uint32_t &lo) {
    const __nv_bfloat16 hx = __float2bfloat16_rn(x), hy = __float2bfloat16_rn(y);
    const __nv_bfloat16 lx = __float2bfloat16_rn(x - __bfloat162float(hx));   // exact rest
    const __nv_bfloat16 ly = __float2bfloat16_rn(y - __bfloat162float(hy));
    lo = (uint32_t)__bfloat16_as_ushort(lx) | ((uint32_t)__bfloat16_as_ushort(ly) << 16);
    return (uint32_t)__bfloat16_as_ushort(hx) | ((uint32_t)__bfloat16_as_ushort(hy) << 16);
}

// log2(e): scores exp(tau x - c) are evaluated as 2^(x tau log2(e) - c log2(e))
// (one FMA and the hardware exp2).
constexpr float LOG2E_F = 1.44269504088896340736f;

// Keys for signed cosine values: order-preserving map of any finite fp32 to
// uint32 (flip all bits of negatives, set the sign bit of non-negatives).
__device__ __forceinline__ uint32_t ordered_bits(float v) {
    uint32_t u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered_bits(uint32_t o) {
    uint32_t u = (o & 0x80000000u) ? (o & 0x7fffffffu) : ~o;
    return __uint_as_float(u);
}

// Set the thread-local message returned by akashic_mem_last_error().
void set_last_error(const char *msg);

// ------------------------------------------------------------------ launchers
// All launchers enqueue on `st` and report launch errors by return value.

// Score (a1) on the tensor cores: u[j, c] = exp(tau * <e_j, q_c> - shift[c])
// for j < n, c < bp (bp = 32, 64, 128 or 256), written chunk-major with row
// stride bp; zpart[r, c] = sum of u over the rows handled by score CTA r,
// for r < *zrows.  score_tiles(n) bounds *zrows.
int64_t score_tiles(int64_t n);
// dead_row (or NULL): rows of deleted chunks score u = 0 (no part in Z).
// row_max / row_min (optional, together): [n] the largest and smallest u of
// each row over the first n_real columns (the real queries), for the
// propagation's row bounds; with them, ext (optional, [2], zeroed before)
// gets their extremes (RowBounds::ext).
// One thread waits on a barrier that nothing signals, giving up after
// `polls` polls like every bounded wait (ETIMEOUT into *status).
cudaError_t launch_wait_timeout_check(int *status, uint32_t polls, cudaStream_t st);
// Raises the score kernel's shared-memory limit for every query width on the
// current device now (launch_score does it lazily per width otherwise).
cudaError_t prepare_score_gemm();
cudaError_t launch_score(const uint16_t *emb, int64_t n, int dim, const uint16_t *qp, int bp,
                         const float *shift, float tau, float *u, float *zpart, int *status,
                         cudaStream_t st, int *launches, int *zrows,
                         const int32_t *dead_row = nullptr, float *row_max = nullptr,
                         float *row_min = nullptr, int n_real = 0, unsigned int *ext = nullptr,
                         const int32_t *done = nullptr);
// The largest shift c of a batch's columns, and a value that no score of the
// batch is below: exp(-2 c) (z >= -c in every column).  The same bits wherever a
// whole warp calls them.
__device__ __forceinline__ float batch_shift(const float *__restrict__ shift, int bp) {
    float c = 0.f;
    for (int i = threadIdx.x & 31; i < bp; i += 32) c = fmaxf(c, shift[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c = fmaxf(c, __shfl_xor_sync(0xffffffffu, c, o));
    return c;
}
__device__ __forceinline__ float batch_u_min(const float *__restrict__ shift, int bp) {
    return exp2f(-2.f * batch_shift(shift, bp) * LOG2E_F);
}
// The same scores with u - batch_u_min(shift) written as split bf16 instead of
// u in fp32: u_hi and u_lo [n][bp] each, their sum within 2^-17 relative (the
// operand form the candidates' tensor-core pass reads); Z's column sums from
// the fp32 values of u.
cudaError_t launch_score_split(const uint16_t *emb, int64_t n, int dim, const uint16_t *qp, int bp,
                               const float *shift, float tau, uint16_t *u_hi, uint16_t *u_lo,
                               float *zpart, int *status, cudaStream_t st, int *launches,
                               int *zrows, const int32_t *dead_row, float *row_max,
                               float *row_min, int n_real, unsigned int *ext,
                               const int32_t *done);

// The score on every stride-th row only: out[v, c] = u[v*stride, c] for
// v < n_sample (same kernel and arithmetic as launch_score, so the values
// are those the full pass computes); zpart receives partial sums of the
// sample (scratch, one row per CTA, at most score_tiles(n_sample) rows).
cudaError_t launch_score_sample(const uint16_t *emb, int64_t n_sample, int64_t stride, int dim,
                                const uint16_t *qp, int bp, const float *shift, float tau,
                                float *out, float *zpart, int *status, cudaStream_t st,
                                int *launches);
// Score with the top-k filter fused and no slab written: zpart as in
// launch_score; the key (u bits, chunk ID ext_of[j]) of every (j, c) with
// c < n_cols that is >= bound[c] is appended to buf[c][...] (count cnt[c],
// capacity cap).
cudaError_t launch_score_filter(const uint16_t *emb, int64_t n, int dim, const uint16_t *qp,
                                int bp, int64_t n_cols, const float *shift, float tau,
                                float *zpart, const int32_t *ext_of,
                                const unsigned long long *bound, unsigned int *cnt,
                                unsigned long long *buf, int64_t cap, NsScope ns, int *status,
                                cudaStream_t st, int *launches, int *zrows);

// Plain dot products out[j, c] = <e_{j*row_stride}, q_c> (bf16 tensor
// cores, fp32 accumulate) for j < n and the n_ctiles * bp columns of qp;
// row stride n_ctiles * bp in out.
cudaError_t launch_dots(const uint16_t *emb, int64_t n, int64_t row_stride_rows, int dim,
                        const uint16_t *qp, int bp, int n_ctiles, float *out, int *status,
                        cudaStream_t st, int *launches);
// Fused relation top-M filter: dots of every row j < n against the
// n_ctiles*256 rows of qp; the selection key (signed dot, chunk ID
// ext_of[j]) of every (j, c) with c < n_cols and ext_of[j] < id_limit that
// is >= bound[c] is appended to buf[c][...] (count cnt[c], capacity cap).
cudaError_t launch_dots_filter(const uint16_t *emb, int64_t n, int dim, const uint16_t *qp,
                               int n_ctiles, int64_t n_cols, const int32_t *ext_of,
                               int64_t id_limit, const unsigned long long *bound,
                               unsigned int *cnt, unsigned long long *buf, int64_t cap,
                               int *status, cudaStream_t st, int *launches,
                               const int32_t *dead_row = nullptr);

// Sampled dots as selection keys, column-major: keys_t[c][j] for the rows
// j < n (row j*row_stride of emb) and the n_ctiles*256 rows c of qp; the
// key is the order-preserving bits of the signed dot, or 0 where row j is
// deleted (dead_row[j], if given) or ext_of[j] >= id_limit.
cudaError_t launch_dots_keys_t(const uint16_t *emb, int64_t n, int64_t row_stride_rows, int dim,
                               const uint16_t *qp, int n_ctiles, const int32_t *ext_of,
                               int64_t id_limit, const int32_t *dead_row, uint32_t *keys_t,
                               int *status, cudaStream_t st, int *launches);

// Query preparation: pad q (b rows) to bp rows of zeros and compute
// shift[c] = tau * |q_c| * max_norm (0 for padding); flags ERANGE.
// zero (or NULL): n_zero words set to 0 (the call's counters), but zero[skip_at]
// (where tried is given) to 1 if the mark *tried says to skip call `now`.
cudaError_t launch_prep_queries(const uint16_t *q, int b, int bp, int dim, float tau,
                                const float *max_norm, uint16_t *qp, float *shift, int *status,
                                cudaStream_t st, unsigned int *zero = nullptr,
                                int n_zero = 0, int skip_at = 0,
                                const unsigned long long *tried = nullptr,
                                unsigned long long now = 0);
// When calls on a stream try the candidates.  The calls with one key (graph,
// alpha, hops, k) since it last changed are numbered; a mark is (key's number <<
// 32 | call's number).  Where the candidates do not suffice for a call, the
// device leaves the mark of the next call to try them, TRY_AGAIN calls later, and
// those before it run the hops alone.  So what a call does follows from the calls
// before it and never from when they end.  The host reads the mark too, as it
// stands, to spare the launches that a skipping call's kernels would return from.
constexpr unsigned int TRY_AGAIN = 16;
__host__ __device__ __forceinline__ bool try_skips(unsigned long long tried,
                                                   unsigned long long now) {
    return (tried >> 32) == (now >> 32) && tried > now;
}

// Running maximum of row norms of emb[0..n) into *max_norm (monotone).
cudaError_t launch_row_norm_max(const uint16_t *emb, int64_t n, int dim, float *max_norm,
                                cudaStream_t st);

// ------------------------------------------------------------------ graph
int device_sm_count();

// Propagation work plan.  Rows with more than SPLIT_T in-edges (the hubs of
// a power-law relation graph) are cut into segments of at most SEG_LEN
// edges that never cross a source window of WIN_ROWS rows; segments are
// processed window by window so that the source rows they gather stay in L2,
// and a fixup pass sums each hub's segment partials in order.
struct SplitParams {
    int64_t split_t = 256;      // in-degree above which a row is split
    int64_t seg_len = 512;      // edges per segment at most
    int64_t win_rows = 32768;   // source window (rows); 32 MB of slab at 256 queries
};
constexpr int ROWS_PER_GRAB = 8;     // rows a warp claims at a time (dynamic scheduling)

// Exclusive prefix sum of `in` (n values) into out (n+1 values; out[n] = total).
// `launches`, if given, is incremented by the kernels launched.
cudaError_t scan_exclusive(const int64_t *in, int64_t *out, int64_t n, void *tmp,
                           size_t tmp_bytes, cudaStream_t st, int *launches = nullptr);

// Stable LSD radix sort of (key, value) pairs on the low `bits` key bits;
// the result lands in (keys, vals) or, if *result_in_alt, in the alt buffers.
// tmp: radix_tmp_bytes(n) bytes (ak_sizes.h).
cudaError_t radix_sort_pairs(uint32_t *keys, uint32_t *vals, uint32_t *keys_alt,
                             uint32_t *vals_alt, int64_t n, int bits, void *tmp,
                             size_t tmp_bytes, cudaStream_t st, bool *result_in_alt,
                             int *launches = nullptr);

// CSR helpers (see ak_graph.cu).
cudaError_t launch_edge_src_check(const int64_t *row_ptr, const int32_t *col, int64_t n_rows,
                                  int64_t row_base, int64_t n_total, int32_t *src, int *status,
                                  cudaStream_t st);
// w = row softmax of the logits, per row: w_e = exp(aff_e - max) * inv with
// inv = 1 / sum exp(aff - max); (max, inv) of row r go to rstat[r] when
// rstat is not NULL, so that any copy of a weight (the in-edge transpose)
// can be recomputed bit for bit by row_softmax_weight.
__device__ __forceinline__ float row_softmax_weight(float aff, float2 stat) {
    return expf(aff - stat.x) * stat.y;
}
cudaError_t launch_row_softmax(const int64_t *row_ptr, const float *aff, float *w, int64_t n_rows,
                               float2 *rstat, cudaStream_t st);
// How many of the sorted keys[0 .. count) are below v.
__device__ __forceinline__ int64_t lower_bound_u32(const uint32_t *__restrict__ keys, int64_t count,
                                                   uint64_t v) {
    int64_t lo = 0, hi = count;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((uint64_t)keys[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}
// Pairs p (M a new chunk) as sort items: key map ? map[ids[p]] : ids[p], value p;
// in their own order or (order) in that of the new chunks order[0], order[1], ...
cudaError_t launch_pair_keys(const int32_t *ids, const int32_t *map, const uint32_t *order, int M,
                             int64_t pairs, uint32_t *keys, uint32_t *vals, cudaStream_t st);
// The store keeps chunks in HBM in page order: row r holds chunk ext_of[r],
// chunk c lives in row row_of[c].  The out-edge CSR stays in chunk IDs; the
// in-edge transpose used by propagation is in rows.
cudaError_t launch_in_degree(const int32_t *col, const int32_t *row_of, int64_t nnz, int64_t *deg,
                             cudaStream_t st);
cudaError_t launch_iota(uint32_t *v, int64_t n, cudaStream_t st);
// out[row_of[first + i]] = in[i], i < n.
cudaError_t launch_scatter_by_row(const int32_t *in, const int32_t *row_of, int64_t first,
                                  int64_t n, int32_t *out, cudaStream_t st);
cudaError_t launch_map_keys(const uint32_t *sel, const int32_t *ids, const int32_t *row_of,
                            uint32_t *keys, int64_t n, cudaStream_t st);
cudaError_t launch_gather_in(const uint32_t *order, const int32_t *src, const int32_t *row_of,
                             const float *w, const float *aff, int32_t *in_src, float *in_w,
                             float *in_aff, int64_t nnz, cudaStream_t st);

// Incremental in-edge transpose after a relation update (ak_inedges.cu).
struct InEdgeUpdate {
    int64_t n;                          // store rows (new chunks included)
    int64_t nnz_new;                    // edges after the update
    const int64_t *in_ptr_old;          // [n+1]
    const int32_t *in_src_old;
    const float *in_aff_old, *in_w_old;
    int64_t *in_ptr_new;                // [n+1]
    int32_t *in_src_new;                // [nnz_new]
    float *in_aff_new, *in_w_new;       // [nnz_new]
    const int32_t *nbr_ids;             // [n_new][M] chosen prior chunk IDs
    const float *nbr_cos;               // [n_new][M]
    float scale;                        // logit = scale * cos
    int64_t first, n_new;
    int M;
    bool reciprocal;
    int row_bits;                       // key bits of a row index
    const int32_t *row_of, *ext_of;
    const float2 *rstat;                // per chunk ID: (max, inv) of its out-row
    const uint32_t *touched;            // bits of the rows whose out-edges changed
};
// The update writes in_w_new for every edge as it places it: the old weight, or
// row_softmax_weight(aff, rstat[ext_of[src]]) for new edges and touched sources.
struct InEdgeScratch {
    uint32_t *keys, *vals, *keys2, *vals2;   // [n_new * M] each
    uint32_t *rows;                     // [4 * n_new]
    uint32_t *move;                     // [move_words(old edges, n_new * M, n_new)]
    void *tmp;
    size_t tmp_bytes;                   // >= radix needs
};
// An edge list moved to make room (ak_inedges.cu): `pairs` edges are inserted, one
// at the end of each row sorted[p] (ascending), and blocks of mult2 edges in the
// empty rows rows2[] (ascending); ptr: the old row starts.
struct MoveEdges {
    int64_t nnz;                        // old edges
    const int32_t *tgt;
    const float *val, *w;               // logits, weights
    int32_t *tgt_out;
    float *val_out, *w_out;
    int64_t mult2;
    const uint32_t *touched;            // or NULL: bit of an edge's tgt set: its weight is
    const int32_t *ext_of;              // row_softmax_weight(val, rstat[ext_of[tgt]])
    const float2 *rstat;
};
int64_t move_words(int64_t nnz, int64_t pairs, int64_t n_rows2);
cudaError_t launch_move_edges(const MoveEdges &m, const int64_t *ptr, const uint32_t *sorted,
                              int64_t pairs, const uint32_t *rows2, int64_t n_rows2,
                              uint32_t *words, cudaStream_t st, int *launches);
cudaError_t launch_in_edges_update(const InEdgeUpdate &u, const InEdgeScratch &s, cudaStream_t st,
                                   int *launches);
cudaError_t launch_batch_layout(const uint32_t *order, int64_t first, int64_t n, int dim,
                                const uint16_t *emb_in, uint16_t *emb, const int32_t *page_in,
                                int64_t first_page, int per_page, int32_t *page_row,
                                int32_t *ext_of, int32_t *row_of, cudaStream_t st);
// Hub plan (see SplitParams), first its sizes: rows = the hub rows in row order
// (at most max_hubs), counts[0] = their number, slot0 = their first partial
// slots, slot0[max_hubs] the number of segments.  scratch:
// hub_plan_words(n, max_hubs) words.
int64_t hub_plan_words(int64_t n, int64_t max_hubs);
cudaError_t launch_hub_count(const SplitParams &sp, const int64_t *in_ptr, const int32_t *in_src,
                             int64_t n, int64_t max_hubs, int32_t *rows, int64_t *slot0,
                             int64_t *counts, int64_t *scratch, cudaStream_t st);
// Then the plan: the split rows and their slots, the segments (by row, then
// window) with their window as sort key and their index as value, the split row
// that owns each slot, and sort keys / values that order the split rows by
// segment count, largest first, ties in row order.
cudaError_t launch_hub_fill(const SplitParams &sp, const int64_t *in_ptr, const int32_t *in_src,
                            const int32_t *rows, const int64_t *slot0, int64_t n_rows,
                            int64_t n_segs, int32_t *split_row, int64_t *split_slot0,
                            int64_t *seg_e0, int64_t *seg_e1, uint32_t *seg_win, uint32_t *seg_id,
                            int32_t *slot_split, uint32_t *row_key, uint32_t *row_id,
                            cudaStream_t st);
// Permute segments into window-major order: dst[i] = src[order[i]], slot[i] = order[i].
cudaError_t launch_seg_permute(const uint32_t *order, const int64_t *e0, const int64_t *e1,
                               int64_t n_segs, int64_t *e0s, int64_t *e1s, int32_t *slot,
                               cudaStream_t st);

// Memory Manager tables (ak_mm.cu): the page directory's slot counters,
// the co-retrieval statistics and the running counters.
struct MmTables {
    int32_t *page_total, *page_live;   // [page capacity] slots used / live chunks per page
    int32_t *sel;                      // [chunk capacity] requests that retrieved the chunk
    unsigned long long *co_key;        // [co_cap] chunk pair (lo << 32 | hi), ~0 = empty
    uint32_t *co_val;                  // [co_cap] requests that retrieved both
    int64_t co_cap;                    // power of two
    unsigned long long *pairs;         // pairs in the table
    unsigned long long *released;      // the last compaction's pages, [1] its moving chunks
};
cudaError_t launch_mm_count(const int64_t *S, int n_req, int s_len, int64_t n,
                            const int32_t *row_of, const int32_t *dead_row, const MmTables &t,
                            int *status, cudaStream_t st);
// g_buf [n_req][64], g_n [n_req] scratch; result [4] (device): the next fresh
// page, the chunks written, the pairs in the table, the status word.
cudaError_t launch_mm_relocate(const int64_t *S, int n_req, int s_len, int64_t n,
                               const int32_t *row_of, const int32_t *dead_row, int32_t *page_row,
                               const MmTables &t, float tau, int64_t next_page, int per_page,
                               int32_t *g_buf, int32_t *g_n, const int *status, int64_t *result,
                               cudaStream_t st);
// cand[p] = 1 for the pages to compact, released[0] = their number.
cudaError_t launch_mm_candidates(const MmTables &t, int64_t n_pages, float theta, int32_t *cand,
                                 cudaStream_t st);
// The live chunks on candidate pages, in ID order: ids and their namespaces'
// order-preserving keys, released[1] = their number, a bitmap of them
// ((n + 31) / 32 words), parent[c] = c.  counts: mm_words(n) words.
int64_t mm_words(int64_t n);
cudaError_t launch_mm_collect(const MmTables &t, int64_t n, const int32_t *row_of,
                              const int32_t *dead_row, const int32_t *page_row,
                              const int32_t *ns_row, const int32_t *cand, uint32_t *moving,
                              int32_t *parent, uint32_t *ids, uint32_t *ns_key,
                              int32_t *counts, cudaStream_t st);
cudaError_t launch_mm_union(const MmTables &t, const uint32_t *moving, const int32_t *row_of,
                            const int32_t *ns_row, float tau, int32_t *parent, int *status,
                            cudaStream_t st);
cudaError_t launch_mm_roots(const uint32_t *ids, int64_t count, const int32_t *parent,
                            uint32_t *root_key, cudaStream_t st);
// At most mm_small_repack() moving chunks: candidate pages released, the chunks
// ordered and written into fresh pages from first_page on, new_pages (device) =
// how many.
int mm_small_repack();
cudaError_t launch_mm_repack_small(const MmTables &t, int64_t n_pages, const int32_t *cand,
                                   const uint32_t *ids, const uint32_t *ns_key, int64_t count,
                                   const int32_t *parent, const int32_t *row_of,
                                   int32_t *page_row, int64_t first_page, int per_page,
                                   int64_t *new_pages, cudaStream_t st);
// part_pages[i] = pages the namespace run starting at i fills (0 inside a run)
cudaError_t launch_mm_part_pages(const uint32_t *ns_sorted, int64_t count, int per_page,
                                 int64_t *part_pages, cudaStream_t st);
// releases the candidate pages, then writes the ordered chunks into fresh
// pages from first_page on, each namespace from its own base page
cudaError_t launch_mm_release_repack(const MmTables &t, int64_t n_pages, const int32_t *cand,
                                     const uint32_t *order_ids, const uint32_t *ns_sorted,
                                     const int64_t *part_base, int64_t count,
                                     const int32_t *row_of, int32_t *page_row, int64_t first_page,
                                     int per_page, cudaStream_t st);
cudaError_t launch_mm_count_pages(const int32_t *page_row, int64_t first, int64_t n,
                                  const MmTables &t, cudaStream_t st);
// out[0..2] = pages in use, slots in use, live slots
cudaError_t launch_mm_stats(const MmTables &t, int64_t n_pages, unsigned long long *out,
                            cudaStream_t st);
cudaError_t launch_mm_rehash(const unsigned long long *old_key, const uint32_t *old_val,
                             int64_t old_cap, const MmTables &t, int *status, cudaStream_t st);
// out[i] = ns_row[row_of[ids[i]]] as an order-preserving unsigned key
cudaError_t launch_mm_ns_keys(const uint32_t *ids, int64_t count, const int32_t *row_of,
                              const int32_t *ns_row, uint32_t *out, cudaStream_t st);
// out[c] = by_row[row_of[c]], c < n
cudaError_t launch_by_id(const int32_t *by_row, const int32_t *row_of, int64_t n, int32_t *out,
                         cudaStream_t st);

// Chunk deletion (ak_delete.cu).  dead_row[row_of[id]] = 1 for the listed
// IDs (out-of-range IDs set EINVAL in *status and are skipped; dead_row
// NULL: check only).
// A newly deleted chunk's slot becomes invalid: page_live[page_row[row]]
// drops by one (page_row / page_live may be NULL).
cudaError_t launch_mark_dead(const int64_t *ids, int64_t n, int64_t n_total, const int32_t *row_of,
                             int32_t *dead_row, int *status, cudaStream_t st,
                             const int32_t *page_row = nullptr, int32_t *page_live = nullptr);
// EDEVICE in *status if any col[e] < first names a deleted chunk.
cudaError_t launch_check_dead_targets(const int32_t *col, int64_t nnz, int64_t first,
                                      const int32_t *row_of, const int32_t *dead_row, int *status,
                                      cudaStream_t st);
// Bitmaps of the deleted chunks, by row and by chunk ID ((n + 31) / 32 words
// each, by_id zeroed before), from dead_row.
cudaError_t launch_dead_bits(const int32_t *dead_row, const int32_t *ext_of, int64_t n,
                             uint32_t *by_row, uint32_t *by_id, cudaStream_t st);
// One edge list without the edges that touch a deleted chunk: an edge survives
// if its target is not deleted (bit tgt of dead_bits) and it is not in the row
// of a listed ID (rows found through own_row_of unless NULL).  Survivors keep
// their order and their logit and weight; where touched is given, an edge whose
// target's bit is set there gets its weight anew, row_softmax_weight(val,
// rstat[ext_of[target]]).
struct DropDead {
    int64_t n_rows, nnz;
    const int64_t *ptr;                 // [n_rows + 1]
    const int32_t *tgt;                 // [nnz]
    const float *val, *w;               // [nnz] logits, weights
    const uint32_t *dead_bits;          // by what tgt holds
    const int64_t *ids;                 // [n_ids] deleted chunk IDs
    int64_t n_ids, n_total;
    const int32_t *own_row_of;          // chunk ID -> row of the list, or NULL (rows are IDs)
    const uint32_t *touched;            // or NULL
    const int32_t *ext_of;
    const float2 *rstat;
    uint32_t *drop_bits;                // scratch [(nnz + 31) / 32], zeroed before
    uint32_t *keep_bits;                // scratch [(nnz + 31) / 32]: the survivors
    int32_t *word_pos;                  // scratch [(nnz + 31) / 32]: survivors before a word
    int32_t *counts;                    // scratch [drop_words(nnz)]
    int32_t *tgt_out;                   // [nnz]
    float *val_out, *w_out;             // [nnz]
};
int64_t drop_words(int64_t nnz);
cudaError_t launch_drop_dead_edges(const DropDead &d, cudaStream_t st);
// The row starts after launch_drop_dead_edges.  w (or NULL): rows that lost an
// edge get their softmax anew (w, rstat) and their row's bit in touched
// (row_of maps the list's rows, chunk IDs; zeroed before).
cudaError_t launch_drop_row_ptr(const DropDead &d, int64_t *ptr_out, float *w, float2 *rstat,
                                const int32_t *row_of, uint32_t *touched, cudaStream_t st);

// Propagation hop (a2): out[j,:] = u[j,:] + alpha * sum_{i->j} w_ij * in[i,:].
struct HopPlan {
    const int32_t *done;        // a reach plan (or NULL): with done[0] = 1 the call's
                                // kernels from the first hop on return at once
    SplitParams split;
    const int64_t *in_ptr;      // n+1
    const int32_t *in_src;      // nnz
    const float *in_w;          // nnz
    int64_t n;
    // rows whose in-degree exceeds the segment length are split
    int64_t n_split_rows;       // number of such rows
    const int32_t *split_row;   // [n_split_rows] row index
    const int64_t *split_slot0; // [n_split_rows+1] first partial slot of each split row
    int64_t n_segs;             // total segments of split rows (= partial slots)
    const int64_t *seg_e0;      // [n_segs] first edge, window-major order
    const int64_t *seg_e1;      // [n_segs] end edge
    const int32_t *seg_slot;    // [n_segs] partial slot (segments of a row are contiguous)
    const int32_t *split_order; // [n_split_rows] split rows by slot count, largest first
    const int32_t *slot_split;  // [n_segs] split row owning each partial slot
};
// Top-k filter fused into a hop's output: every written value whose key
// (score bits, ~chunk ID) is >= bound[column] is appended to that column's
// buffer, as the selection's filter pass would (see ak_select.cu).
struct HopFilter {
    const int32_t *ext_of;            // row -> chunk ID
    const unsigned long long *bound;  // [bp]
    unsigned int *cnt;                // [bp]
    unsigned long long *buf;          // [bp][cap]
    int64_t cap;
    NsScope ns;                       // candidates only within the query's namespace
};
// What the last hop may leave out, given a floor that every real query's k-th
// largest final value reaches (launch_prune_floor): rows whose upper bound
// (RowBounds) stays below it append nothing in any column, so the filter's
// output is unchanged without them (launch_keep).
struct HopBound {
    const int32_t *split_skip; // [n_split_rows] 1: split row to skip
    const int32_t *kept_rows;  // [n] rows kept whole that reach the floor ...
    const int64_t *kept_count; // ... [0] their number, [1] that of kept_segs (device)
    const int32_t *kept_segs;  // [n_segs] segments of the unpruned split rows
};
// Graph-only mass vectors for the row bounds, levels t0..t1 (level 0, all
// ones, already in place): mup[t] >= g (1 + eps) sum_i w_ij mup[t-1]_i and
// mdn[t] <= g' (1 - eps) sum_i w_ij mdn[t-1]_i, g / g' the rounding growth of
// a hop's sum over the row's edges.  mup / mdn are [levels + 1][n];
// `zeros` is [n]; split_vu/vl [n_split_rows] scratch.  With them, for every
// real query column (U0 / L0 u's row maxima / minima, Umax / Lmin their
// extremes over the live rows):
//   s^(H)_j <= (U0_j + Umax sum_{t<=H} alpha^t mup[t]_j) (1 + eps),
//   s^(H)_j >= (L0_j + Lmin sum_{t<=H} alpha^t mdn[t]_j) (1 - eps)
// (by induction over the hops: every source's value lies in
// [Lmin (1 + ...), Umax (1 + ...)]).
cudaError_t launch_mass_levels(const HopPlan &p, int t0, int t1, float *mup, float *mdn,
                               const float *zeros, float *split_vu, float *split_vl,
                               cudaStream_t st);
// The row bounds of the last hop's output, evaluated where they are needed
// (the at most ~3H roundings of the evaluation stay far below the 1e-5,
// ~168 eps, for H <= 16):
// ub_j = (U0_j + Umax sum_t alpha^t Mup[t]_j)(1 + 1e-5),
// lb_j = (L0_j + Lmin sum_t alpha^t Mdn[t]_j)(1 - 1e-5), Horner over t.
__device__ __forceinline__ float row_upper_bound(const float *u0, const float *mup, int64_t n,
                                                 int H, float alpha, float umax, int64_t j) {
    float c = 0.f;
    for (int t = H; t >= 1; --t) c = alpha * (c + __ldg(mup + (int64_t)t * n + j));
    return fmaf(umax, c, u0[j]) * (1.f + 1e-5f);
}
__device__ __forceinline__ float row_lower_bound(const float *l0, const float *mdn, int64_t n,
                                                 int H, float alpha, float lmin, int64_t j) {
    if (!(lmin < INFINITY)) return 0.f;
    float c = 0.f;
    for (int t = H; t >= 1; --t) c = alpha * (c + __ldg(mdn + (int64_t)t * n + j));
    return fmaf(lmin, c, l0[j]) * (1.f - 1e-5f);
}
__device__ __forceinline__ float ext_umax(const unsigned int *ext) { return __uint_as_float(ext[0]); }
__device__ __forceinline__ float ext_lmin(const unsigned int *ext) {
    return __uint_as_float(0x7f800000u - ext[1]);
}
// What the bounds of a call's last hop come from: u's row maxima and minima,
// the mass levels 0..H [H + 1][n], and ext [2] from the score GEMM's epilogue:
// ext[0] the bits of Umax = max_j u0_j, ext[1] 0x7f800000 minus the bits of
// Lmin = min over u0_j > 0 of l0_j (both maxima, so zero is the empty value).
struct RowBounds {
    const float *u0, *l0, *mup, *mdn;
    const unsigned int *ext;
    int64_t n;
    int H;
    float alpha;
};
// Floors of a namespace-scoped last hop: a row can only be selected by the
// batch's queries of its own namespace, so its floor is that namespace's
// (tag_floor[i] for tags[i] == its tag; the tags are the batch's distinct
// query namespaces, ascending), or +inf when no query of the batch has its
// namespace.  ns_row == NULL: the one device floor applies to every row.
struct NsFloors {
    const int32_t *ns_row;    // [n] namespace tag of each row
    const int32_t *tags;      // [<= PF_TAGS] distinct query tags, ascending
    const int *n_tags;        // their number (device)
    const float *tag_floor;   // [<= PF_TAGS]
};
constexpr int PF_TAGS = 256;
// split_skip, kept_rows, kept_segs and kept_count (HopBound; kept_count zeroed
// before) against the floor, or with nf the rows' namespaces' floors.
// words: keep_words(p) words of scratch.
int64_t keep_words(const HopPlan &p);
cudaError_t launch_keep(const HopPlan &p, const RowBounds &rb, const float *floor_p,
                        const NsFloors *nf, int32_t *split_skip, int32_t *kept_rows,
                        int32_t *kept_segs, int64_t *kept_count, int32_t *words,
                        cudaStream_t st, int *launches);
// The floors of a scoped batch: tags = the distinct q_ns of the n_real query
// columns, and for each tag the largest of (a) the smallest score that the
// filter bound of any of its queries admits and (b) the k-th largest lower
// bound over the split rows of that namespace, taken heaviest first (split_order), at
// most PF_ROWS of them (any subset of a namespace's rows gives a floor that
// each of its queries' k-th largest final score reaches).
// The filter bounds are raised to the floors, which hold for them too.
cudaError_t launch_ns_floors(unsigned long long *bound, const int32_t *q_ns, int n_real,
                             const RowBounds &rb, const int32_t *ns_row, const int32_t *split_row,
                             const int32_t *split_order, int64_t n_split, int k, int32_t *tags,
                             int *n_tags, float *tag_floor, cudaStream_t st);
// floor = max(the smallest score any real column's filter bound admits,
// and, if lb_rows != NULL, the k-th largest lower bound over the rows
// lb_rows[order[i]], i < n_lb_rows), written to floor_out; the filter bounds
// are raised to it.  The second term is only valid when every row may be
// selected by every query (no namespace scope).
cudaError_t launch_prune_floor(unsigned long long *bound, int n_real, const RowBounds &rb,
                               const int32_t *lb_rows, const int32_t *order, int64_t n_lb_rows,
                               int k, float *floor_out, const int32_t *done, cudaStream_t st);
cudaError_t launch_fill_f32(float *v, int64_t n, float x, cudaStream_t st);

// ------------------------------------------------------------------ reach (ak_reach.cu)
// Final scores of a few candidate rows straight from u: s^(H)_j = u_j +
// sum_t alpha^t sum_k C_t[k][j] u_k with graph-only reach coefficients.
constexpr int REACH_T = 128;         // candidate rows kept
constexpr int REACH_MAX_H = 4;       // hop counts it serves: 2 .. REACH_MAX_H
struct ReachBuild {
    int64_t n;
    const float *mup;                // mass levels 0..2 [3][n] (candidate choice)
    const int64_t *in_ptr;           // in-edge CSR (row space)
    const int32_t *in_src;
    const float *in_w;
    const int64_t *row_ptr;          // out-edge CSR (chunk IDs)
    const int32_t *col, *row_of;
    const float *w;
    int32_t *rows;                   // [REACH_T] candidate rows
    int *t_cnt;                      // their number (device)
    int32_t *map;                    // [n] row -> candidate slot or -1
    unsigned long long *pick;        // [reach_pick_words()] scratch
};
int64_t reach_pick_words();
struct ReachLevels {
    const float *level[REACH_MAX_H]; // C_1, C_2, ...: [n][REACH_T] each
};
// The candidates, their map and C_1; then Cn = C_{t+1} from Cp = C_t.
cudaError_t launch_reach_pick(const ReachBuild &rb, float *C1, cudaStream_t st);
cudaError_t launch_reach_level(const ReachBuild &rb, const float *Cp, float *Cn, cudaStream_t st);
// The reach path's floor, flags and plan: floor = the k-th largest lower bound
// over the candidates; then every row's upper bound against it: keep[REACH_T]
// flags the candidates that reach it, *bad counts the other rows that do, and
// the last CTA to finish writes the plan (REACH_PLAN_INTS below).  ws:
// int32[REACH_WS] scratch (keep, bad, done), zeroed before.
constexpr int REACH_WS = REACH_T + 2;
struct ReachFlags {
    const float *u0, *l0;            // u's row maxima / minima [n]
    const float *mup, *mdn;          // mass levels [H + 1][n]
    const unsigned int *ext;         // Umax / Lmin (RowBounds::ext)
    int64_t n;
    int H;
    float alpha;
    const int32_t *rows;             // the candidates
    int k;
    const int32_t *map;              // row -> candidate slot or -1
    const int *t_cnt;                // candidates (device)
    int32_t *ws;
    int32_t *plan;                   // [REACH_PLAN_INTS]
    const int32_t *skip;             // or NULL: with skip[0] = 1 the hops run, unseen
    unsigned long long *tried, *told;    // or NULL: where the candidates do not
    unsigned long long again;            // suffice get the mark `again` (told: host)
    const float *shift;              // the query columns' shifts (or NULL): the hops run
    int bp;                          // above REACH_SPLIT_SHIFT
};
// The largest shift c of a batch that the candidates' tensor-core pass takes from
// the hops.  Its operands hold 16 bits of u - exp(-2c), which is at most 1 - exp(-2c)
// of u, so its error grows with c where the hops' does not: against 64 bits (rms of
// the scores; 65,537 and 262,144 chunks, 48 and 200 queries, two to four hops)
// 4e-8 at 2c = 0.06 (dim 1024 at the default temperature), 6e-8 at 0.25 (dim 64),
// up to 9.7e-8 at 0.5, 1.6e-7 at 1 and 2.9e-7 at 2; the hops 9e-8 to 1.7e-7
// throughout.  (Two hops with 65 queries and more took the tensor cores before
// there was a limit, with a larger error, and have none.)
constexpr float REACH_SPLIT_SHIFT = 0.1875f;
cudaError_t launch_reach_flags(const ReachFlags &f, cudaStream_t st, int *launches);
int reach_parts();                   // CTAs of the candidates' pass (partial rows)
// The call's plan on the device (int32[REACH_PLAN_INTS], written by
// launch_reach_flags): plan[0] = 1 when the flagged candidates suffice for
// top-k (else the hops run), plan[1] = their number nk, plan[2..] their
// slots in ascending order, plan[REACH_PLAN_WIDE] = 1 when a flagged slot
// is 64 or above.
constexpr int REACH_PLAN_WIDE = REACH_T + 2;
constexpr int REACH_PLAN_INTS = REACH_T + 3;
// Rows of the packed coefficients: n rounded up to a whole 64-row stage.
int64_t reach_pad_rows(int64_t n);
// Every candidate's combined coefficients sum_t alpha^t C_t as bf16 hi + lo,
// [REACH_T][reach_pad_rows(n)] each, and their column sums in 64 bits
// (sums[REACH_T]; reach_sum_words(n) words in all, the rest scratch)
// (graph-only; repacked when the graph, alpha or H change).
int64_t reach_sum_words(int64_t n);
cudaError_t launch_reach_pack(const ReachLevels &C, int64_t n, int H, float alpha,
                              uint16_t *coef_hi, uint16_t *coef_lo, double *sums, cudaStream_t st);
// partial: [reach_parts()][REACH_T][bp] scratch; with plan[0] = 1 the
// flagged candidates' keys are written to each real column's buffer
// (cnt[b] = nk); with plan[0] = 0 both kernels return at once.  bp = 64, 128
// or 256.  u_hi, u_lo: the score GEMM's split-bf16 u - batch_u_min(shift).
cudaError_t launch_reach_scores(const uint16_t *u_hi, const uint16_t *u_lo, const float *shift,
                                int bp, int B, int64_t n, const uint16_t *coef_hi,
                                const uint16_t *coef_lo, const double *sums, const int32_t *plan,
                                const int32_t *rows, const int32_t *ext_of, float *partial,
                                unsigned int *cnt, unsigned long long *buf, int64_t cap,
                                int *status, cudaStream_t st, int *launches);
// The same in fp32, for B <= 32: coef [n][REACH_T] the combined coefficients,
// sums as above, u [n][bp] the score slab, ext u's extremes, partial
// [reach_fma_parts(n)][REACH_T][bp] scratch.
cudaError_t launch_reach_combine(const ReachLevels &C, int64_t n, int H, float alpha, float *coef,
                                 double *sums, cudaStream_t st);
int reach_fma_parts(int64_t n);
cudaError_t launch_reach_fma(const float *u, int bp, int B, int64_t n, const float *coef,
                             const double *sums, const unsigned int *ext, const int32_t *plan,
                             const int32_t *rows, const int32_t *ext_of, float *partial,
                             unsigned int *cnt, unsigned long long *buf, int64_t cap,
                             cudaStream_t st, int *launches);
// `counters` = 2 device ints (work queues), zeroed before.
// `flt` may be NULL (no filter), `hb` NULL (no row bounds).
cudaError_t launch_hop(const HopPlan &p, const float *u, const float *in, float *out, int bp,
                       float alpha, float *partial, int *counters, const HopFilter *flt,
                       cudaStream_t st, int *launches, const HopBound *hb = nullptr);

// ------------------------------------------------------------------ selection
// Top-k of every column of a slab (a3): bound from a row sample, filter
// pass, merge (see ak_select.cu).  The workspace holds sp.words 64-bit words.
struct SelectPlan {
    int64_t n;          // rows
    int bp, k;
    int64_t stride;     // sample every stride-th row
    int64_t n_sample;
    int64_t cap;        // buffer capacity per column
    // workspace offsets in 64-bit words: bounds, counts, buffers, the
    // sample transposed to [bp][n_sample] 32-bit keys
    int64_t off_bound, off_cnt, off_buf, off_tr, words;
};
// force_stride > 0 samples every force_stride-th row instead of the default.
SelectPlan select_plan(int64_t n, int bp, int k, int sm_count, int64_t force_stride = 0);

// keysT [sp.bp][sp.n_sample]: the last hop's selection keys of the sample
// rows, none above its row's final key (see k_hop_sample).
cudaError_t launch_hop_sample(const HopPlan &p, const SelectPlan &sp, const float *u,
                              const float *in, float alpha, NsScope ns, uint32_t *keysT,
                              cudaStream_t st, int *launches);

// Retrieval: rows are store rows; keys and outputs carry chunk IDs
// (ext_of), so ties resolve to the lower chunk ID; page_row is indexed by
// row (row_of).  Scores are divided by Z = sum of zpart's first n_ztiles rows.
// With a scope (ns.q_ns != NULL) a query whose namespace holds fewer than k
// chunks gets its list padded with ID -1, score 0, page -1; with
// sort_by_time the k winners are written in ascending chunk ID order
// (Algorithm 1, SortByTime) instead of by score.
cudaError_t launch_select(const SelectPlan &sp, const float *s, int b, unsigned long long *ws,
                          const float *zpart, int64_t n_ztiles, const int32_t *ext_of,
                          const int32_t *row_of, const int32_t *page_row, int64_t *ids,
                          float *scores, int32_t *page_ids, int32_t *n_pages, int *status,
                          NsScope ns, int sort_by_time, cudaStream_t st, int *launches);
// Same selection over signed values (cosines) among rows whose chunk ID is
// below id_limit: the k best of each of the b columns go to nbr_ids /
// nbr_cos rows c_base .. c_base+b-1.
cudaError_t launch_select_signed(const SelectPlan &sp, const float *s, int b,
                                 unsigned long long *ws, const int32_t *ext_of, int64_t id_limit,
                                 int64_t c_base, int32_t *nbr_ids, float *nbr_cos, int *status,
                                 cudaStream_t st, int *launches, NsScope ns = NsScope{});
// Bound pass alone (retrieval): ws + sp.off_bound gets the k-th largest sampled
// key of the b real columns (padding columns an all-ones bound), the column counts
// are cleared.  For a filter fused into the score, from the sampled score slab
// `s`, or (s == NULL) into the last hop, from the keys that launch_hop_sample left
// at ws + sp.off_tr.  `slack` lowers each bound by that many units of the score's
// last place (margin for a sample computed by another launch).
cudaError_t launch_sample_bound(const SelectPlan &sp, const float *s, int b,
                                const int32_t *ext_of, unsigned long long *ws, cudaStream_t st,
                                int *launches, uint32_t slack = 0, NsScope ns = NsScope{},
                                const int32_t *done = nullptr);
// A column of the last hop recomputed by the merge when the filter fused
// into that hop (which writes no output slab) overflowed its buffer:
// dst[j,c] = u[j,c] + alpha * sum_{e in in(j)} in_w[e] * prev[in_src[e],c].
// Without hops (the score itself, fused with the filter, wrote no slab):
// dst[j,c] = exp(tau <e_j, q_c> - shift[c]) from the stored bf16 values.
struct ColumnRecompute {
    int kind;     // 0 none, 1 last hop, 2 score
    const float *u, *prev;
    const int64_t *in_ptr;
    const int32_t *in_src;
    const float *in_w;
    float alpha;
    const uint16_t *emb, *qp;   // kind 2: E [n][dim], padded queries [bp][dim]
    int dim;
    float tau;
    const float *shift;
    float *dst;   // [n][bp]; the merge reads the overflowed column from here
};
// Row j -> chunk ID of a strided sample: out[v] = ext_of[v * stride].
cudaError_t launch_ext_sample(const int32_t *ext_of, int64_t n_sample, int64_t stride,
                              int32_t *out, cudaStream_t st);
// Merge only: the k winners per column from the buffers filled by a filter
// pass (falls back to the column of `s` where a buffer overflowed, after
// recomputing it into s when `rc` is given; then s must be rc->dst).
cudaError_t launch_topk_merge(const SelectPlan &sp, const float *s, int b,
                              const unsigned long long *ws, const float *zpart, int64_t n_ztiles,
                              const int32_t *ext_of, const int32_t *row_of,
                              const int32_t *page_row, int64_t *ids, float *scores,
                              int32_t *page_ids, int32_t *n_pages, int *status,
                              const ColumnRecompute *rc, NsScope ns, int sort_by_time,
                              cudaStream_t st, int *launches);
// Small stores (topk_direct(n)): the same selection straight from the slab of
// final scores, in one launch.
bool topk_direct(int64_t n);
cudaError_t launch_topk_direct(const float *s, int64_t n, int bp, int b, int k,
                               const float *zpart, int64_t n_ztiles, const int32_t *ext_of,
                               const int32_t *row_of, const int32_t *page_row, int64_t *ids,
                               float *scores, int32_t *page_ids, int32_t *n_pages, int *status,
                               NsScope ns, int sort_by_time, cudaStream_t st, int *launches);
// bound[c] = the k-th largest of the n_sample keys keys_t[c][*] (k <= 64) as a
// key with the chunk-ID half zero, 0 if fewer than k keys are nonzero; ~0
// for the padding columns b <= c < bp; cnt[c] = 0.  One CTA a column.
cudaError_t launch_sample_kth_keys(const uint32_t *keys_t, int64_t n_sample, int bp, int b, int k,
                                   unsigned long long *bound, unsigned int *cnt, cudaStream_t st,
                                   int *launches);
// Top-k of each column's filter buffer (no overflow): nbr rows 0..n_cols-1.
cudaError_t launch_buf_merge_signed(const unsigned int *cnt, const unsigned long long *buf,
                                    int64_t cap, int64_t n_cols, int k, int32_t *nbr_ids,
                                    float *nbr_cos, int *status, cudaStream_t st, int *launches);

}  // namespace ak
