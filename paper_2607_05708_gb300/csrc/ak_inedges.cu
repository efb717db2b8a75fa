// Incremental update of the in-edge transpose after a relation update
// (a7, §4.1 cross-chunk relations): instead of re-sorting every edge of the
// store, the old in-edge lists are moved to their new offsets and only the
// new edges are placed; the in-edges of sources whose rows gained edges get
// their weights anew from their logits and those rows' softmax statistics.
//
// Layout facts this relies on (all enforced by the update's preconditions):
//   * the new chunks' rows come after every old row (appends grow the store
//     at the end), so in an old target's list the new sources sort after
//     all old ones;
//   * new chunks have no in-edges before the update and are not linked to
//     each other, so a new chunk's in-edges are exactly its M reciprocal
//     edges;
//   * the out-edge weights are w = exp(aff - max_row) * inv_row with the
//     per-row (max, inv) kept in `rstat`, so a weight recomputed here for a
//     source whose row gained edges has the same bits as the out-edge's, and
//     the other edges keep theirs.
#include "ak_common.cuh"

namespace ak {

// New list starts: the old ones moved by the forward pairs into the rows
// before (counted in the sorted target rows) and by the new rows before (M
// reciprocal edges each, counted in the sorted new rows).
__global__ void k_new_in_ptr(const int64_t *__restrict__ in_ptr_old, int64_t n,
                             const uint32_t *__restrict__ fwd, int64_t pairs,
                             const uint32_t *__restrict__ new_rows, int64_t n_new, int M,
                             int64_t *__restrict__ in_ptr_new) {
    griddep_wait();
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= n;
         r += (int64_t)gridDim.x * blockDim.x)
        in_ptr_new[r] = in_ptr_old[r] + lower_bound_u32(fwd, pairs, (uint64_t)r) +
                        (int64_t)M * lower_bound_u32(new_rows, n_new, (uint64_t)r);
}

__global__ void k_row_keys(const int32_t *__restrict__ row_of, int64_t first, int64_t n_new,
                           uint32_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    griddep_wait();
    for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < n_new;
         a += (int64_t)gridDim.x * blockDim.x) {
        keys[a] = (uint32_t)row_of[first + a];
        vals[a] = (uint32_t)a;
    }
}

// ------------------------------------------------------------------ moved edges
// Old edges to their new places, each with its logit and weight.  An edge moves
// by the edges inserted before its row, so its shift only changes where a row
// that gained edges ends: cut[] holds those ends (one entry an inserted edge,
// ascending), cut2[] the starts of rows whose insertions come in equal blocks of
// mult2 edges (the new rows, which had none).  A CTA takes MOVE_TILE consecutive
// edges; 32 with no cut among them, as most, move together, else an edge
// searches the few cuts there.  Bound by memory, 24 bytes an edge
// (finding every edge's row instead: 60 us for 8.4M edges, 29 so; 16 edges a
// thread 38, as the registers then cost a CTA an SM).
// Weights are kept, or recomputed where touched has the bit of the edge's tgt.
constexpr int MOVE_PER = 8, MOVE_TILE = 256 * MOVE_PER;

// cut[p] = ptr[sorted[p] + end], p < count
__global__ void k_move_cuts(const int64_t *__restrict__ ptr, const uint32_t *__restrict__ sorted,
                            int64_t count, int end, uint32_t *__restrict__ cut) {
    griddep_wait();
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < count;
         p += (int64_t)gridDim.x * blockDim.x)
        cut[p] = (uint32_t)ptr[sorted[p] + end];
}

// tile_cut[t] / tile_cut2[t]: the cuts before edge t * MOVE_TILE.
__global__ void k_move_tiles(const uint32_t *__restrict__ cut, int64_t n_cut,
                             const uint32_t *__restrict__ cut2, int64_t n_cut2, int64_t tiles,
                             int32_t *__restrict__ tile_cut, int32_t *__restrict__ tile_cut2) {
    griddep_wait();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t > tiles) return;
    tile_cut[t] = (int32_t)lower_bound_u32(cut, n_cut, (uint64_t)t * MOVE_TILE);
    tile_cut2[t] = (int32_t)lower_bound_u32(cut2, n_cut2, (uint64_t)t * MOVE_TILE);
}

__global__ __launch_bounds__(256, 4) void k_move_edges(const MoveEdges m,
                                                       const uint32_t *__restrict__ cut,
                                                       const uint32_t *__restrict__ cut2,
                                                       const int32_t *__restrict__ tile_cut,
                                                       const int32_t *__restrict__ tile_cut2) {
    griddep_wait();
    const int64_t tile = blockIdx.x, e0 = tile * MOVE_TILE + threadIdx.x;
    int32_t t[MOVE_PER];
    float v[MOVE_PER], w[MOVE_PER];
#pragma unroll
    for (int j = 0; j < MOVE_PER; ++j) {
        const int64_t e = e0 + 256 * j;
        const bool ok = e < m.nnz;
        t[j] = ok ? __ldcs(m.tgt + e) : 0;
        v[j] = ok ? __ldcs(m.val + e) : 0.f;
        w[j] = ok ? __ldcs(m.w + e) : 0.f;
    }
    const int32_t c0 = tile_cut[tile], c1 = tile_cut[tile + 1];
    const int32_t d0 = tile_cut2[tile], d1 = tile_cut2[tile + 1];
    // lane j: the cuts at or before the first and the last edge of the warp's j-th
    // 32 edges
    const int lane = threadIdx.x & 31;
    const int64_t w0 = e0 - lane + 256 * (lane & (MOVE_PER - 1));
    auto upto = [&](const uint32_t *c, int32_t lo, int32_t hi, int64_t e) {
        return hi > lo ? lo + (int32_t)lower_bound_u32(c + lo, hi - lo, (uint64_t)e + 1) : lo;
    };
    const int32_t fa = upto(cut, c0, c1, w0), fb = upto(cut, c0, c1, w0 + 31);
    const int32_t ga = upto(cut2, d0, d1, w0), gb = upto(cut2, d0, d1, w0 + 31);
    // touched sources' statistics, all gathers in flight together
    if (m.touched) {
        uint32_t hit = 0u;
#pragma unroll
        for (int j = 0; j < MOVE_PER; ++j)
            hit |= ((__ldg(m.touched + (t[j] >> 5)) >> (t[j] & 31)) & 1u) << j;
        if (__any_sync(0xffffffffu, hit != 0u)) {
            int32_t id[MOVE_PER];
#pragma unroll
            for (int j = 0; j < MOVE_PER; ++j) id[j] = (hit >> j) & 1u ? m.ext_of[t[j]] : -1;
#pragma unroll
            for (int j = 0; j < MOVE_PER; ++j)
                if (id[j] >= 0) w[j] = row_softmax_weight(v[j], m.rstat[id[j]]);
        }
    }
#pragma unroll
    for (int j = 0; j < MOVE_PER; ++j) {
        const int64_t e = e0 + 256 * j;
        const int32_t ca = __shfl_sync(0xffffffffu, fa, j), cb = __shfl_sync(0xffffffffu, fb, j);
        const int32_t da = __shfl_sync(0xffffffffu, ga, j), db = __shfl_sync(0xffffffffu, gb, j);
        if (e >= m.nnz) continue;
        const int64_t by = cb > ca ? upto(cut, ca, cb, e) : ca;
        const int64_t by2 = db > da ? upto(cut2, da, db, e) : da;
        const int64_t p = e + by + by2 * m.mult2;
        __stcs(m.tgt_out + p, t[j]);
        __stcs(m.val_out + p, v[j]);
        __stcs(m.w_out + p, w[j]);
    }
}

int64_t move_words(int64_t nnz, int64_t pairs, int64_t rows2) {
    return pairs + rows2 + 2 * (ceil_div<int64_t>(nnz, MOVE_TILE) + 1);
}

cudaError_t launch_move_edges(const MoveEdges &m, const int64_t *ptr, const uint32_t *sorted,
                              int64_t pairs, const uint32_t *rows2, int64_t n_rows2,
                              uint32_t *words, cudaStream_t st, int *launches) {
    if (m.nnz <= 0) return cudaSuccess;
    const int64_t tiles = ceil_div<int64_t>(m.nnz, MOVE_TILE), cap = (int64_t)device_sm_count() * 4;
    uint32_t *cut = words, *cut2 = cut + pairs;
    int32_t *tc = (int32_t *)(cut2 + n_rows2), *tc2 = tc + tiles + 1;
    auto grid = [&](int64_t n) {
        const int64_t want = ceil_div<int64_t>(n, 256);
        return (unsigned)(want < cap ? want : cap);
    };
    if (pairs > 0) launch_pdl(k_move_cuts, dim3((unsigned)(grid(pairs))), dim3(256), 0, st, ptr,
                              sorted, pairs, 1, cut);
    if (n_rows2 > 0) launch_pdl(k_move_cuts, dim3((unsigned)(grid(n_rows2))), dim3(256), 0, st,
                                ptr, rows2, n_rows2, 0, cut2);
    launch_pdl(k_move_tiles, dim3((unsigned)ceil_div<int64_t>(tiles + 1, 256)), dim3(256), 0, st,
               cut, pairs, cut2, n_rows2, tiles, tc, tc2);
    launch_pdl(k_move_edges, dim3((unsigned)tiles), dim3(256), 0, st, m, cut, cut2, tc, tc2);
    if (launches) *launches += 2 + (pairs > 0) + (n_rows2 > 0);
    return cudaGetLastError();
}

// Forward edges c -> t, pairs sorted by the row of t (fwd), those of one row by the
// row of c: after the row's old list, in that order.  (A place counted among the
// row's pairs instead took every one of them a scan of all: the square of the new
// chunks that chose one target.)
__global__ void k_place_fwd(const uint32_t *__restrict__ fwd, const uint32_t *__restrict__ order,
                            int64_t pairs, const float *__restrict__ nbr_cos, float scale,
                            int64_t first, int M, const int32_t *__restrict__ row_of,
                            const int64_t *__restrict__ in_ptr_old,
                            const int64_t *__restrict__ in_ptr_new, int32_t *__restrict__ src_new,
                            float *__restrict__ aff_new, const float2 *__restrict__ rstat,
                            float *__restrict__ w_new) {
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < pairs;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t p = order[i], rt = fwd[i];
        const int64_t rank = i - lower_bound_u32(fwd, i, rt);
        const int64_t pos = in_ptr_new[rt] + (in_ptr_old[rt + 1] - in_ptr_old[rt]) + rank;
        const float a = scale * nbr_cos[p];
        src_new[pos] = row_of[first + p / M];
        aff_new[pos] = a;
        w_new[pos] = row_softmax_weight(a, rstat[first + p / M]);   // source: chunk first + p / M
    }
}

// Reciprocal edges t -> c: new chunk c's list holds its M chosen chunks'
// rows in ascending order (rank by counting; one warp per new chunk).
__global__ void k_place_recip(const int32_t *__restrict__ nbr_ids, const float *__restrict__ nbr_cos,
                              float scale, int64_t first, int64_t n_new, int M,
                              const int32_t *__restrict__ row_of,
                              const int64_t *__restrict__ in_ptr_new, int32_t *__restrict__ src_new,
                              float *__restrict__ aff_new, const float2 *__restrict__ rstat,
                              float *__restrict__ w_new) {
    griddep_wait();
    const int lane = threadIdx.x & 31;
    int64_t a = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (; a < n_new; a += stride) {
        const int32_t *ids = nbr_ids + a * M;
        const int64_t o = in_ptr_new[row_of[first + a]];
        for (int t = lane; t < M; t += 32) {
            const int32_t rt = row_of[ids[t]];
            int rank = 0;
            for (int u = 0; u < M; ++u) rank += row_of[ids[u]] < rt;
            const float af = scale * nbr_cos[a * M + t];
            src_new[o + rank] = rt;
            aff_new[o + rank] = af;
            w_new[o + rank] = row_softmax_weight(af, rstat[ids[t]]);   // source: chunk ids[t]
        }
    }
}

cudaError_t launch_in_edges_update(const InEdgeUpdate &u, const InEdgeScratch &s, cudaStream_t st,
                                   int *launches) {
    const int sms = device_sm_count();
    const int64_t pairs = u.n_new * u.M;
    if (pairs <= 0) return cudaErrorInvalidValue;
    int L = 4;
    // the new rows (each gets M reciprocal edges), then the forward pairs by target
    // row: taken in the order of the new rows, as the sort is stable
    bool alt = false, alt_r = false;
    uint32_t *rk = s.rows, *rv = rk + u.n_new, *rk2 = rv + u.n_new, *rv2 = rk2 + u.n_new;
    const int64_t want = ceil_div<int64_t>(u.n_new, 256);
    launch_pdl(k_row_keys, dim3((unsigned)(want < sms ? want : sms)), dim3(256), 0, st, u.row_of,
               u.first, u.n_new, rk, rv);
    cudaError_t e = radix_sort_pairs(rk, rv, rk2, rv2, u.n_new, u.row_bits, s.tmp, s.tmp_bytes, st,
                                     &alt_r, &L);
    const uint32_t *rows = alt_r ? rk2 : rk, *by_row = alt_r ? rv2 : rv;
    if (e == cudaSuccess)
        e = launch_pair_keys(u.nbr_ids, u.row_of, by_row, u.M, pairs, s.keys, s.vals, st);
    if (e == cudaSuccess)
        e = radix_sort_pairs(s.keys, s.vals, s.keys2, s.vals2, pairs, u.row_bits, s.tmp,
                             s.tmp_bytes, st, &alt, &L);
    const int64_t recip_rows = u.reciprocal ? u.n_new : 0;
    if (e != cudaSuccess) return e;
    const uint32_t *fwd = alt ? s.keys2 : s.keys, *order = alt ? s.vals2 : s.vals;
    launch_pdl(k_new_in_ptr, dim3((unsigned)(sms * 8)), dim3(256), 0, st, u.in_ptr_old, u.n, fwd,
               pairs, rows, recip_rows, u.M, u.in_ptr_new);
    const int64_t nnz_old = u.nnz_new - pairs * (u.reciprocal ? 2 : 1);
    MoveEdges mv{nnz_old, u.in_src_old, u.in_aff_old, u.in_w_old, u.in_src_new, u.in_aff_new,
                 u.in_w_new, u.M, u.touched, u.ext_of, u.rstat};
    e = launch_move_edges(mv, u.in_ptr_old, fwd, pairs, rows, recip_rows, s.move, st, &L);
    if (e != cudaSuccess) return e;
    launch_pdl(k_place_fwd, dim3((unsigned)(sms * 2)), dim3(256), 0, st, fwd, order, pairs,
               u.nbr_cos, u.scale, u.first, u.M, u.row_of, u.in_ptr_old, u.in_ptr_new,
               u.in_src_new, u.in_aff_new, u.rstat, u.in_w_new);
    if (u.reciprocal) {
        launch_pdl(k_place_recip, dim3((unsigned)(sms * 2)), dim3(256), 0, st, u.nbr_ids,
                   u.nbr_cos, u.scale, u.first, u.n_new, u.M, u.row_of, u.in_ptr_new, u.in_src_new,
                   u.in_aff_new, u.rstat, u.in_w_new);
        ++L;
    }
    if (launches) *launches += L;
    return cudaGetLastError();
}

}  // namespace ak
