// Chunk deletion (the deletions D of JointCompact, Algorithm 1; invalidated
// copies are logically tombstoned, §4.2): a deleted chunk keeps its row but
// is marked dead, gets no score, is never a candidate, and every relation
// edge into or out of it is dropped from both the out-edge CSR and the
// in-edge transpose.  Each list is compacted edge-parallel: a pass over its
// targets marks what it keeps (a mask every 32 edges) and counts it by tile, a
// pass over targets, logits and weights moves them; the masks and the counts
// before them give the new row starts.  Rows that lost nothing keep their
// weights.
#include "ak_common.cuh"

namespace ak {

// dead_row[row_of[id]] = 1 for every listed ID (dead_row NULL: only check);
// IDs outside [0, n_total) set EINVAL in the status word and are skipped.
__global__ void k_mark_dead(const int64_t *__restrict__ ids, int64_t n, int64_t n_total,
                            const int32_t *__restrict__ row_of, int32_t *__restrict__ dead_row,
                            int *status, const int32_t *__restrict__ page_row,
                            int32_t *__restrict__ page_live) {
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t id = ids[i];
        if (id < 0 || id >= n_total) {
            set_status(status, AKASHIC_EINVAL);
            continue;
        }
        if (!dead_row) continue;
        const int64_t r = row_of[id];
        if (atomicExch(&dead_row[r], 1) == 0 && page_live) atomicSub(&page_live[page_row[r]], 1);
    }
}

__global__ void k_dead_bits(const int32_t *__restrict__ dead_row,
                            const int32_t *__restrict__ ext_of, int64_t n,
                            uint32_t *__restrict__ by_row, uint32_t *__restrict__ by_id) {
    griddep_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // warp-uniform trip count: whole words
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < ((n + 31) & ~(int64_t)31);
         r += stride) {
        const bool dead = r < n && dead_row[r] != 0;
        const unsigned bits = __ballot_sync(0xffffffffu, dead);
        if ((threadIdx.x & 31) == 0) by_row[r >> 5] = bits;
        if (dead) {
            const uint32_t id = (uint32_t)ext_of[r];
            atomicOr(&by_id[id >> 5], 1u << (id & 31));
        }
    }
}

cudaError_t launch_dead_bits(const int32_t *dead_row, const int32_t *ext_of, int64_t n,
                             uint32_t *by_row, uint32_t *by_id, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    launch_pdl(k_dead_bits, dim3((unsigned)(device_sm_count() * 4)), dim3(256), 0, st, dead_row,
               ext_of, n, by_row, by_id);
    return cudaGetLastError();
}

// Every edge of the listed IDs' own rows is dropped (their out-edges in the
// out-CSR, their in-edges in the transpose): one CTA per deleted chunk, a word
// of 32 edges a thread (a hub's row has 10^5 and more).
__global__ void k_drop_rows(const int64_t *__restrict__ ids, int64_t n, int64_t n_total,
                            const int32_t *__restrict__ row_of, const int64_t *__restrict__ ptr,
                            uint32_t *__restrict__ drop_bits) {
    griddep_wait();
    for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
        const int64_t id = ids[i];
        if (id < 0 || id >= n_total) continue;
        const int64_t r = row_of ? row_of[id] : id;
        const int64_t a = ptr[r], b = ptr[r + 1];
        if (a >= b) continue;
        for (int64_t w = (a >> 5) + threadIdx.x; w <= (b - 1) >> 5; w += blockDim.x) {
            const int lo = a > 32 * w ? (int)(a - 32 * w) : 0;
            const int hi = b < 32 * (w + 1) ? (int)(b - 32 * w) : 32;
            const uint32_t m = (hi == 32 ? ~0u : (1u << hi) - 1u) & ~((1u << lo) - 1u);
            atomicOr(&drop_bits[w], m);
        }
    }
}

// The compaction, DROP_TILE consecutive edges a CTA, DROP_WORDS words of 32
// edges a warp: first the masks and the tiles' counts, then the move.  Bound by
// memory: 4 bytes an edge read to mark it, 12 read and written to move it, the
// bitmaps cached.  (It took flags, a scan and positions of 8 bytes an edge in
// memory before, ~60 bytes an edge more, and a softmax of every row: 1.20 ms
// for 200 chunks of 524,288 with 16.8M edges, read-back included, 0.59 now; a
// list's 470 MB take 88 us.)
constexpr int DROP_WORDS = 16;                          // a warp
constexpr int DROP_TILE = 8 * 32 * DROP_WORDS;
static int64_t drop_tiles(int64_t nnz) { return ceil_div<int64_t>(nnz, DROP_TILE); }
int64_t drop_words(int64_t nnz) { return tile_words(drop_tiles(nnz)); }

__global__ __launch_bounds__(256) void k_drop_mark(const DropDead d) {
    griddep_wait();
    __shared__ int warp_n[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t e0 = (int64_t)blockIdx.x * DROP_TILE + warp * 32 * DROP_WORDS;
    int32_t t[DROP_WORDS];
#pragma unroll
    for (int j = 0; j < DROP_WORDS; ++j) {
        const int64_t e = e0 + 32 * j + lane;
        t[j] = e < d.nnz ? d.tgt[e] : -1;
    }
    // lane j holds word j's bits from here on
    const bool has_word = lane < DROP_WORDS && e0 + 32 * lane < d.nnz;
    const uint32_t drop = has_word ? d.drop_bits[(e0 >> 5) + lane] : ~0u;
    uint32_t mine = 0u;
#pragma unroll
    for (int j = 0; j < DROP_WORDS; ++j) {
        const bool live = t[j] >= 0 && !((__ldg(d.dead_bits + (t[j] >> 5)) >> (t[j] & 31)) & 1u);
        const uint32_t keep = __ballot_sync(0xffffffffu, live);
        if (lane == j) mine = keep & ~drop;
    }
    if (has_word) d.keep_bits[(e0 >> 5) + lane] = mine;
    int n = __popc(mine);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0) warp_n[warp] = n;
    __syncthreads();
    if (threadIdx.x == 0) {
        int own = 0;
        for (int w = 0; w < 8; ++w) own += warp_n[w];
        d.counts[blockIdx.x] = own;
    }
}

__global__ __launch_bounds__(256, 4) void k_drop_edges(const DropDead d) {
    griddep_wait();
    __shared__ int warp_n[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t e0 = (int64_t)blockIdx.x * DROP_TILE + warp * 32 * DROP_WORDS;
    const int64_t word0 = e0 >> 5;
    const bool has_word = lane < DROP_WORDS && e0 + 32 * lane < d.nnz;
    const uint32_t mine = has_word ? d.keep_bits[word0 + lane] : 0u;   // lane j: word j
    int32_t t[DROP_WORDS];
    float v[DROP_WORDS], w[DROP_WORDS];
#pragma unroll
    for (int j = 0; j < DROP_WORDS; ++j) {
        const int64_t e = e0 + 32 * j + lane;
        const bool ok = e < d.nnz;
        t[j] = ok ? __ldcs(d.tgt + e) : 0;
        v[j] = ok ? __ldcs(d.val + e) : 0.f;
        w[j] = ok ? __ldcs(d.w + e) : 0.f;
    }
    // survivors before each word of the warp, before the warp, before the tile
    int incl = __popc(mine);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    const int pre = incl - __popc(mine);
    if (lane == 31) warp_n[warp] = incl;
    int64_t base = tile_base(d.counts, 0, blockIdx.x);   // (syncs the CTA)
    for (int x = 0; x < warp; ++x) base += warp_n[x];
    if (has_word) d.word_pos[word0 + lane] = (int32_t)(base + pre);
#pragma unroll
    for (int j = 0; j < DROP_WORDS; ++j) {
        const uint32_t keep = __shfl_sync(0xffffffffu, mine, j);
        const int at = __shfl_sync(0xffffffffu, pre, j);
        if (!((keep >> lane) & 1u)) continue;
        const int64_t p = base + at + __popc(keep & lt);
        float wj = w[j];
        if (d.touched && ((__ldg(d.touched + (t[j] >> 5)) >> (t[j] & 31)) & 1u))
            wj = row_softmax_weight(v[j], d.rstat[d.ext_of[t[j]]]);
        __stcs(d.tgt_out + p, t[j]);
        __stcs(d.val_out + p, v[j]);
        __stcs(d.w_out + p, wj);
    }
}

// new start of a row = the survivors before its old first edge
// (e = nnz: all of them, by the last word)
__device__ __forceinline__ int64_t kept_before(const DropDead &d, int64_t e) {
    if (e >= d.nnz) {
        const int64_t w = (d.nnz - 1) >> 5;
        return d.word_pos[w] + __popc(d.keep_bits[w]);
    }
    return d.word_pos[e >> 5] + __popc(d.keep_bits[e >> 5] & ((1u << (e & 31)) - 1u));
}

// Eight lanes a row: the new starts, and (out-CSR) the softmax of the rows that
// lost an edge, as k_row_softmax does it.
__global__ __launch_bounds__(256) void k_drop_row_ptr(const DropDead d,
                                                      int64_t *__restrict__ ptr_out,
                                                      float *__restrict__ w,
                                                      float2 *__restrict__ rstat,
                                                      const int32_t *__restrict__ row_of,
                                                      uint32_t *__restrict__ touched) {
    griddep_wait();
    constexpr int L = 8;
    const int lane = threadIdx.x & 31, sub = lane % L;
    const int64_t step = ((int64_t)gridDim.x * blockDim.x) / L;
    const int64_t warp0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 / L);
    for (int64_t r0 = warp0; r0 <= d.n_rows; r0 += step) {   // (warp-uniform)
        const int64_t r = r0 + lane / L;
        int64_t old = 0, a = 0, b = 0;
        if (r < d.n_rows) {
            const int64_t p0 = d.ptr[r], p1 = d.ptr[r + 1];
            old = p1 - p0;
            a = kept_before(d, p0);
            b = kept_before(d, p1);
            if (sub == 0) ptr_out[r] = a;
        } else if (r == d.n_rows && sub == 0) {
            ptr_out[r] = kept_before(d, d.nnz);
        }
        const bool lost = w && r < d.n_rows && b - a != old;
        if (!__any_sync(0xffffffffu, lost)) continue;
        float m = -INFINITY;
        if (lost)
            for (int64_t e = a + sub; e < b; e += L) m = fmaxf(m, d.val_out[e]);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        float s = 0.f;
        if (lost)
            for (int64_t e = a + sub; e < b; e += L) s += expf(d.val_out[e] - m);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lost && b > a) {
            const float2 stat = make_float2(m, 1.f / s);
            if (sub == 0) {
                rstat[r] = stat;
                const uint32_t row = (uint32_t)row_of[r];
                atomicOr(&touched[row >> 5], 1u << (row & 31));
            }
            for (int64_t e = a + sub; e < b; e += L) w[e] = row_softmax_weight(d.val_out[e], stat);
        }
    }
}

// Edges handed to an append may not point at a deleted chunk (targets below
// `first`; the batch's own chunks cannot be deleted yet).
__global__ void k_check_dead_targets(const int32_t *__restrict__ col, int64_t nnz, int64_t first,
                                     const int32_t *__restrict__ row_of,
                                     const int32_t *__restrict__ dead_row, int *status) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = col[e];
        if (c >= 0 && (int64_t)c < first && dead_row[row_of[c]]) set_status(status, AKASHIC_EDEVICE);
    }
}

cudaError_t launch_check_dead_targets(const int32_t *col, int64_t nnz, int64_t first,
                                      const int32_t *row_of, const int32_t *dead_row, int *status,
                                      cudaStream_t st) {
    if (nnz <= 0) return cudaSuccess;
    k_check_dead_targets<<<device_sm_count() * 4, 256, 0, st>>>(col, nnz, first, row_of, dead_row,
                                                                status);
    return cudaGetLastError();
}

cudaError_t launch_mark_dead(const int64_t *ids, int64_t n, int64_t n_total, const int32_t *row_of,
                             int32_t *dead_row, int *status, cudaStream_t st,
                             const int32_t *page_row, int32_t *page_live) {
    if (n <= 0) return cudaSuccess;
    launch_pdl(k_mark_dead, dim3((unsigned)(device_sm_count())), dim3(256), 0, st, ids, n, n_total,
               row_of, dead_row, status, page_row, page_live);
    return cudaGetLastError();
}

cudaError_t launch_drop_dead_edges(const DropDead &d, cudaStream_t st) {
    const int sms = device_sm_count();
    if (d.nnz <= 0) return cudaErrorInvalidValue;
    if (d.n_ids > 0) {
        const int64_t g = d.n_ids < (int64_t)sms * 16 ? d.n_ids : (int64_t)sms * 16;
        launch_pdl(k_drop_rows, dim3((unsigned)g), dim3(128), 0, st, d.ids, d.n_ids, d.n_total,
                   d.own_row_of, d.ptr, d.drop_bits);
    }
    const unsigned tiles = (unsigned)drop_tiles(d.nnz);
    launch_pdl(k_drop_mark, dim3(tiles), dim3(256), 0, st, d);
    cudaError_t e = launch_tile_groups(d.counts, tiles, st);
    if (e != cudaSuccess) return e;
    launch_pdl(k_drop_edges, dim3(tiles), dim3(256), 0, st, d);
    return cudaGetLastError();
}

cudaError_t launch_drop_row_ptr(const DropDead &d, int64_t *ptr_out, float *w, float2 *rstat,
                                const int32_t *row_of, uint32_t *touched, cudaStream_t st) {
    const int64_t want = ceil_div<int64_t>((d.n_rows + 1) * 8, 256);
    const int64_t cap = (int64_t)device_sm_count() * 16;
    launch_pdl(k_drop_row_ptr, dim3((unsigned)(want < cap ? want : cap)), dim3(256), 0, st, d,
               ptr_out, w, rstat, row_of, touched);
    return cudaGetLastError();
}

}  // namespace ak
