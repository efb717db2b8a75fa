// Relation update (a6, a7): for new chunks, the top-M related prior chunks
// by cosine of the stored embeddings, then the reciprocal insertion of those
// edges into the relation graph's CSR (arXiv 2607.05708, §4.1: cross-chunk
// inference selects the related prior chunks of each new chunk; Algorithm 1's
// LLMSelect of related prior chunks, in its Dense-only form of §5.5).
#include "ak_update.cuh"

namespace ak {

// Gather the embeddings of chunks c0 .. c0+b-1 (rows row_of[c]) into a
// zero-padded bp-row block.  Bound by latency: eight values a load (dim is a
// multiple of 64, both buffers are allocations of the library's own), 4096 rows
// of 1024 45 -> 9 us.
__global__ void k_gather_rows(const uint16_t *__restrict__ emb, const int32_t *__restrict__ row_of,
                              int64_t c0, int b, int bp, int dim, uint16_t *__restrict__ dst) {
    griddep_wait();
    const int per = dim / 8;
    const int64_t total = (int64_t)bp * per;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / per, t = i % per;
        reinterpret_cast<uint4 *>(dst)[i] =
            r < b ? reinterpret_cast<const uint4 *>(emb + (int64_t)row_of[c0 + r] * dim)[t]
                  : make_uint4(0u, 0u, 0u, 0u);
    }
}

__global__ void k_ext_sample(const int32_t *__restrict__ ext_of, int64_t n_sample, int64_t stride,
                             int32_t *__restrict__ out) {
    griddep_wait();
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_sample;
         v += (int64_t)gridDim.x * blockDim.x)
        out[v] = ext_of[v * stride];
}

cudaError_t launch_ext_sample(const int32_t *ext_of, int64_t n_sample, int64_t stride,
                              int32_t *out, cudaStream_t st) {
    if (n_sample <= 0) return cudaSuccess;
    launch_pdl(k_ext_sample, dim3((unsigned)(device_sm_count())), dim3(256), 0, st, ext_of,
               n_sample, stride, out);
    return cudaGetLastError();
}

// Exact path, batch by batch: dots of every row against 256 new chunks
// written to a slab, then the three-pass selection (used when a fused
// filter buffer overflows).
static akashic_status_t relate_top_m_batched(const UpdateArgs &a, cudaStream_t st, int *launches) {
    const int64_t n_old = a.n_rows;
    int bp_max = 32;
    while (bp_max < 256 && bp_max < a.n_new) bp_max <<= 1;
    int64_t words = 0;
    for (int bp = 32; bp <= bp_max; bp <<= 1) {
        SelectPlan sp = select_plan(n_old, bp, a.M, device_sm_count());
        words = sp.words > words ? sp.words : words;
    }
    uint16_t *qp = (uint16_t *)a.get(SCR_QP, (size_t)bp_max * a.dim * 2);
    float *dots = (float *)a.get(SCR_DOTS, (size_t)n_old * bp_max * 4);
    unsigned long long *cand = (unsigned long long *)a.get(SCR_CAND, (size_t)words * 8);
    akashic_status_t rc = (qp && dots && cand) ? AKASHIC_OK : AKASHIC_ENOMEM;
    cudaError_t e = cudaSuccess;
    for (int64_t off = 0; rc == AKASHIC_OK && off < a.n_new; off += 256) {
        const int b = (int)(a.n_new - off < 256 ? a.n_new - off : 256);
        int bp = 32;
        while (bp < b) bp <<= 1;
        launch_pdl(k_gather_rows, dim3((unsigned)(device_sm_count())), dim3(256), 0, st, a.emb,
                   a.row_of, a.first + off, b, bp, a.dim, qp);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = launch_dots(a.emb, n_old, 1, a.dim, qp, bp, 1, dots, a.status, st, launches);
        const SelectPlan sp = select_plan(n_old, bp, a.M, device_sm_count());
        if (e == cudaSuccess)
            e = launch_select_signed(sp, dots, b, cand, a.ext_of, a.first, off, a.nbr_ids,
                                     a.nbr_cos, a.status, st, launches,
                                     NsScope{nullptr, nullptr, a.dead_row});
        if (e != cudaSuccess) rc = AKASHIC_ECUDA;
        if (launches) *launches += 1;
    }
    if (rc == AKASHIC_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = AKASHIC_ECUDA;
    return rc;
}

// Fused path (a6): a per-new-chunk bound from every stride-th row of the
// store, then ONE tensor-core pass over all rows x all new chunks whose
// epilogue keeps only the keys above the bounds, then an exact selection
// of the M best among them.  The dots are never written to memory.
akashic_status_t relate_top_m(const UpdateArgs &a, cudaStream_t st, int *launches,
                              int *dev_status) {
    // every row of the store is scored; rows holding chunks >= first are
    // masked in the selection (rows are in page order, not ID order)
    const int64_t n = a.n_rows;
    const int sms = device_sm_count();
    const int n_ct = (int)ceil_div<int64_t>(a.n_new, 256);
    const int64_t n_pad = (int64_t)n_ct * 256;
    // every stride-th row is sampled: about 512 M rows, so the bound (the
    // M-th largest sampled value) lets through about M * stride rows per
    // new chunk, which the merge stages in shared memory
    int64_t stride = n / ((int64_t)512 * a.M);
    stride = stride < 1 ? 1 : (stride > 64 ? 64 : stride);
    const int64_t n_sample = ceil_div<int64_t>(n, stride);
    const int64_t cap = 4 * (int64_t)a.M * stride > 8192 ? 4 * (int64_t)a.M * stride : 8192;
    // the sample bounds of G column tiles come from one dots GEMM that
    // writes the sampled keys column-major and one k-th launch (G tiles of
    // sampled keys: <= 512 MB)
    const int64_t tile_bytes = n_sample * 256 * 4;
    int64_t G = ((int64_t)512 << 20) / tile_bytes;
    G = G < 1 ? 1 : (G > n_ct ? n_ct : G);
    SelectPlan sp = select_plan(n_sample, (int)G * 256, a.M, sms, 1);
    sp.cap = 0;                      // no candidate buffers: bounds only
    sp.off_tr = sp.off_buf;
    sp.words = sp.off_tr + ceil_div<int64_t>(sp.n_sample * sp.bp, 2);
    uint16_t *qp = (uint16_t *)a.get(SCR_QP, (size_t)n_pad * a.dim * 2);
    int32_t *ext_s = (int32_t *)a.get(SCR_EXTS, (size_t)n_sample * 4);
    unsigned long long *ws = (unsigned long long *)a.get(SCR_WS, (size_t)sp.words * 8);
    unsigned long long *bound = (unsigned long long *)a.get(SCR_BOUND, (size_t)n_pad * 8);
    unsigned int *cnt = (unsigned int *)a.get(SCR_CNT, (size_t)n_pad * 4);
    unsigned long long *buf = (unsigned long long *)a.get(SCR_BUF, (size_t)a.n_new * cap * 8);
    akashic_status_t rc =
        (qp && ext_s && ws && bound && cnt && buf) ? AKASHIC_OK : AKASHIC_ENOMEM;
    cudaError_t e = cudaSuccess;
    bool overflow = false;
    if (rc == AKASHIC_OK) {
        launch_pdl(k_gather_rows, dim3((unsigned)(sms * 2)), dim3(256), 0, st, a.emb, a.row_of,
                   a.first, (int)a.n_new, (int)n_pad, a.dim, qp);
        launch_pdl(k_ext_sample, dim3(sms), dim3(256), 0, st, a.ext_of, n_sample, stride, ext_s);
        e = cudaGetLastError();
        // deleted chunks are never neighbours: their sample rows carry no key
        const int32_t *dead_s = nullptr;
        if (e == cudaSuccess && a.dead_row) {
            int32_t *ds = (int32_t *)a.get(SCR_DEAD_S, (size_t)n_sample * 4);
            if (!ds) {
                rc = AKASHIC_ENOMEM;
            } else {
                launch_pdl(k_ext_sample, dim3(sms), dim3(256), 0, st, a.dead_row, n_sample, stride,
                           ds);
                e = cudaGetLastError();
                dead_s = ds;
            }
        }
        for (int64_t g0 = 0; rc == AKASHIC_OK && e == cudaSuccess && g0 < n_ct; g0 += G) {
            const int gt = (int)(n_ct - g0 < G ? n_ct - g0 : G);
            const int64_t left = a.n_new - g0 * 256;
            const int b = (int)(left < (int64_t)gt * 256 ? left : (int64_t)gt * 256);
            uint32_t *keys_t = (uint32_t *)(ws + sp.off_tr);
            e = launch_dots_keys_t(a.emb, n_sample, stride, a.dim, qp + g0 * 256 * a.dim, gt,
                                   ext_s, a.first, dead_s, keys_t, a.status, st, launches);
            if (e == cudaSuccess)
                e = launch_sample_kth_keys(keys_t, n_sample, gt * 256, b, a.M, bound + g0 * 256,
                                           (unsigned int *)(ws + sp.off_cnt), st, launches);
        }
        if (rc == AKASHIC_OK && e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (size_t)n_pad * 4, st);
        if (rc == AKASHIC_OK && e == cudaSuccess)
            e = launch_dots_filter(a.emb, n, a.dim, qp, n_ct, a.n_new, a.ext_of, a.first, bound,
                                   cnt, buf, cap, a.status, st, launches, a.dead_row);
        // the merge is queued before the host knows whether a buffer
        // overflowed (then the exact batched path starts over)
        if (rc == AKASHIC_OK && e == cudaSuccess)
            e = launch_buf_merge_signed(cnt, buf, cap, a.n_new, a.M, a.nbr_ids, a.nbr_cos,
                                        a.status, st, launches);
        unsigned int max_cnt = 0;
        if (rc == AKASHIC_OK && e == cudaSuccess) {
            unsigned int *h = (unsigned int *)malloc((size_t)a.n_new * 4);
            if (!h) {
                rc = AKASHIC_ENOMEM;
            } else {
                e = cudaMemcpyAsync(h, cnt, (size_t)a.n_new * 4, cudaMemcpyDeviceToHost, st);
                if (e == cudaSuccess)
                    e = cudaMemcpyAsync(dev_status, a.status, 4, cudaMemcpyDeviceToHost, st);
                if (e == cudaSuccess) e = cudaStreamSynchronize(st);
                for (int64_t c = 0; e == cudaSuccess && c < a.n_new; ++c)
                    max_cnt = h[c] > max_cnt ? h[c] : max_cnt;
                free(h);
            }
        }
        overflow = (int64_t)max_cnt > cap && *dev_status == 0;
        if (e != cudaSuccess && rc == AKASHIC_OK) rc = AKASHIC_ECUDA;
    }
    if (rc == AKASHIC_OK && overflow) {
        rc = relate_top_m_batched(a, st, launches);
        if (rc == AKASHIC_OK && cudaMemcpy(dev_status, a.status, 4, cudaMemcpyDeviceToHost) !=
                                    cudaSuccess)
            rc = AKASHIC_ECUDA;
    }
    return rc;
}

// ------------------------------------------------------------------ CSR insert
// The update's preconditions, by a thread a new chunk: EINVAL if the range's
// rows have out-edges, EDEVICE if an edge points at one of its chunks (its
// reciprocal edge would be a repeat).
__global__ void k_check_new_rows(const int64_t *__restrict__ rp, const int64_t *__restrict__ in_ptr,
                                 const int32_t *__restrict__ row_of, int64_t first, int64_t n_new,
                                 int *status) {
    griddep_wait();
    if (rp[first] != rp[first + n_new]) {
        set_status(status, AKASHIC_EINVAL);
        return;
    }
    for (int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; a < n_new;
         a += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = row_of[first + a];
        if (in_ptr[r + 1] != in_ptr[r]) set_status(status, AKASHIC_EDEVICE);
    }
}

cudaError_t launch_check_new_rows(const int64_t *rp, const int64_t *in_ptr, const int32_t *row_of,
                                  int64_t first, int64_t n_new, int *status, cudaStream_t st) {
    const int64_t want = ceil_div<int64_t>(n_new, 256), cap = device_sm_count();
    launch_pdl(k_check_new_rows, dim3((unsigned)(want < cap ? want : cap)), dim3(256), 0, st, rp,
               in_ptr, row_of, first, n_new, status);
    return cudaGetLastError();
}

__global__ void k_pair_keys(const int32_t *__restrict__ ids, const int32_t *__restrict__ map,
                            const uint32_t *__restrict__ order, int M, int64_t pairs,
                            uint32_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < pairs;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = order ? (int64_t)order[i / M] * M + i % M : i;
        keys[i] = (uint32_t)(map ? map[ids[p]] : ids[p]);
        vals[i] = (uint32_t)p;
    }
}

cudaError_t launch_pair_keys(const int32_t *ids, const int32_t *map, const uint32_t *order, int M,
                             int64_t pairs, uint32_t *keys, uint32_t *vals, cudaStream_t st) {
    if (pairs <= 0) return cudaSuccess;
    const int64_t want = ceil_div<int64_t>(pairs, 256), cap = (int64_t)device_sm_count() * 4;
    launch_pdl(k_pair_keys, dim3((unsigned)(want < cap ? want : cap)), dim3(256), 0, st, ids, map,
               order, M, pairs, keys, vals);
    return cudaGetLastError();
}

// New row starts: the old ones moved by the new rows before the row (M edges
// each) and by the reciprocal edges of the rows before it, counted in the
// sorted target IDs (a search of cached words a row instead of counting,
// adding up and scanning arrays of all rows).
__global__ void k_new_row_ptr(const int64_t *__restrict__ rp, int64_t n_rows, int64_t first,
                              int64_t n_new, int M, const uint32_t *__restrict__ tgt,
                              int64_t recips, int64_t *__restrict__ nrp) {
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n_rows;
         i += (int64_t)gridDim.x * blockDim.x) {
        int64_t before = i - first;
        before = before < 0 ? 0 : (before > n_new ? n_new : before);
        nrp[i] = rp[i] + before * M + lower_bound_u32(tgt, recips, (uint64_t)i);
    }
}

// Rows of the new chunks: their M neighbours in ascending ID order (one warp
// per new row; rank of each neighbour among the row's M by ID).
__global__ void k_fill_new_rows(const int32_t *__restrict__ nbr, const float *__restrict__ cosv,
                                int64_t first, int64_t n_new, int M, float scale,
                                const int64_t *__restrict__ nrp, int32_t *__restrict__ ncol,
                                float *__restrict__ naff) {
    griddep_wait();
    const int lane = threadIdx.x & 31;
    int64_t a = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (; a < n_new; a += stride) {
        const int32_t *row = nbr + a * M;
        const int64_t o = nrp[first + a];
        for (int t = lane; t < M; t += 32) {
            const int32_t id = row[t];
            int rank = 0;
            for (int u = 0; u < M; ++u) rank += row[u] < id;
            ncol[o + rank] = id;
            naff[o + rank] = scale * cosv[a * M + t];
        }
    }
}

// Reciprocal edges j -> new chunk, appended after row j's old edges in
// ascending new-chunk order.  `order` lists the (new, slot) pair indices
// stably sorted by target j (tgt), so pairs of one j come in ascending new ID.
__global__ void k_fill_recip(const uint32_t *__restrict__ order, const uint32_t *__restrict__ tgt,
                             int64_t pairs, const float *__restrict__ cosv, int64_t first, int M,
                             float scale, const int64_t *__restrict__ rp,
                             const int64_t *__restrict__ nrp, int32_t *__restrict__ ncol,
                             float *__restrict__ naff) {
    griddep_wait();
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < pairs;
         p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t pair = order[p];
        const int64_t j = tgt[p];
        const int64_t rank = p - lower_bound_u32(tgt, p, (uint64_t)j);
        const int64_t pos = nrp[j] + (rp[j + 1] - rp[j]) + rank;
        ncol[pos] = (int32_t)(first + pair / M);
        naff[pos] = scale * cosv[pair];
    }
}

__global__ void k_first_row(int64_t first, uint32_t *__restrict__ out) {
    griddep_wait(); *out = (uint32_t)first; }

// The softmax of the rows that gained edges (the new rows, then each target's
// row, at its first pair), eight lanes a row in k_row_softmax's order, and
// their rows' bits in touched.
__global__ __launch_bounds__(256) void k_gained_softmax(const uint32_t *__restrict__ tgt,
                                                        int64_t recips, int64_t first,
                                                        int64_t n_new,
                                                        const int64_t *__restrict__ nrp,
                                                        const float *__restrict__ naff,
                                                        const int32_t *__restrict__ row_of,
                                                        float *__restrict__ nw_,
                                                        float2 *__restrict__ rstat,
                                                        uint32_t *__restrict__ touched) {
    griddep_wait();
    constexpr int L = 8;
    const int lane = threadIdx.x & 31, sub = lane % L;
    const int64_t items = n_new + recips;
    const int64_t step = ((int64_t)gridDim.x * blockDim.x) / L;
    const int64_t warp0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 / L);
    for (int64_t i0 = warp0; i0 < items; i0 += step) {   // (warp-uniform)
        const int64_t i = i0 + lane / L;
        int64_t r = -1;
        if (i < n_new) {
            r = first + i;
        } else if (i < items) {
            const int64_t p = i - n_new;
            if (p == 0 || tgt[p - 1] != tgt[p]) r = tgt[p];
        }
        const int64_t a = r >= 0 ? nrp[r] : 0, b = r >= 0 ? nrp[r + 1] : 0;
        float m = -INFINITY;
        for (int64_t e = a + sub; e < b; e += L) m = fmaxf(m, naff[e]);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        float s = 0.f;
        for (int64_t e = a + sub; e < b; e += L) s += expf(naff[e] - m);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (b > a) {
            const float2 stat = make_float2(m, 1.f / s);
            if (sub == 0) {
                rstat[r] = stat;
                const uint32_t row = (uint32_t)row_of[r];
                atomicOr(&touched[row >> 5], 1u << (row & 31));
            }
            for (int64_t e = a + sub; e < b; e += L) nw_[e] = row_softmax_weight(naff[e], stat);
        }
    }
}

akashic_status_t csr_insert(const UpdateArgs &a, const int64_t *rp, const int32_t *col,
                            const float *aff, const float *w, int64_t nnz, int64_t *new_rp,
                            int32_t *new_col, float *new_aff, float *new_w, float2 *rstat,
                            uint32_t *touched, cudaStream_t st, int *launches) {
    const int64_t n_rows = a.n_rows, pairs = a.n_new * a.M, recips = a.reciprocal ? pairs : 0;
    const int sms = device_sm_count();
    const size_t tmp_bytes = radix_tmp_bytes(pairs) + 4096;
    uint32_t *keys = (uint32_t *)a.get(SCR_KEYS, (size_t)pairs * 4 + 16);
    uint32_t *vals = (uint32_t *)a.get(SCR_VALS, (size_t)pairs * 4 + 16);
    uint32_t *keys2 = (uint32_t *)a.get(SCR_KEYS2, (size_t)pairs * 4 + 16);
    uint32_t *vals2 = (uint32_t *)a.get(SCR_VALS2, (size_t)pairs * 4 + 16);
    void *tmp = a.get(SCR_TMP, tmp_bytes);
    uint32_t *words = (uint32_t *)a.get(SCR_MOVE, (size_t)(1 + move_words(nnz, pairs, a.n_new)) * 4);
    if (!keys || !vals || !keys2 || !vals2 || !tmp || !words) return AKASHIC_ENOMEM;
    cudaError_t e = cudaMemsetAsync(touched, 0, (size_t)ceil_div<int64_t>(n_rows, 32) * 4, st);
    int L = 5;
    bool alt = false;
    if (e == cudaSuccess && recips > 0) {
        int bits = 0;
        while (bits < 32 && ((int64_t)1 << bits) <= a.first - 1) ++bits;
        e = launch_pair_keys(a.nbr_ids, nullptr, nullptr, a.M, pairs, keys, vals, st);
        if (e == cudaSuccess)
            e = radix_sort_pairs(keys, vals, keys2, vals2, pairs, bits, tmp, tmp_bytes, st, &alt, &L);
        L += 2;
    }
    const uint32_t *tgt = alt ? keys2 : keys, *order = alt ? vals2 : vals;
    if (e == cudaSuccess) {
        launch_pdl(k_new_row_ptr, dim3((unsigned)(sms * 8)), dim3(256), 0, st, rp, n_rows, a.first,
                   a.n_new, a.M, tgt, recips, new_rp);
        // old edges keep their order at the front of each row, and their weights
        // (the rows that gain edges get theirs anew below); the new rows' edges
        // go in as one block before row first's place
        launch_pdl(k_first_row, dim3(1), dim3(1), 0, st, a.first, words);
        MoveEdges mv{nnz, col, aff, w, new_col, new_aff, new_w, a.n_new * a.M, nullptr, nullptr,
                     nullptr};
        e = launch_move_edges(mv, rp, tgt, recips, words, 1, words + 1, st, &L);
    }
    if (e == cudaSuccess) {
        launch_pdl(k_fill_new_rows, dim3((unsigned)(sms * 2)), dim3(256), 0, st, a.nbr_ids,
                   a.nbr_cos, a.first, a.n_new, a.M, a.scale, new_rp, new_col, new_aff);
        if (recips > 0)
            launch_pdl(k_fill_recip, dim3((unsigned)(sms * 2)), dim3(256), 0, st, order, tgt,
                       pairs, a.nbr_cos, a.first, a.M, a.scale, rp, new_rp, new_col, new_aff);
        const int64_t want = ceil_div<int64_t>((a.n_new + recips) * 8, 256);
        const int64_t cap = (int64_t)sms * 16;
        launch_pdl(k_gained_softmax, dim3((unsigned)(want < cap ? want : cap)), dim3(256), 0, st,
                   tgt, recips, a.first, a.n_new, new_rp, new_aff, a.row_of, new_w, rstat, touched);
        e = cudaGetLastError();
    }
    if (launches) *launches += L;
    return e == cudaSuccess ? AKASHIC_OK : AKASHIC_ECUDA;
}

}  // namespace ak
