// Memory Manager on the device (arXiv 2607.05708, §4.2 and Algorithm 2):
// the page directory, co-retrieval statistics, association-driven
// relocation of retrieved chunks into fresh pages (out of place, old slots
// tombstoned) and compaction of pages whose invalid ratio reaches a
// threshold.  The paper's model calls have dense stand-ins:
//   affinity(a, b) = co(a, b) / (sel(a) + sel(b) - co(a, b)), the Jaccard
//     index of the request sets that retrieved a and b, "high association"
//     when co >= tau * (sel(a) + sel(b) - co) (fp64, tau rounded to fp32);
//   LLMCoLocate(S) = the chunks of S with a partner in S at or above tau;
//   LLMGroup(P) = connected components of those pairs within a namespace.
// A batch of requests adds its statistics first; its relocations then run
// in request order (one CTA walks the requests, 32 at a time).
#include "ak_common.cuh"

namespace ak {

constexpr unsigned long long MM_EMPTY = ~0ull;
constexpr int MM_MAX_S = 64;   // chunks per request set

// MurmurHash3's 64-bit finaliser (Appleby), spreading pair keys over the table.
__device__ __forceinline__ unsigned long long mm_mix(unsigned long long k) {
    k ^= k >> 33;
    k *= 0xff51afd7ed558ccdull;
    k ^= k >> 33;
    k *= 0xc4ceb9fe1a85ec53ull;
    k ^= k >> 33;
    return k;
}

__device__ __forceinline__ unsigned long long mm_pair(int32_t a, int32_t b) {
    const uint32_t lo = (uint32_t)(a < b ? a : b), hi = (uint32_t)(a < b ? b : a);
    return ((unsigned long long)lo << 32) | hi;
}

// co(a, b) += 1 (linear probing; a full table sets ECAPACITY)
__device__ void mm_co_add(const MmTables &t, unsigned long long key, int *status) {
    unsigned long long h = mm_mix(key) & (t.co_cap - 1);
    for (int64_t probe = 0; probe < t.co_cap; ++probe) {
        const unsigned long long prev = atomicCAS(&t.co_key[h], MM_EMPTY, key);
        if (prev == MM_EMPTY || prev == key) {
            atomicAdd(&t.co_val[h], 1u);
            if (prev == MM_EMPTY) atomicAdd(t.pairs, 1ull);
            return;
        }
        h = (h + 1) & (t.co_cap - 1);
    }
    set_status(status, AKASHIC_ECAPACITY);
}

__device__ uint32_t mm_co_get(const MmTables &t, unsigned long long key) {
    unsigned long long h = mm_mix(key) & (t.co_cap - 1);
    for (int64_t probe = 0; probe < t.co_cap; ++probe) {
        const unsigned long long k = t.co_key[h];
        if (k == key) return t.co_val[h];
        if (k == MM_EMPTY) return 0u;
        h = (h + 1) & (t.co_cap - 1);
    }
    return 0u;
}

__device__ __forceinline__ bool mm_assoc(uint32_t co, int32_t sa, int32_t sb, float tau) {
    const double uni = (double)sa + (double)sb - (double)co;
    return co > 0u && (double)co >= (double)tau * uni;
}

// Pages of per_page slots that `chunks` chunks fill (per_page up to 2^31 - 1).
__device__ __forceinline__ int mm_pages(int chunks, int per_page) {
    return (int)(((int64_t)chunks + per_page - 1) / per_page);
}

// The distinct valid chunks of request r (order of first appearance): IDs
// in [0, n), not deleted, first occurrence only.  Warp-cooperative; returns
// the count (same in every lane); set[] in shared memory.
__device__ int mm_request_set(const int64_t *__restrict__ S, int r, int s_len, int64_t n,
                              const int32_t *__restrict__ row_of,
                              const int32_t *__restrict__ dead_row, int32_t *set) {
    const int lane = threadIdx.x & 31;
    int32_t mine[2];
    bool ok[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h;
        int64_t c = i < s_len ? S[(int64_t)r * s_len + i] : -1;
        ok[h] = c >= 0 && c < n && !(dead_row && dead_row[row_of[c]]);
        mine[h] = ok[h] ? (int32_t)c : -1;
    }
    // drop repeats of an earlier position
    for (int j = 0; j < 32; ++j) {
        const int32_t o0 = __shfl_sync(0xffffffffu, mine[0], j);
        const int32_t o1 = __shfl_sync(0xffffffffu, mine[1], j);
        if (mine[0] >= 0 && j < lane && o0 == mine[0]) ok[0] = false;
        if (mine[1] >= 0 && (o0 == mine[1] || (j < lane && o1 == mine[1]))) ok[1] = false;
    }
    // compact the survivors in position order
    int count = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const unsigned m = __ballot_sync(0xffffffffu, ok[h]);
        if (ok[h]) set[count + __popc(m & ((1u << lane) - 1u))] = mine[h];
        count += __popc(m);
    }
    __syncwarp();
    return count;
}

// Statistics of a batch: one warp per request.
__global__ void k_mm_count(const int64_t *__restrict__ S, int n_req, int s_len, int64_t n,
                           const int32_t *__restrict__ row_of,
                           const int32_t *__restrict__ dead_row, MmTables t, int *status) {
    griddep_wait();
    __shared__ int32_t sets[8][MM_MAX_S];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = blockIdx.x * 8 + w; r < n_req; r += gridDim.x * 8) {
        const int cnt = mm_request_set(S, r, s_len, n, row_of, dead_row, sets[w]);
        for (int i = lane; i < cnt; i += 32) atomicAdd(&t.sel[sets[w][i]], 1);
        for (int p = lane; p < cnt * cnt; p += 32) {
            const int i = p / cnt, j = p % cnt;
            if (i < j) mm_co_add(t, mm_pair(sets[w][i], sets[w][j]), status);
        }
        __syncwarp();
    }
}

// LLMCoLocate stand-in for every request of the batch (the statistics of
// the whole batch are in place): G = the chunks of the set associated with
// some other chunk of it, their rows in chunk ID order.  One warp per request.
__global__ void k_mm_colocate(const int64_t *__restrict__ S, int n_req, int s_len, int64_t n,
                              const int32_t *__restrict__ row_of,
                              const int32_t *__restrict__ dead_row, MmTables t, float tau,
                              int32_t *__restrict__ g_out, int32_t *__restrict__ g_n) {
    griddep_wait();
    __shared__ int32_t sets[8][MM_MAX_S];
    __shared__ int flags[8][MM_MAX_S];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = blockIdx.x * 8 + w; r < n_req; r += gridDim.x * 8) {
        const int cnt = mm_request_set(S, r, s_len, n, row_of, dead_row, sets[w]);
        for (int i = lane; i < MM_MAX_S; i += 32) flags[w][i] = 0;
        __syncwarp();
        for (int p = lane; p < cnt * cnt; p += 32) {
            const int i = p / cnt, j = p % cnt;
            if (i >= j) continue;
            const int32_t a = sets[w][i], b = sets[w][j];
            if (mm_assoc(mm_co_get(t, mm_pair(a, b)), t.sel[a], t.sel[b], tau)) {
                flags[w][i] = 1;
                flags[w][j] = 1;
            }
        }
        __syncwarp();
        int ng = 0;
        for (int i = 0; i < cnt; ++i) ng += flags[w][i];
        // G in chunk ID order (SortByTime): rank by counting
        for (int i = lane; i < cnt; i += 32) {
            if (!flags[w][i]) continue;
            const int32_t a = sets[w][i];
            int rk = 0;
            for (int j = 0; j < cnt; ++j) rk += flags[w][j] && sets[w][j] < a;
            g_out[(int64_t)r * MM_MAX_S + rk] = row_of[a];
        }
        if (lane == 0) g_n[r] = ng;
        __syncwarp();
    }
}

// Relocation in request order: a G of two or more chunks not all on one page
// is written into fresh pages, old slots become invalid.  One CTA, 32 requests
// at a time, a warp each: every warp looks whether its G lies on one page; the
// requests before the first that does not are done, that one moves, and the
// ones after it look again (their chunks may just have moved).  A request that
// stays costs a 32nd of a look (one warp that took the requests in turn, a
// chain of four dependent loads each, needed ~0.9 us for every one of them:
// relocation 238 us a batch of 256, 92 so).
// result: the next fresh page, the chunks written, the pairs in the table, the
// status word.
__global__ __launch_bounds__(1024) void k_mm_relocate(const int32_t *__restrict__ g_in,
                                                      const int32_t *__restrict__ g_n, int n_req,
                                                      int32_t *page_row, MmTables t,
                                                      int64_t next_page, int per_page,
                                                      const int *status, int64_t *result) {
    griddep_wait();
    __shared__ int need[32];
    __shared__ int64_t next_s, writes_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        next_s = next_page;
        writes_s = 0;
    }
    // the next 32 requests' rows are loaded while these are looked at (slots
    // past a request's count hold what an earlier batch left there)
    int ng_n = warp < n_req ? g_n[warp] : 0;
    int32_t row_n[2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
        row_n[h] = warp < n_req ? g_in[(int64_t)warp * MM_MAX_S + lane + 32 * h] : -1;
    for (int r0 = 0; r0 < n_req; r0 += 32) {
        const int ng = ng_n, r = r0 + 32 + warp;
        int64_t row[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) row[h] = lane + 32 * h < ng ? (int64_t)row_n[h] : -1;
        ng_n = r < n_req ? g_n[r] : 0;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            row_n[h] = r < n_req ? g_in[(int64_t)r * MM_MAX_S + lane + 32 * h] : -1;
        bool done = ng < 2;
        while (true) {
            bool moves = false;
            if (!done) {
                // (pages are written by other warps: not through the L1)
                int32_t p[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) p[h] = row[h] >= 0 ? __ldcg(page_row + row[h]) : 0;
                const int32_t p0 = __shfl_sync(0xffffffffu, p[0], 0);
                moves = __any_sync(0xffffffffu, (row[0] >= 0 && p[0] != p0) ||
                                                    (row[1] >= 0 && p[1] != p0));
            }
            if (lane == 0) need[warp] = moves ? 1 : 0;
            __syncthreads();
            const unsigned nd = __ballot_sync(0xffffffffu, need[lane] != 0);
            if (nd == 0u) break;
            const int first = __ffs(nd) - 1;
            if (warp < first) done = true;
            if (warp == first) {
                done = true;
                const int64_t next = next_s;
                __syncwarp();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (row[h] < 0) continue;
                    atomicSub(&t.page_live[__ldcg(page_row + row[h])], 1);
                    const int32_t q = (int32_t)(next + (lane + 32 * h) / per_page);
                    __stcg(page_row + row[h], q);
                    atomicAdd(&t.page_total[q], 1);
                    atomicAdd(&t.page_live[q], 1);
                }
                if (lane == 0) {
                    next_s = next + mm_pages(ng, per_page);
                    writes_s += ng;
                }
            }
            __syncthreads();
        }
        __syncthreads();   // need[] is rewritten by the next 32
    }
    if (threadIdx.x == 0) {
        result[0] = next_s;
        result[1] = writes_s;
        result[2] = (int64_t)*t.pairs;
        result[3] = *status;
    }
}

// ------------------------------------------------------------------ compaction
__global__ void k_mm_candidates(MmTables t, int64_t n_pages, float theta, int32_t *__restrict__ cand) {
    griddep_wait();
    // warp-uniform trip count, so the whole warp takes part in every ballot
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n_pages;
         base += stride) {
        const int64_t p = base + (threadIdx.x & 31);
        bool c = false;
        if (p < n_pages) {
            const int32_t tot = t.page_total[p], live = t.page_live[p];
            c = tot > 0 && (double)(tot - live) >= (double)theta * (double)tot;
            cand[p] = c;
        }
        const unsigned ballot = __ballot_sync(0xffffffffu, c);
        if ((threadIdx.x & 31) == 0 && ballot) atomicAdd(t.released, (unsigned long long)__popc(ballot));
    }
}

// The live chunks on candidate pages, in ID order: ids[] and their namespaces'
// sort keys, a bitmap of them, parent[c] = c; count = how many.  The first pass
// over the directory makes the bitmap and the tiles' counts (tile_base), the
// second reads these alone.
constexpr int MM_TILE = 1024;
__global__ __launch_bounds__(256) void k_mm_moving(int64_t n, const int32_t *__restrict__ row_of,
                                                   const int32_t *__restrict__ dead_row,
                                                   const int32_t *__restrict__ page_row,
                                                   const int32_t *__restrict__ cand,
                                                   uint32_t *__restrict__ moving,
                                                   int32_t *__restrict__ counts) {
    griddep_wait();
    const int t = threadIdx.x;
    int64_t row[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t c = (int64_t)blockIdx.x * MM_TILE + q * 256 + t;
        row[q] = c < n ? row_of[c] : -1;
    }
    int mine = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t c = (int64_t)blockIdx.x * MM_TILE + q * 256 + t;
        const bool mv =
            row[q] >= 0 && cand[page_row[row[q]]] && !(dead_row && dead_row[row[q]]);
        const unsigned bal = __ballot_sync(0xffffffffu, mv);
        if ((t & 31) == 0 && c < n) moving[c >> 5] = bal;
        mine += mv ? 1 : 0;
    }
    const int own = __syncthreads_count(mine > 0) ? 1 : 0;
    // (mostly none moves: only then is there nothing to add up)
    if (own == 0) {
        if (t == 0) counts[blockIdx.x] = 0;
        return;
    }
    __shared__ int sum;
    if (t == 0) sum = 0;
    __syncthreads();
    if (mine) atomicAdd(&sum, mine);
    __syncthreads();
    if (t == 0) counts[blockIdx.x] = sum;
}

__global__ __launch_bounds__(256) void k_mm_list(int64_t n, const int32_t *__restrict__ row_of,
                                                 const int32_t *__restrict__ ns_row,
                                                 const uint32_t *__restrict__ moving,
                                                 int32_t *__restrict__ parent,
                                                 uint32_t *__restrict__ ids,
                                                 uint32_t *__restrict__ ns_key,
                                                 unsigned long long *__restrict__ count,
                                                 const int32_t *__restrict__ counts) {
    griddep_wait();
    const int t = threadIdx.x;
    const int64_t tile = blockIdx.x;
    const int own = counts[tile];
    if (own == 0 && tile != gridDim.x - 1) return;
    const int64_t base = tile_base(counts, 0, tile);
    if (t == 0 && tile == gridDim.x - 1) *count = (unsigned long long)(base + own);
    if (own == 0) return;
    unsigned bal[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t c = tile * MM_TILE + q * 256 + t;
        bal[q] = c < n ? moving[c >> 5] : 0u;
        bal[q] = __shfl_sync(0xffffffffu, bal[q], 0);   // (a warp's 32 chunks share a word)
    }
    int places[4];
    tile_places(bal, places);
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if ((bal[q] >> (t & 31)) & 1u) {
            const int64_t c = tile * MM_TILE + q * 256 + t, i = base + places[q];
            ids[i] = (uint32_t)c;
            ns_key[i] = (uint32_t)ns_row[row_of[c]] ^ 0x80000000u;   // signed order
            parent[c] = (int32_t)c;
        }
}

__device__ int32_t mm_find(volatile int32_t *parent, int32_t x) {
    for (int it = 0; it < (1 << 24); ++it) {
        const int32_t p = parent[x];
        if (p == x) return x;
        x = p;
    }
    return x;
}

// union of every associated pair of moving chunks in one namespace; roots
// hook under the smaller root, so a group's root is its earliest chunk
__global__ void k_mm_union(MmTables t, const uint32_t *__restrict__ moving,
                           const unsigned long long *__restrict__ count,
                           const int32_t *__restrict__ row_of, const int32_t *__restrict__ ns_row,
                           float tau, int32_t *__restrict__ parent, int *status) {
    griddep_wait();
    if (*count < 2) return;   // no pair of them: the table need not be looked through
    for (int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < t.co_cap;
         h += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long key = t.co_key[h];
        if (key == MM_EMPTY) continue;
        const int32_t a = (int32_t)(key >> 32), b = (int32_t)(key & 0xffffffffu);
        if (!((moving[a >> 5] >> (a & 31)) & 1u) || !((moving[b >> 5] >> (b & 31)) & 1u) ||
            ns_row[row_of[a]] != ns_row[row_of[b]])
            continue;
        if (!mm_assoc(t.co_val[h], t.sel[a], t.sel[b], tau)) continue;
        volatile int32_t *vp = parent;
        int it = 0;
        for (; it < (1 << 20); ++it) {
            const int32_t ra = mm_find(vp, a), rb = mm_find(vp, b);
            if (ra == rb) break;
            const int32_t hi = ra > rb ? ra : rb, lo = ra > rb ? rb : ra;
            if (atomicCAS(&parent[hi], hi, lo) == hi) break;
        }
        if (it == (1 << 20)) set_status(status, AKASHIC_ETIMEOUT);
    }
}

// keys for the ordered repack: (namespace, group root, chunk ID); the moving
// chunks arrive in ID order
__global__ void k_mm_roots(const uint32_t *__restrict__ ids, int64_t count,
                           const int32_t *__restrict__ parent, uint32_t *__restrict__ root_key) {
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x)
        root_key[i] = (uint32_t)mm_find((volatile int32_t *)parent, (int32_t)ids[i]);
}

__global__ void k_mm_ns_keys(const uint32_t *__restrict__ ids, int64_t count,
                             const int32_t *__restrict__ row_of,
                             const int32_t *__restrict__ ns_row, uint32_t *__restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (uint32_t)ns_row[row_of[ids[i]]] ^ 0x80000000u;
}

// The whole repack of at most MM_SMALL chunks by one CTA: their order
// (namespace, group root, chunk ID), the pages of each namespace's run (every
// namespace starts on a fresh page), the chunks written there.  new_pages: the
// pages used.  (Sorts, page counts, a scan and the writes took 15 launches and
// a read-back for the few dozen chunks that a compaction mostly moves.)
constexpr int MM_SMALL = 2048;
__global__ __launch_bounds__(1024) void k_mm_repack_small(const uint32_t *__restrict__ ids,
                                                          const uint32_t *__restrict__ ns_key,
                                                          int count,
                                                          const int32_t *__restrict__ parent,
                                                          const int32_t *__restrict__ row_of,
                                                          int32_t *__restrict__ page_row,
                                                          MmTables t, int64_t first_page,
                                                          int per_page, int64_t *new_pages) {
    griddep_wait();
    __shared__ unsigned long long key[MM_SMALL];   // (namespace, root)
    __shared__ uint16_t at[MM_SMALL];              // place in ids
    __shared__ int32_t run_page[MM_SMALL];         // at a run's head: its first page
    __shared__ int wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int size = 32;
    while (size < count) size <<= 1;
    for (int i = tid; i < size; i += 1024) {
        key[i] = i < count ? ((unsigned long long)ns_key[i] << 32) |
                                 (uint32_t)mm_find((volatile int32_t *)parent, (int32_t)ids[i])
                           : ~0ull;
        at[i] = (uint16_t)i;
    }
    __syncthreads();
    // ascending by (key, place): places are in chunk ID order; absent ones last
    for (int sz = 2; sz <= size; sz <<= 1)
        for (int stride = sz >> 1; stride > 0; stride >>= 1) {
            for (int i = tid; i < size; i += 1024) {
                const int o = i ^ stride;
                if (o > i) {
                    const unsigned long long a = key[i], b = key[o];
                    const uint16_t pa = at[i], pb = at[o];
                    const bool gt = a > b || (a == b && pa > pb);
                    if (gt == ((i & sz) == 0)) {
                        key[i] = b;
                        key[o] = a;
                        at[i] = pb;
                        at[o] = pa;
                    }
                }
            }
            __syncthreads();
        }
    // runs of equal namespaces: two places a thread, 0 .. 2047
    int head[2], len[2] = {0, 0}, pages = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = 2 * tid + h;
        head[h] = i < count && (i == 0 || (key[i] >> 32) != (key[i - 1] >> 32));
        if (head[h]) {
            // the run's end: first place with a larger namespace
            int lo = i + 1, hi = count;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if ((key[mid] >> 32) > (key[i] >> 32)) hi = mid;
                else lo = mid + 1;
            }
            len[h] = lo - i;
        }
        pages += mm_pages(len[h], per_page);
    }
    // base pages: exclusive scan of the runs' pages over the threads
    int incl = pages;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int base = incl - pages;
    for (int w = 0; w < warp; ++w) base += wsum[w];
    if (tid == 1023) *new_pages = base + pages;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (head[h]) run_page[2 * tid + h] = base;
        base += mm_pages(len[h], per_page);
    }
    __syncthreads();
    // place i: its run's head is the first place with its namespace
    for (int i = tid; i < count; i += 1024) {
        int lo = 0, hi = i;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((key[mid] >> 32) < (key[i] >> 32)) lo = mid + 1;
            else hi = mid;
        }
        const int32_t p = (int32_t)(first_page + run_page[lo] + (i - lo) / per_page);
        page_row[row_of[ids[at[i]]]] = p;
        atomicAdd(&t.page_total[p], 1);
        atomicAdd(&t.page_live[p], 1);
    }
}

cudaError_t launch_mm_ns_keys(const uint32_t *ids, int64_t count, const int32_t *row_of,
                              const int32_t *ns_row, uint32_t *out, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    k_mm_ns_keys<<<device_sm_count() * 2, 256, 0, st>>>(ids, count, row_of, ns_row, out);
    return cudaGetLastError();
}

__global__ void k_mm_release(MmTables t, int64_t n_pages, const int32_t *__restrict__ cand) {
    griddep_wait();
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n_pages;
         p += (int64_t)gridDim.x * blockDim.x)
        if (cand[p]) {
            t.page_total[p] = 0;
            t.page_live[p] = 0;
        }
}

// Every namespace (partition) starts on a fresh page: at the first
// position of each run of equal namespace keys, the pages that run fills
// (ceil(run / P)); zero elsewhere.  An exclusive scan of these gives each
// partition's first page relative to the first fresh page.
__global__ void k_mm_part_pages(const uint32_t *__restrict__ ns_sorted, int64_t count,
                                int per_page, int64_t *__restrict__ part_pages) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = ns_sorted[i];
        int64_t v = 0;
        if (i == 0 || ns_sorted[i - 1] != k) {
            const int64_t end = lower_bound_u32(ns_sorted, count, (uint64_t)k + 1);
            v = (end - i + per_page - 1) / per_page;
        }
        part_pages[i] = v;
    }
}

cudaError_t launch_mm_part_pages(const uint32_t *ns_sorted, int64_t count, int per_page,
                                 int64_t *part_pages, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    k_mm_part_pages<<<device_sm_count() * 2, 256, 0, st>>>(ns_sorted, count, per_page, part_pages);
    return cudaGetLastError();
}

// chunk i of the ordered list: page = first page + its partition's base
// page + (offset inside the partition) / P
__global__ void k_mm_repack(const uint32_t *__restrict__ order_ids,
                            const uint32_t *__restrict__ ns_sorted,
                            const int64_t *__restrict__ part_base, int64_t count,
                            const int32_t *__restrict__ row_of, int32_t *__restrict__ page_row,
                            MmTables t, int64_t first_page, int per_page) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = lower_bound_u32(ns_sorted, count, ns_sorted[i]);
        const int32_t p = (int32_t)(first_page + part_base[s] + (i - s) / per_page);
        page_row[row_of[order_ids[i]]] = p;
        atomicAdd(&t.page_total[p], 1);
        atomicAdd(&t.page_live[p], 1);
    }
}

// ------------------------------------------------------------------ bookkeeping
// new rows [first, first+n): their pages gain a live slot each
__global__ void k_mm_count_pages(const int32_t *__restrict__ page_row, int64_t first, int64_t n,
                                 MmTables t) {
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = page_row[first + i];
        atomicAdd(&t.page_total[p], 1);
        atomicAdd(&t.page_live[p], 1);
    }
}

__global__ void k_mm_stats(MmTables t, int64_t n_pages, unsigned long long *__restrict__ out) {
    unsigned long long in_use = 0, tot = 0, live = 0;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n_pages;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = t.page_total[p];
        in_use += a > 0;
        tot += (unsigned long long)(a > 0 ? a : 0);
        live += (unsigned long long)(a > 0 ? t.page_live[p] : 0);
    }
    for (int o = 16; o > 0; o >>= 1) {
        in_use += __shfl_xor_sync(0xffffffffu, in_use, o);
        tot += __shfl_xor_sync(0xffffffffu, tot, o);
        live += __shfl_xor_sync(0xffffffffu, live, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&out[0], in_use);
        atomicAdd(&out[1], tot);
        atomicAdd(&out[2], live);
    }
}

__global__ void k_mm_rehash(const unsigned long long *__restrict__ old_key,
                            const uint32_t *__restrict__ old_val, int64_t old_cap, MmTables t,
                            int *status) {
    for (int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < old_cap;
         h += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long key = old_key[h];
        if (key == MM_EMPTY) continue;
        unsigned long long j = mm_mix(key) & (t.co_cap - 1);
        int64_t probe = 0;
        for (; probe < t.co_cap; ++probe) {
            if (atomicCAS(&t.co_key[j], MM_EMPTY, key) == MM_EMPTY) {
                t.co_val[j] = old_val[h];
                break;
            }
            j = (j + 1) & (t.co_cap - 1);
        }
        if (probe == t.co_cap) set_status(status, AKASHIC_ECAPACITY);
    }
}

__global__ void k_by_id(const int32_t *__restrict__ by_row, const int32_t *__restrict__ row_of,
                        int64_t n, int32_t *__restrict__ out) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n;
         c += (int64_t)gridDim.x * blockDim.x)
        out[c] = by_row[row_of[c]];
}

// ------------------------------------------------------------------ launchers
cudaError_t launch_mm_count(const int64_t *S, int n_req, int s_len, int64_t n,
                            const int32_t *row_of, const int32_t *dead_row, const MmTables &t,
                            int *status, cudaStream_t st) {
    if (n_req <= 0) return cudaSuccess;
    const int grid = (int)ceil_div<int64_t>(n_req, 8);
    launch_pdl(k_mm_count,
               dim3((unsigned)(grid < device_sm_count() * 8 ? grid : device_sm_count() * 8)),
               dim3(256), 0, st, S, n_req, s_len, n, row_of, dead_row, t, status);
    return cudaGetLastError();
}

cudaError_t launch_mm_relocate(const int64_t *S, int n_req, int s_len, int64_t n,
                               const int32_t *row_of, const int32_t *dead_row, int32_t *page_row,
                               const MmTables &t, float tau, int64_t next_page, int per_page,
                               int32_t *g_buf, int32_t *g_n, const int *status, int64_t *result,
                               cudaStream_t st) {
    if (n_req <= 0) return cudaSuccess;
    const int grid = (int)ceil_div<int64_t>(n_req, 8);
    launch_pdl(k_mm_colocate,
               dim3((unsigned)(grid < device_sm_count() * 8 ? grid : device_sm_count() * 8)),
               dim3(256), 0, st, S, n_req, s_len, n, row_of, dead_row, t, tau, g_buf, g_n);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    launch_pdl(k_mm_relocate, dim3(1), dim3(1024), 0, st, g_buf, g_n, n_req, page_row, t,
               next_page, per_page, status, result);
    return cudaGetLastError();
}

cudaError_t launch_mm_candidates(const MmTables &t, int64_t n_pages, float theta, int32_t *cand,
                                 cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(t.released, 0, 8, st);
    if (e != cudaSuccess || n_pages <= 0) return e;
    const int64_t want = ceil_div<int64_t>(n_pages, 256), cap = (int64_t)device_sm_count() * 2;
    launch_pdl(k_mm_candidates, dim3((unsigned)(want < cap ? want : cap)), dim3(256), 0, st, t,
               n_pages, theta, cand);
    return cudaGetLastError();
}

static int64_t mm_tiles(int64_t n) { return ceil_div<int64_t>(n, MM_TILE); }
int64_t mm_words(int64_t n) { return tile_words(mm_tiles(n)); }

cudaError_t launch_mm_collect(const MmTables &t, int64_t n, const int32_t *row_of,
                              const int32_t *dead_row, const int32_t *page_row,
                              const int32_t *ns_row, const int32_t *cand, uint32_t *moving,
                              int32_t *parent, uint32_t *ids, uint32_t *ns_key, int32_t *counts,
                              cudaStream_t st) {
    if (n <= 0) return cudaErrorInvalidValue;
    const unsigned tiles = (unsigned)mm_tiles(n);
    launch_pdl(k_mm_moving, dim3(tiles), dim3(256), 0, st, n, row_of, dead_row, page_row, cand,
               moving, counts);
    cudaError_t e = launch_tile_groups(counts, tiles, st);
    if (e != cudaSuccess) return e;
    launch_pdl(k_mm_list, dim3(tiles), dim3(256), 0, st, n, row_of, ns_row, moving, parent, ids,
               ns_key, t.released + 1, counts);
    return cudaGetLastError();
}

cudaError_t launch_mm_union(const MmTables &t, const uint32_t *moving, const int32_t *row_of,
                            const int32_t *ns_row, float tau, int32_t *parent, int *status,
                            cudaStream_t st) {
    launch_pdl(k_mm_union, dim3((unsigned)(device_sm_count() * 8)), dim3(256), 0, st, t, moving,
               t.released + 1, row_of, ns_row, tau, parent, status);
    return cudaGetLastError();
}

cudaError_t launch_mm_roots(const uint32_t *ids, int64_t count, const int32_t *parent,
                            uint32_t *root_key, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    launch_pdl(k_mm_roots, dim3((unsigned)(device_sm_count() * 2)), dim3(256), 0, st, ids, count,
               parent, root_key);
    return cudaGetLastError();
}

int mm_small_repack() { return MM_SMALL; }
cudaError_t launch_mm_repack_small(const MmTables &t, int64_t n_pages, const int32_t *cand,
                                   const uint32_t *ids, const uint32_t *ns_key, int64_t count,
                                   const int32_t *parent, const int32_t *row_of,
                                   int32_t *page_row, int64_t first_page, int per_page,
                                   int64_t *new_pages, cudaStream_t st) {
    if (count < 1 || count > MM_SMALL) return cudaErrorInvalidValue;
    if (n_pages > 0) launch_pdl(k_mm_release, dim3((unsigned)(device_sm_count() * 2)), dim3(256),
                                0, st, t, n_pages, cand);
    launch_pdl(k_mm_repack_small, dim3(1), dim3(1024), 0, st, ids, ns_key, (int)count, parent,
               row_of, page_row, t, first_page, per_page, new_pages);
    return cudaGetLastError();
}

cudaError_t launch_mm_release_repack(const MmTables &t, int64_t n_pages, const int32_t *cand,
                                     const uint32_t *order_ids, const uint32_t *ns_sorted,
                                     const int64_t *part_base, int64_t count,
                                     const int32_t *row_of, int32_t *page_row, int64_t first_page,
                                     int per_page, cudaStream_t st) {
    const int sms = device_sm_count();
    if (n_pages > 0) launch_pdl(k_mm_release, dim3((unsigned)(sms * 2)), dim3(256), 0, st, t,
                                n_pages, cand);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || count <= 0) return e;
    k_mm_repack<<<sms * 2, 256, 0, st>>>(order_ids, ns_sorted, part_base, count, row_of, page_row,
                                         t, first_page, per_page);
    return cudaGetLastError();
}

cudaError_t launch_mm_count_pages(const int32_t *page_row, int64_t first, int64_t n,
                                  const MmTables &t, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    launch_pdl(k_mm_count_pages, dim3((unsigned)(device_sm_count() * 2)), dim3(256), 0, st,
               page_row, first, n, t);
    return cudaGetLastError();
}

cudaError_t launch_mm_stats(const MmTables &t, int64_t n_pages, unsigned long long *out,
                            cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(out, 0, 3 * sizeof(unsigned long long), st);
    if (e != cudaSuccess || n_pages <= 0) return e;
    k_mm_stats<<<device_sm_count() * 2, 256, 0, st>>>(t, n_pages, out);
    return cudaGetLastError();
}

cudaError_t launch_mm_rehash(const unsigned long long *old_key, const uint32_t *old_val,
                             int64_t old_cap, const MmTables &t, int *status, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(t.co_key, 0xff, (size_t)t.co_cap * 8, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(t.co_val, 0, (size_t)t.co_cap * 4, st);
    if (e != cudaSuccess || old_cap <= 0) return e;
    k_mm_rehash<<<device_sm_count() * 8, 256, 0, st>>>(old_key, old_val, old_cap, t, status);
    return cudaGetLastError();
}

cudaError_t launch_by_id(const int32_t *by_row, const int32_t *row_of, int64_t n, int32_t *out,
                         cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_by_id<<<device_sm_count() * 2, 256, 0, st>>>(by_row, row_of, n, out);
    return cudaGetLastError();
}

}  // namespace ak
