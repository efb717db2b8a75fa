// The C ABI declared in include/akashic_mem.h: store lifecycle, appends,
// relation-graph maintenance, retrieval orchestration, read-back, status and
// phase timing.  All arithmetic runs in the kernels of the other files.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <string>
#include <unordered_map>
#include <vector>

#include "ak_common.cuh"
#include "ak_update.cuh"

using namespace ak;

// ------------------------------------------------------------------ errors
static thread_local std::string g_last_error;

void ak::set_last_error(const char *msg) { g_last_error = msg ? msg : ""; }

static akashic_status_t fail(akashic_status_t st, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_last_error = buf;
    return st;
}

#define CUDA_TRY(call)                                                                         \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess)                                                                 \
            return fail(e_ == cudaErrorMemoryAllocation ? AKASHIC_ENOMEM : AKASHIC_ECUDA,      \
                        "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__);  \
    } while (0)

#define AK_TRY(call)                                                                           \
    do {                                                                                       \
        akashic_status_t s_ = (call);                                                          \
        if (s_ != AKASHIC_OK) return s_;                                                       \
    } while (0)

// ------------------------------------------------------------------ device buffers
// The store whose reach tables an allocation of this thread may have freed when
// the device has no room for it (Reclaim; release_tables frees them, if it can).
static thread_local akashic_mem *g_reclaim = nullptr;
static bool release_tables(akashic_mem *m);
struct Reclaim {
    akashic_mem *prev = g_reclaim;
    explicit Reclaim(akashic_mem *m) { g_reclaim = m; }
    ~Reclaim() { g_reclaim = prev; }
};

struct DevBuf {
    void *p = nullptr;
    size_t cap = 0;
    ~DevBuf() { release(); }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        cap = 0;
    }
    // Grow to at least `bytes`; contents are not preserved unless keep.
    akashic_status_t ensure(size_t bytes, bool keep = false, cudaStream_t st = 0) {
        if (bytes <= cap) return AKASHIC_OK;
        size_t want = bytes < 256 ? 256 : bytes;
        void *q = nullptr;
        cudaError_t e = cudaMalloc(&q, want);
        if (e == cudaErrorMemoryAllocation && g_reclaim) {
            cudaGetLastError();
            if (release_tables(g_reclaim)) e = cudaMalloc(&q, want);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(AKASHIC_ENOMEM, "device allocation of %zu bytes failed", want);
        }
        if (keep && p && cap) {
            e = cudaMemcpyAsync(q, p, cap, cudaMemcpyDeviceToDevice, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) {
                cudaFree(q);
                return fail(AKASHIC_ECUDA, "buffer growth copy: %s", cudaGetErrorString(e));
            }
        }
        if (p) cudaFree(p);
        p = q;
        cap = want;
        return AKASHIC_OK;
    }
    template <typename T> T *as() const { return (T *)p; }
};

static void swap_bufs(DevBuf &x, DevBuf &y) {
    std::swap(x.p, y.p);
    std::swap(x.cap, y.cap);
}

// Words of StreamScratch::words: u's extremes [2], the kept lists' lengths
// (int64 [2]), whether this call skips the candidates (away from the flags' counters,
// which every CTA of k_reach_flags adds to: 1.2 us a call beside them), the hops'
// work queues ([2] a hop), the candidates' flags.
constexpr int CW_EXT = 0, CW_KEPT = 2, CW_SKIP = 6, CW_QUEUE = 8,
              CW_REACH = CW_QUEUE + 2 * AKASHIC_MAX_HOPS, CW_COUNT = CW_REACH + REACH_WS;

struct StreamScratch {
    DevBuf qp, shift, u, sa, sb, zpart, partial, cand;
    DevBuf words;                // a call's counters (CW_*), zeroed by its first kernel
    DevBuf samp, ext_s, zsamp;   // retrieval without hops: the score's row sample
    DevBuf qns, ns_s, dead_s;    // scope: per query column, per sample row
    DevBuf rmax_u, rmin_u;       // u's row maxima / minima over the real queries
    DevBuf pfloor;               // the last hop's floor and what it keeps
    DevBuf skip_split, kept_rows, kept_segs, keep_scr;
    DevBuf reach_part, reach_plan;   // the candidates' partials, the plan
    DevBuf nsf;                  // scoped last hop: tags, their floors, their count
    // every candidate's combined coefficients (bf16 hi, lo), and their key
    DevBuf coef_hi, coef_lo, coef_sum;
    uint64_t coef_build = ~0ull;
    float coef_alpha = -1.f;
    int coef_H = 0;
    int64_t coef_n = -1;
    // the call's plan read back: pinned host words and the event after
    // their copy (the host waits for that point only)
    int32_t *plan_host = nullptr;
    cudaEvent_t plan_ev = nullptr;
    // the fp32 pass: the combined coefficients and their key
    DevBuf coef_f, cf_sum;
    int64_t no_room_n = -1, no_room_sync_n = -1;   // rows at which the tables did not fit
    uint64_t cf_build = ~0ull;
    float cf_alpha = -1.f;
    int cf_H = 0;
    int64_t cf_n = -1;
    // the calls that could use the candidates, by key (try_skips): a key's number
    // and theirs; its mark on the device and the copy the host sees
    struct TryKey {
        uint64_t build = ~0ull, used = 0;
        int64_t n = -1;
        float alpha = -1.f;
        int H = 0, k = 0, mode = 0;
        uint32_t number = 0, calls = 0;
    };
    static constexpr int TRY_KEYS = 8;
    TryKey keys[TRY_KEYS];
    uint32_t key_numbers = 0;
    uint64_t key_uses = 0;
    DevBuf tried;                // [TRY_KEYS]
    unsigned long long *told = nullptr;
    TryKey &try_key(uint64_t build, int64_t n, float alpha, int H, int k, int mode) {
        TryKey *at = keys;
        for (TryKey &t : keys) {
            if (t.build == build && t.n == n && t.alpha == alpha && t.H == H && t.k == k &&
                t.mode == mode && t.calls < (1u << 30)) {
                t.used = ++key_uses;
                return t;
            }
            if (t.used < at->used) at = &t;
        }
        *at = TryKey{build, ++key_uses, n, alpha, H, k, mode, ++key_numbers, 0};
        return *at;
    }
    ~StreamScratch() {
        if (plan_host) cudaFreeHost(plan_host);
        if (plan_ev) cudaEventDestroy(plan_ev);
    }
};

struct ProfRec {
    int phase;
    cudaEvent_t a, b;
    int launches;
};

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

struct akashic_mem {
    int device = 0;
    int dim = 0;
    int64_t cap = 0;
    int per_page = 1;
    float tau = 0.f;
    float rel_scale = 10.f;
    int64_t n = 0;
    int64_t next_page = 0;
    // chunks live in HBM in page order: row r holds chunk ext_of[r], chunk c
    // is in row row_of[c]; page_of is indexed by row
    DevBuf emb, page_of, ext_of, row_of, max_norm, status;
    DevBuf ns_row;               // namespace tag of the chunk in each row (0 by default)
    DevBuf dead_row;             // 1 in the rows of deleted chunks
    bool has_dead = false;       // any chunk deleted (enables the masks)
    // memory manager: per-page slot counters, co-retrieval statistics
    DevBuf page_total, page_live, sel, co_key, co_val, mm_ctr;
    int64_t page_cap = 0, co_cap = 0, co_pairs = 0;
    int64_t appended = 0, moves = 0;
    // canonical out-edge CSR
    int64_t nnz = 0;
    DevBuf row_ptr, col, aff, w;
    // in-edge transpose + split plan for the propagation hop
    DevBuf in_ptr, in_src, in_w, in_aff;
    DevBuf rstat;                // per chunk ID: (max, 1/sum) of its out-row softmax
    // spares the relation update writes the next CSR / transpose into (then
    // swapped with the live arrays), and grow-only scratch for its temporaries
    DevBuf rp2, col2, aff2, w2, in_ptr2, in_src2, in_aff2, in_w2;
    DevBuf scr[SCR_COUNT];
    bool inc_transpose = true;   // relation updates patch the transpose instead of re-sorting
    SplitParams split;
    bool fuse_filter = true;     // top-k filter in the last hop's epilogue
    bool hop_prune = true;       // last hop skips rows bounded below every filter threshold
    int64_t n_split = 0, n_segs = 0;
    DevBuf split_row, split_slot0, seg_e0, seg_e1, seg_slot, split_order, slot_split;
    // graph-only mass vectors of the last hop's row bounds, levels 0..mass_levels
    // (recomputed lazily after the graph changes)
    DevBuf mass_up, mass_dn, mass_zero, mass_vu, mass_vl;
    int mass_levels = -1;
    int64_t mass_n = -1;      // rows they were computed for
    // reach coefficients of the candidate rows (ak_reach.cu), same lifetime
    DevBuf reach_rows, reach_t, reach_map, reach_pick, reach_c[REACH_MAX_H];
    int reach_levels = -1;    // levels C_1.. in place (0 or less: no candidates either)
    int64_t reach_n = -1;     // rows they were computed for
    double hop_work = 0;      // query columns x hops run through the hops since the
    int64_t hop_work_n = -1;  // graph (or the number of rows) last changed
    // what the tables of this graph had to save to pay (0: none built for small
    // batches), what they have saved (in the same unit), and how many times that
    // cost the hops have to reach before tables are built (table_turn)
    double table_cost = 0, table_saved = 0, table_wait = 1;
    uint64_t reach_build = 0; // incremented by every rebuild
    bool reach_on = true;     // AKASHIC_REACH=0: always run the hops
    std::atomic<int> table_users{0};   // calls between taking the tables (table_mu) and
                                       // having queued all that reads them
    // the mass levels and reach tables are built by whichever retrieve needs
    // them first, on its own stream: table_mu serialises the builders and
    // every retrieve that reads them waits on table_ev, recorded after the
    // last build (retrieves on other streams may run concurrently)
    std::mutex table_mu;
    cudaEvent_t table_ev = nullptr;
    std::mutex mu;
    std::unordered_map<void *, StreamScratch *> scratch;
    // profiling
    bool prof = false;
    std::vector<ProfRec> recs;
    std::vector<cudaEvent_t> ev_pool;
    ~akashic_mem() {
        for (auto &kv : scratch) delete kv.second;
        for (auto &r : recs) {
            cudaEventDestroy(r.a);
            cudaEventDestroy(r.b);
        }
        for (auto e : ev_pool) cudaEventDestroy(e);
        if (table_ev) cudaEventDestroy(table_ev);
    }
};

// ------------------------------------------------------------------ profiling helpers
struct PhaseScope {
    akashic_mem *m;
    int phase;
    cudaStream_t st;
    cudaEvent_t a = nullptr;
    int launches = 0;
    PhaseScope(akashic_mem *m_, int ph, cudaStream_t s) : m(m_), phase(ph), st(s) {
        if (!m->prof) return;
        a = take_event();
        if (a) cudaEventRecord(a, st);
    }
    cudaEvent_t take_event() {
        std::lock_guard<std::mutex> g(m->mu);
        cudaEvent_t e = nullptr;
        if (!m->ev_pool.empty()) {
            e = m->ev_pool.back();
            m->ev_pool.pop_back();
        } else if (cudaEventCreate(&e) != cudaSuccess) {
            cudaGetLastError();
            e = nullptr;
        }
        return e;
    }
    // close the scope early (once); the destructor then does nothing
    void end() {
        if (!m->prof || !a) return;
        cudaEvent_t b = take_event();
        if (b) {
            cudaEventRecord(b, st);
            std::lock_guard<std::mutex> g(m->mu);
            m->recs.push_back(ProfRec{phase, a, b, launches});
        }
        a = nullptr;
    }
    ~PhaseScope() {
        if (!m->prof || !a) return;
        cudaEvent_t b = take_event();
        if (!b) return;
        cudaEventRecord(b, st);
        std::lock_guard<std::mutex> g(m->mu);
        m->recs.push_back(ProfRec{phase, a, b, launches});
    }
};

// ------------------------------------------------------------------ small kernels
__global__ void k_page_max(const int32_t *page_of, int64_t n, int *out_max, int *status) {
    int best = -1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int p = page_of[i];
        if (p < 0) set_status(status, AKASHIC_EDEVICE);
        best = p > best ? p : best;
    }
    atomicMax(out_max, best);
}

// row_ptr of the appended rows in the store's CSR: dst[r] = base + src[r] - src[0]
__global__ void k_rebase_ptr(const int64_t *src, int64_t *dst, int64_t n1, int64_t base) {
    const int64_t p0 = src ? src[0] : 0;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n1;
         r += (int64_t)gridDim.x * blockDim.x)
        dst[r] = src ? base + src[r] - p0 : base;
}

static int bits_for(int64_t max_value) {
    int b = 0;
    while (b < 32 && ((int64_t)1 << b) <= max_value) ++b;
    return b;
}

static akashic_status_t check_status(akashic_mem *m, cudaStream_t st, const char *what) {
    int code = 0;
    CUDA_TRY(cudaMemcpyAsync(&code, m->status.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    if (code != 0) {
        CUDA_TRY(cudaMemset(m->status.p, 0, sizeof(int)));
        return fail((akashic_status_t)code, "%s: device reported status %d", what, code);
    }
    return AKASHIC_OK;
}

// Grow-only scratch of a store (UpdateArgs::scratch): 1/8 headroom when a
// slot has to grow, so slowly growing sizes do not reallocate every call.
static void *store_scratch(void *ctx, int slot, size_t bytes) {
    akashic_mem *m = (akashic_mem *)ctx;
    if (slot < 0 || slot >= SCR_COUNT) return nullptr;
    DevBuf &b = m->scr[slot];
    if (bytes > b.cap && b.ensure(bytes + bytes / 8) != AKASHIC_OK) return nullptr;
    return b.p;
}

static MmTables mm_tables(akashic_mem *m) {
    MmTables t;
    t.page_total = m->page_total.as<int32_t>();
    t.page_live = m->page_live.as<int32_t>();
    t.sel = m->sel.as<int32_t>();
    t.co_key = m->co_key.as<unsigned long long>();
    t.co_val = m->co_val.as<uint32_t>();
    t.co_cap = m->co_cap;
    t.pairs = m->mm_ctr.as<unsigned long long>();
    t.released = m->mm_ctr.as<unsigned long long>() + 1;
    return t;
}

// Page counters for page IDs below `need` (grown by doubling, new tail zeroed).
static akashic_status_t mm_ensure_pages(akashic_mem *m, int64_t need, cudaStream_t st) {
    if (need <= m->page_cap) return AKASHIC_OK;
    int64_t cap = m->page_cap > 0 ? m->page_cap : 1024;
    while (cap < need) cap *= 2;
    AK_TRY(m->page_total.ensure((size_t)cap * 4, true, st));
    AK_TRY(m->page_live.ensure((size_t)cap * 4, true, st));
    CUDA_TRY(cudaMemsetAsync(m->page_total.as<int32_t>() + m->page_cap, 0,
                             (size_t)(cap - m->page_cap) * 4, st));
    CUDA_TRY(cudaMemsetAsync(m->page_live.as<int32_t>() + m->page_cap, 0,
                             (size_t)(cap - m->page_cap) * 4, st));
    m->page_cap = cap;
    return AKASHIC_OK;
}

// Co-retrieval table able to take `more` new pairs at load <= 1/2.
static akashic_status_t mm_ensure_pairs(akashic_mem *m, int64_t more, cudaStream_t st,
                                        int *launches = nullptr) {
    if (m->co_cap > 0 && m->co_pairs + more <= m->co_cap / 2) return AKASHIC_OK;
    int64_t cap = m->co_cap > 0 ? m->co_cap : ((int64_t)1 << 20);
    while (m->co_pairs + more > cap / 2) cap *= 2;
    DevBuf nk, nv;
    AK_TRY(nk.ensure((size_t)cap * 8));
    AK_TRY(nv.ensure((size_t)cap * 4));
    swap_bufs(m->co_key, nk);
    swap_bufs(m->co_val, nv);
    const int64_t old_cap = m->co_cap;
    m->co_cap = cap;
    CUDA_TRY(launch_mm_rehash(nk.as<unsigned long long>(), nv.as<uint32_t>(), old_cap,
                              mm_tables(m), m->status.as<int>(), st));
    if (launches && old_cap > 0) *launches += 1;
    CUDA_TRY(cudaStreamSynchronize(st));   // the old table is freed on return
    return AKASHIC_OK;
}

// A scratch buffer seen through the DevBuf-like accessors.
struct Tmp {
    void *p;
    size_t cap;
    template <typename T> T *as() const { return (T *)p; }
};

// Grow a spare buffer with 1/4 headroom (contents not kept).
static akashic_status_t ensure_spare(DevBuf &b, size_t bytes) {
    return bytes > b.cap ? b.ensure(bytes + bytes / 4) : AKASHIC_OK;
}

// The reach tables of the store and of its streams, freed unless a call is using
// them (cudaFree waits for the kernels that do); none is built again for this many
// rows.  True if there was something to free.  table_mu held.
static bool release_tables_locked(akashic_mem *m) {
    if (m->table_users.load() != 0) return false;
    size_t freed = 0;
    auto drop = [&](DevBuf &b) {
        freed += b.cap;
        b.release();
    };
    for (DevBuf &b : m->reach_c) drop(b);
    drop(m->reach_map);
    m->reach_levels = -1;
    std::lock_guard<std::mutex> lk(m->mu);
    for (auto &kv : m->scratch) {
        StreamScratch *sc = kv.second;
        for (DevBuf *b : {&sc->coef_hi, &sc->coef_lo, &sc->coef_sum, &sc->coef_f, &sc->cf_sum,
                          &sc->reach_part})
            drop(*b);
        sc->coef_build = sc->cf_build = ~0ull;
        sc->no_room_n = m->n;
    }
    return freed > 0;
}
static bool release_tables(akashic_mem *m) {
    std::lock_guard<std::mutex> lk(m->table_mu);
    return release_tables_locked(m);
}

// The graph, or the number of rows, has changed: the work done on it starts over.
// Where its tables had not saved what they cost, the next ones are built after twice
// as much work (16 times at most), else after the least again.
static void table_turn(akashic_mem *m) {
    if (m->table_cost > 0) {
        const bool paid = m->table_saved >= m->table_cost;
        m->table_wait = paid ? 1 : (m->table_wait < 16 ? 2 * m->table_wait : 16);
    }
    m->table_cost = m->table_saved = m->hop_work = 0;
}

// Rows that a table is sized for when it grows: a quarter more, to the capacity.
static int64_t table_rows(const akashic_mem *m) {
    const int64_t room = m->n + m->n / 4;
    return room < m->cap ? room : m->cap;
}

static akashic_status_t ensure_table(DevBuf &b, size_t now, size_t grown) {
    return now > b.cap ? b.ensure(grown) : AKASHIC_OK;
}

static akashic_status_t build_split_plan(akashic_mem *m, cudaStream_t st);

// Rebuild the in-edge transpose (stable by source, hence sorted by source
// within each destination), its weights, and the split plan of long rows.
static akashic_status_t rebuild_in_edges(akashic_mem *m, cudaStream_t st) {
    const int64_t n = m->n, nnz = m->nnz;
    AK_TRY(m->in_ptr.ensure((size_t)(m->cap + 1) * sizeof(int64_t)));
    AK_TRY(m->in_src.ensure((size_t)(nnz > 0 ? nnz : 1) * sizeof(int32_t)));
    AK_TRY(m->in_w.ensure((size_t)(nnz > 0 ? nnz : 1) * sizeof(float)));
    AK_TRY(m->in_aff.ensure((size_t)(nnz > 0 ? nnz : 1) * sizeof(float)));
    DevBuf src, keys, vals, keys2, vals2, tmp, deg;
    const size_t tmp_bytes = (radix_tmp_bytes(nnz) > scan_tmp_bytes(n + 1) ? radix_tmp_bytes(nnz)
                                                                             : scan_tmp_bytes(n + 1)) +
                             4096;
    AK_TRY(tmp.ensure(tmp_bytes));
    AK_TRY(deg.ensure((size_t)(n + 1) * sizeof(int64_t) * 2));
    if (nnz > 0) {
        AK_TRY(src.ensure((size_t)nnz * 4));
        AK_TRY(keys.ensure((size_t)nnz * 4));
        AK_TRY(vals.ensure((size_t)nnz * 4));
        AK_TRY(keys2.ensure((size_t)nnz * 4));
        AK_TRY(vals2.ensure((size_t)nnz * 4));
        const int32_t *row_of = m->row_of.as<int32_t>();
        CUDA_TRY(launch_edge_src_check(m->row_ptr.as<int64_t>(), m->col.as<int32_t>(), n, 0, n,
                                       src.as<int32_t>(), m->status.as<int>(), st));
        // edges ordered by (target row, source row): sort by source row, then
        // stably by target row
        CUDA_TRY(launch_map_keys(nullptr, src.as<int32_t>(), row_of, keys.as<uint32_t>(), nnz, st));
        CUDA_TRY(launch_iota(vals.as<uint32_t>(), nnz, st));
        bool alt = false;
        CUDA_TRY(radix_sort_pairs(keys.as<uint32_t>(), vals.as<uint32_t>(), keys2.as<uint32_t>(),
                                  vals2.as<uint32_t>(), nnz, bits_for(n - 1), tmp.p, tmp.cap, st,
                                  &alt));
        uint32_t *k1 = alt ? keys2.as<uint32_t>() : keys.as<uint32_t>();
        uint32_t *v1 = alt ? vals2.as<uint32_t>() : vals.as<uint32_t>();
        uint32_t *k2 = alt ? keys.as<uint32_t>() : keys2.as<uint32_t>();
        uint32_t *v2 = alt ? vals.as<uint32_t>() : vals2.as<uint32_t>();
        CUDA_TRY(launch_map_keys(v1, m->col.as<int32_t>(), row_of, k1, nnz, st));
        bool alt2 = false;
        CUDA_TRY(radix_sort_pairs(k1, v1, k2, v2, nnz, bits_for(n - 1), tmp.p, tmp.cap, st, &alt2));
        const uint32_t *order = alt2 ? v2 : v1;
        CUDA_TRY(launch_gather_in(order, src.as<int32_t>(), row_of, m->w.as<float>(),
                                  m->aff.as<float>(), m->in_src.as<int32_t>(), m->in_w.as<float>(),
                                  m->in_aff.as<float>(), nnz, st));
    }
    int64_t *degp = deg.as<int64_t>();
    CUDA_TRY(cudaMemsetAsync(degp, 0, (size_t)(n + 1) * sizeof(int64_t), st));
    CUDA_TRY(launch_in_degree(m->col.as<int32_t>(), m->row_of.as<int32_t>(), nnz, degp, st));
    CUDA_TRY(scan_exclusive(degp, m->in_ptr.as<int64_t>(), n, tmp.p, tmp.cap, st));
    return build_split_plan(m, st);
}

// Split plan: hub rows cut into window segments, segments in window-major
// order, split rows heaviest first.
static akashic_status_t build_split_plan(akashic_mem *m, cudaStream_t st) {
    const int64_t n = m->n;
    m->mass_levels = -1;   // the graph changed
    m->reach_levels = -1;
    table_turn(m);
    // temporaries from the store's scratch (slots SCR_SPLIT0..11)
    akashic_status_t sc_rc = AKASHIC_OK;
    auto get = [&](int i, size_t bytes) -> Tmp {
        void *q = store_scratch(m, SCR_SPLIT0 + i, bytes);
        if (!q) sc_rc = AKASHIC_ENOMEM;
        return Tmp{q, bytes};
    };
    // sizes first (read back once), then the plan
    const int64_t max_hubs = m->nnz / (m->split.split_t + 1);
    const Tmp words = get(0, (size_t)hub_plan_words(n, max_hubs) * 8);
    const Tmp rows = get(1, (size_t)(max_hubs + 1) * 4), slot0 = get(2, (size_t)(max_hubs + 1) * 8);
    const Tmp counts = get(3, 16);
    if (sc_rc != AKASHIC_OK) return fail(sc_rc, "relation graph rebuild: out of device memory");
    CUDA_TRY(launch_hub_count(m->split, m->in_ptr.as<int64_t>(), m->in_src.as<int32_t>(), n,
                              max_hubs, rows.as<int32_t>(), slot0.as<int64_t>(),
                              counts.as<int64_t>(), words.as<int64_t>(), st));
    int64_t got[2] = {0, 0};
    CUDA_TRY(cudaMemcpyAsync(got, counts.p, 8, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(got + 1, slot0.as<int64_t>() + max_hubs, 8, cudaMemcpyDeviceToHost,
                             st));
    AK_TRY(check_status(m, st, "relation graph rebuild"));
    const int64_t n_split = got[0], n_segs = got[1];
    if (n_segs > 0x7fffffffLL) return fail(AKASHIC_ECAPACITY, "too many hub segments");
    m->n_segs = n_segs;
    m->n_split = n_split;
    if (n_split <= 0) return AKASHIC_OK;
    // grown with headroom: every relation update adds a few segments, and
    // a reallocation would synchronise the device
    AK_TRY(ensure_spare(m->split_row, (size_t)n_split * 4));
    AK_TRY(ensure_spare(m->split_slot0, (size_t)(n_split + 1) * 8));
    AK_TRY(ensure_spare(m->seg_e0, (size_t)n_segs * 8));
    AK_TRY(ensure_spare(m->seg_e1, (size_t)n_segs * 8));
    AK_TRY(ensure_spare(m->seg_slot, (size_t)n_segs * 4));
    AK_TRY(ensure_spare(m->split_order, (size_t)n_split * 4));
    AK_TRY(ensure_spare(m->slot_split, (size_t)n_segs * 4));
    const Tmp e0 = get(4, (size_t)n_segs * 8), e1 = get(5, (size_t)n_segs * 8);
    const Tmp win = get(6, (size_t)n_segs * 4), order = get(7, (size_t)n_segs * 4);
    const Tmp win2 = get(8, (size_t)n_segs * 4), order2 = get(9, (size_t)n_segs * 4);
    const Tmp rkey = get(10, (size_t)n_split * 8), rtmp = get(11, radix_tmp_bytes(n_segs) + 4096);
    if (sc_rc != AKASHIC_OK) return fail(sc_rc, "relation graph rebuild: out of device memory");
    uint32_t *row_key = rkey.as<uint32_t>(), *row_id = row_key + n_split;
    CUDA_TRY(launch_hub_fill(m->split, m->in_ptr.as<int64_t>(), m->in_src.as<int32_t>(),
                             rows.as<int32_t>(), slot0.as<int64_t>(), n_split, n_segs,
                             m->split_row.as<int32_t>(), m->split_slot0.as<int64_t>(),
                             e0.as<int64_t>(), e1.as<int64_t>(), win.as<uint32_t>(),
                             order.as<uint32_t>(), m->slot_split.as<int32_t>(), row_key, row_id,
                             st));
    bool alt = false;
    CUDA_TRY(radix_sort_pairs(win.as<uint32_t>(), order.as<uint32_t>(), win2.as<uint32_t>(),
                              order2.as<uint32_t>(), n_segs, bits_for((n - 1) / m->split.win_rows),
                              rtmp.p, rtmp.cap, st, &alt));
    CUDA_TRY(launch_seg_permute(alt ? order2.as<uint32_t>() : order.as<uint32_t>(),
                                e0.as<int64_t>(), e1.as<int64_t>(), n_segs,
                                m->seg_e0.as<int64_t>(), m->seg_e1.as<int64_t>(),
                                m->seg_slot.as<int32_t>(), st));
    // split rows heaviest first (the hop's fixup order); the segments' sort
    // buffers are free again
    bool alt2 = false;
    CUDA_TRY(radix_sort_pairs(row_key, row_id, win.as<uint32_t>(), win2.as<uint32_t>(), n_split,
                              bits_for(n_segs), rtmp.p, rtmp.cap, st, &alt2));
    CUDA_TRY(cudaMemcpyAsync(m->split_order.p, alt2 ? win2.p : row_id, (size_t)n_split * 4,
                             cudaMemcpyDeviceToDevice, st));
    return AKASHIC_OK;
}

// ================================================================== ABI
extern "C" {

const char *akashic_mem_last_error(void) { return g_last_error.c_str(); }

akashic_status_t akashic_mem_create(const akashic_mem_config_t *cfg, akashic_mem_t **out) {
    g_last_error.clear();
    if (!cfg || !out) return fail(AKASHIC_EINVAL, "create: NULL argument");
    *out = nullptr;
    if (cfg->dim < 64 || cfg->dim > 4096 || cfg->dim % 64 != 0)
        return fail(AKASHIC_EINVAL, "create: dim must be a multiple of 64 in [64, 4096]");
    if (cfg->capacity < 1 || cfg->capacity > 0x7fffffffLL)
        return fail(AKASHIC_EINVAL, "create: capacity must be in [1, 2^31-1]");
    if (cfg->chunks_per_page < 1) return fail(AKASHIC_EINVAL, "create: chunks_per_page < 1");
    if (!(cfg->temperature >= 0.f) || !isfinite(cfg->temperature) ||
        !(cfg->relation_scale >= 0.f) || !isfinite(cfg->relation_scale))
        return fail(AKASHIC_EINVAL, "create: temperature/relation_scale must be finite and >= 0");
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || cfg->device < 0 || cfg->device >= ndev) {
        cudaGetLastError();
        return fail(AKASHIC_EINVAL, "create: no CUDA device %d", cfg->device);
    }
    DeviceGuard g(cfg->device);
    akashic_mem *m = new (std::nothrow) akashic_mem();
    if (!m) return fail(AKASHIC_ENOMEM, "create: host allocation failed");
    m->device = cfg->device;
    m->dim = cfg->dim;
    m->cap = cfg->capacity;
    m->per_page = cfg->chunks_per_page;
    m->tau = cfg->temperature > 0.f ? cfg->temperature : 1.0f / sqrtf((float)cfg->dim);
    m->rel_scale = cfg->relation_scale > 0.f ? cfg->relation_scale : 10.f;
    // propagation plan knobs (tuning only; results do not depend on them
    // beyond fp32 summation order)
    if (const char *v = getenv("AKASHIC_SPLIT_T")) m->split.split_t = atoll(v) > 0 ? atoll(v) : m->split.split_t;
    if (const char *v = getenv("AKASHIC_SEG_LEN")) m->split.seg_len = atoll(v) > 0 ? atoll(v) : m->split.seg_len;
    if (const char *v = getenv("AKASHIC_FUSE_FILTER")) m->fuse_filter = atoi(v) != 0;
    if (const char *v = getenv("AKASHIC_HOP_PRUNE")) m->hop_prune = atoi(v) != 0;
    if (const char *v = getenv("AKASHIC_REACH")) m->reach_on = atoi(v) != 0;
    if (const char *v = getenv("AKASHIC_FULL_TRANSPOSE")) m->inc_transpose = atoi(v) == 0;
    if (const char *v = getenv("AKASHIC_WIN_ROWS")) m->split.win_rows = atoll(v) > 0 ? atoll(v) : m->split.win_rows;
    akashic_status_t s;
    if ((s = m->emb.ensure((size_t)m->cap * m->dim * 2)) != AKASHIC_OK ||
        (s = m->page_of.ensure((size_t)m->cap * 4)) != AKASHIC_OK ||
        (s = m->ext_of.ensure((size_t)m->cap * 4)) != AKASHIC_OK ||
        (s = m->row_of.ensure((size_t)m->cap * 4)) != AKASHIC_OK ||
        (s = m->max_norm.ensure(4)) != AKASHIC_OK || (s = m->status.ensure(4)) != AKASHIC_OK ||
        (s = m->rstat.ensure((size_t)m->cap * 8)) != AKASHIC_OK ||
        (s = m->ns_row.ensure((size_t)m->cap * 4)) != AKASHIC_OK ||
        (s = m->dead_row.ensure((size_t)m->cap * 4)) != AKASHIC_OK ||
        (s = m->row_ptr.ensure((size_t)(m->cap + 1) * 8)) != AKASHIC_OK ||
        (s = m->in_ptr.ensure((size_t)(m->cap + 1) * 8)) != AKASHIC_OK) {
        delete m;
        return s;
    }
    if (cudaMemset(m->max_norm.p, 0, 4) != cudaSuccess || cudaMemset(m->status.p, 0, 4) != cudaSuccess ||
        cudaMemset(m->row_ptr.p, 0, 8) != cudaSuccess || cudaMemset(m->in_ptr.p, 0, 8) != cudaSuccess ||
        cudaMemset(m->ns_row.p, 0, (size_t)m->cap * 4) != cudaSuccess ||
        cudaMemset(m->dead_row.p, 0, (size_t)m->cap * 4) != cudaSuccess ||
        m->sel.ensure((size_t)m->cap * 4) != AKASHIC_OK ||
        cudaMemset(m->sel.p, 0, (size_t)m->cap * 4) != cudaSuccess ||
        m->mm_ctr.ensure(64) != AKASHIC_OK || cudaMemset(m->mm_ctr.p, 0, 64) != cudaSuccess ||
        mm_ensure_pages(m, 1024, 0) != AKASHIC_OK || mm_ensure_pairs(m, 0, 0) != AKASHIC_OK ||
        cudaDeviceSynchronize() != cudaSuccess) {
        delete m;
        return fail(AKASHIC_ECUDA, "create: initialisation failed");
    }
    *out = m;
    return AKASHIC_OK;
}

void akashic_mem_destroy(akashic_mem_t *m) {
    if (!m) return;
    DeviceGuard g(m->device);
    cudaDeviceSynchronize();
    delete m;
}

akashic_status_t akashic_mem_size(const akashic_mem_t *m, int64_t *n_chunks, int64_t *nnz) {
    if (!m) return fail(AKASHIC_EINVAL, "size: NULL store");
    if (n_chunks) *n_chunks = m->n;
    if (nnz) *nnz = m->nnz;
    return AKASHIC_OK;
}

akashic_status_t akashic_mem_sync(akashic_mem_t *m, void *stream) {
    if (!m) return fail(AKASHIC_EINVAL, "sync: NULL store");
    DeviceGuard g(m->device);
    return check_status(m, (cudaStream_t)stream, "sync");
}

akashic_status_t akashic_mem_check_wait_timeout(akashic_mem_t *m, uint32_t polls, void *stream) {
    g_last_error.clear();
    if (!m) return fail(AKASHIC_EINVAL, "check_wait_timeout: NULL store");
    if (polls < 1 || polls > (1u << 26))
        return fail(AKASHIC_EINVAL, "check_wait_timeout: polls must be in [1, 2^26]");
    DeviceGuard g(m->device);
    CUDA_TRY(launch_wait_timeout_check(m->status.as<int>(), polls, (cudaStream_t)stream));
    return AKASHIC_OK;
}

akashic_status_t akashic_mem_sort_pairs(uint32_t *keys, uint32_t *vals, int64_t n, int32_t bits,
                                        void *stream) {
    g_last_error.clear();
    if (n < 0 || n > 0x7fffffffLL || bits < 0 || bits > 32 || (n > 1 && (!keys || !vals)))
        return fail(AKASHIC_EINVAL, "sort_pairs: bad n, bits or buffers");
    if (n <= 1 || bits == 0) return AKASHIC_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t words = ((size_t)n * 8 + 255) & ~(size_t)255;
    const size_t tb = radix_tmp_bytes(n) + 4096;
    void *buf = nullptr;
    if (cudaMalloc(&buf, words + tb) != cudaSuccess) {
        cudaGetLastError();
        return fail(AKASHIC_ENOMEM, "sort_pairs: %lld bytes of scratch", (long long)(words + tb));
    }
    uint32_t *k2 = (uint32_t *)buf, *v2 = k2 + n;
    bool alt = false;
    cudaError_t e = radix_sort_pairs(keys, vals, k2, v2, n, bits, (uint8_t *)buf + words, tb, st,
                                     &alt);
    if (e == cudaSuccess && alt)
        e = cudaMemcpyAsync(keys, k2, (size_t)n * 4, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && alt)
        e = cudaMemcpyAsync(vals, v2, (size_t)n * 4, cudaMemcpyDeviceToDevice, st);
    const cudaError_t es = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = es;
    cudaFree(buf);
    if (e != cudaSuccess) return fail(AKASHIC_ECUDA, "sort_pairs: %s", cudaGetErrorString(e));
    return AKASHIC_OK;
}

akashic_status_t akashic_mem_append_chunks(akashic_mem_t *m, const uint16_t *emb, int64_t n,
                                           const int32_t *page_of, const int64_t *row_ptr,
                                           const int32_t *col, const float *aff,
                                           int64_t *first_id_out, void *stream) {
    g_last_error.clear();
    if (!m) return fail(AKASHIC_EINVAL, "append: NULL store");
    if (n < 0 || (n > 0 && !emb)) return fail(AKASHIC_EINVAL, "append: bad n or emb");
    if (((uintptr_t)emb & 15u) != 0) return fail(AKASHIC_EINVAL, "append: emb must be 16-byte aligned");
    const bool has_edges = row_ptr != nullptr;
    if (!row_ptr && (col || aff))
        return fail(AKASHIC_EINVAL, "append: col/aff given without row_ptr");
    if (m->n + n > m->cap)
        return fail(AKASHIC_ECAPACITY, "append: %lld + %lld chunks exceed capacity %lld",
                    (long long)m->n, (long long)n, (long long)m->cap);
    if (first_id_out) *first_id_out = m->n;
    if (n == 0) return AKASHIC_OK;
    DeviceGuard g(m->device);
    Reclaim reclaim(m);
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t first = m->n;
    PhaseScope ph(m, AKASHIC_PHASE_GRAPH, st);
    // -- validate the new edges before anything is committed
    int64_t e_lo = 0, e_hi = 0;
    if (has_edges) {
        CUDA_TRY(cudaMemcpyAsync(&e_lo, row_ptr, 8, cudaMemcpyDeviceToHost, st));
        CUDA_TRY(cudaMemcpyAsync(&e_hi, row_ptr + n, 8, cudaMemcpyDeviceToHost, st));
        CUDA_TRY(launch_edge_src_check(row_ptr, col, n, first, first + n, nullptr,
                                       m->status.as<int>(), st));
        AK_TRY(check_status(m, st, "append: edge check"));
        if (e_hi < e_lo) return fail(AKASHIC_EINVAL, "append: row_ptr decreases");
        if (m->has_dead && e_hi > e_lo && col) {
            CUDA_TRY(launch_check_dead_targets(col + e_lo, e_hi - e_lo, first,
                                               m->row_of.as<int32_t>(), m->dead_row.as<int32_t>(),
                                               m->status.as<int>(), st));
            AK_TRY(check_status(m, st, "append: an edge points at a deleted chunk"));
        }
        if (e_hi > e_lo && !(col && aff))
            return fail(AKASHIC_EINVAL, "append: edges given without col or aff");
        if (m->nnz + (e_hi - e_lo) > 0x7fffffffLL)
            return fail(AKASHIC_ECAPACITY, "append: more than 2^31-1 relation edges");
    }
    int64_t max_page = -1;
    if (page_of) {
        DevBuf pm;
        AK_TRY(pm.ensure(4));
        int init = -1;
        CUDA_TRY(cudaMemcpyAsync(pm.p, &init, 4, cudaMemcpyHostToDevice, st));
        k_page_max<<<device_sm_count(), 256, 0, st>>>(page_of, n, pm.as<int>(), m->status.as<int>());
        CUDA_TRY(cudaGetLastError());
        int mx = -1;
        CUDA_TRY(cudaMemcpyAsync(&mx, pm.p, 4, cudaMemcpyDeviceToHost, st));
        AK_TRY(check_status(m, st, "append: page_of must be >= 0"));
        max_page = mx;
    }
    const int64_t new_nnz = e_hi - e_lo;
    if (new_nnz > 0) {
        const size_t need = (size_t)(m->nnz + new_nnz);
        size_t grow = need + need / 4;
        AK_TRY(m->col.ensure(grow * 4, true, st));
        AK_TRY(m->aff.ensure(grow * 4, true, st));
        AK_TRY(m->w.ensure(grow * 4, true, st));
    }
    // -- the batch's rows in page order (stable: ID order within a page)
    DevBuf okeys, ovals, okeys2, ovals2, otmp;
    const uint32_t *order = nullptr;
    if (page_of && max_page > 0 && n > 1) {
        AK_TRY(okeys.ensure((size_t)n * 4));
        AK_TRY(ovals.ensure((size_t)n * 4));
        AK_TRY(okeys2.ensure((size_t)n * 4));
        AK_TRY(ovals2.ensure((size_t)n * 4));
        AK_TRY(otmp.ensure(radix_tmp_bytes(n) + 4096));
        CUDA_TRY(cudaMemcpyAsync(okeys.p, page_of, (size_t)n * 4, cudaMemcpyDeviceToDevice, st));
        CUDA_TRY(launch_iota(ovals.as<uint32_t>(), n, st));
        bool alt = false;
        CUDA_TRY(radix_sort_pairs(okeys.as<uint32_t>(), ovals.as<uint32_t>(), okeys2.as<uint32_t>(),
                                  ovals2.as<uint32_t>(), n, bits_for(max_page), otmp.p, otmp.cap,
                                  st, &alt));
        order = alt ? ovals2.as<uint32_t>() : ovals.as<uint32_t>();
    }
    // -- commit
    CUDA_TRY(launch_batch_layout(order, first, n, m->dim, emb, m->emb.as<uint16_t>(), page_of,
                                 m->next_page, m->per_page, m->page_of.as<int32_t>(),
                                 m->ext_of.as<int32_t>(), m->row_of.as<int32_t>(), st));
    if (page_of) {
        if (max_page + 1 > m->next_page) m->next_page = max_page + 1;
    } else {
        m->next_page += ceil_div<int64_t>(n, m->per_page);
    }
    // the new chunks occupy a slot of their pages
    AK_TRY(mm_ensure_pages(m, m->next_page + 1, st));
    CUDA_TRY(launch_mm_count_pages(m->page_of.as<int32_t>(), first, n, mm_tables(m), st));
    m->appended += n;
    CUDA_TRY(launch_row_norm_max(m->emb.as<uint16_t>() + first * m->dim, n, m->dim,
                                 m->max_norm.as<float>(), st));
    int64_t *rp = m->row_ptr.as<int64_t>() + first;   // rp[0] is already m->nnz
    k_rebase_ptr<<<device_sm_count() * 4, 256, 0, st>>>(has_edges ? row_ptr : nullptr, rp, n + 1,
                                                         m->nnz);
    CUDA_TRY(cudaGetLastError());
    if (new_nnz > 0) {
        CUDA_TRY(cudaMemcpyAsync(m->col.as<int32_t>() + m->nnz, col + e_lo, (size_t)new_nnz * 4,
                                 cudaMemcpyDeviceToDevice, st));
        CUDA_TRY(cudaMemcpyAsync(m->aff.as<float>() + m->nnz, aff + e_lo, (size_t)new_nnz * 4,
                                 cudaMemcpyDeviceToDevice, st));
        CUDA_TRY(launch_row_softmax(rp, m->aff.as<float>(), m->w.as<float>(), n,
                                    m->rstat.as<float2>() + first, st));
    }
    m->n += n;
    m->nnz += new_nnz;
    if (new_nnz == 0 && first > 0) {
        // no new edges: the new rows have no in-edges, the transpose and the
        // hub plan are unchanged; only the row pointers are extended
        k_rebase_ptr<<<device_sm_count() * 4, 256, 0, st>>>(nullptr, m->in_ptr.as<int64_t>() + first + 1,
                                                             n, m->nnz);
        CUDA_TRY(cudaGetLastError());
        return check_status(m, st, "append");
    }
    AK_TRY(rebuild_in_edges(m, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    return AKASHIC_OK;
}

akashic_status_t akashic_mem_update_relations(akashic_mem_t *m, int64_t first, int64_t n,
                                              int32_t M, int32_t reciprocal, void *stream) {
    g_last_error.clear();
    if (!m) return fail(AKASHIC_EINVAL, "update: NULL store");
    if (first < 0 || n < 0 || first + n > m->n)
        return fail(AKASHIC_EINVAL, "update: range [%lld, %lld) outside the store of %lld",
                    (long long)first, (long long)(first + n), (long long)m->n);
    if (M < 1 || M > 64 || M > first)
        return fail(AKASHIC_EINVAL, "update: M must be in [1, min(64, first)]");
    if (n == 0) return AKASHIC_OK;
    DeviceGuard g(m->device);
    Reclaim reclaim(m);
    cudaStream_t st = (cudaStream_t)stream;
    UpdateArgs ua;
    ua.emb = m->emb.as<uint16_t>();
    ua.dim = m->dim;
    ua.n_rows = m->n;
    ua.first = first;
    ua.n_new = n;
    ua.M = M;
    ua.reciprocal = reciprocal != 0;
    ua.scale = m->rel_scale;
    ua.status = m->status.as<int>();
    ua.ext_of = m->ext_of.as<int32_t>();
    ua.row_of = m->row_of.as<int32_t>();
    int64_t nnz_new = m->nnz + n * M * (reciprocal ? 2 : 1);
    if (nnz_new > 0x7fffffffLL)
        return fail(AKASHIC_ECAPACITY, "update: more than 2^31-1 relation edges");
    ua.scratch = store_scratch;
    ua.scratch_ctx = m;
    ua.dead_row = m->has_dead ? m->dead_row.as<int32_t>() : nullptr;
    ua.nbr_ids = (int32_t *)store_scratch(m, SCR_NBR_IDS, (size_t)n * M * 4);
    ua.nbr_cos = (float *)store_scratch(m, SCR_NBR_COS, (size_t)n * M * 4);
    if (!ua.nbr_ids || !ua.nbr_cos) return fail(AKASHIC_ENOMEM, "update: out of device memory");
    DevBuf &ncol = m->col2, &naff = m->aff2, &nrp = m->rp2;
    AK_TRY(ensure_spare(ncol, (size_t)nnz_new * 4));
    AK_TRY(ensure_spare(naff, (size_t)nnz_new * 4));
    AK_TRY(ensure_spare(nrp, (size_t)(m->cap + 1) * 8));
    AK_TRY(ensure_spare(m->w2, (size_t)nnz_new * 4));
    uint32_t *touched =
        (uint32_t *)store_scratch(m, SCR_TOUCHED, (size_t)ceil_div<int64_t>(m->n, 32) * 4);
    if (!touched) return fail(AKASHIC_ENOMEM, "update: out of device memory");
    // the transpose is patched (or built anew, where there is none), into spares
    // that are taken now too: both lists change together or not at all (csr_insert
    // is done with the slots that it shares, of the same sizes)
    const int64_t nnz_old = m->nnz, pairs = n * (int64_t)M;
    const bool patch = m->inc_transpose && nnz_old > 0;
    DevBuf &ptr2 = m->in_ptr2, &src2 = m->in_src2, &aff2 = m->in_aff2, &w2 = m->in_w2;
    const size_t tb = radix_tmp_bytes(pairs) + 4096;   // pairs >= n: the new rows' sort too
    InEdgeScratch sc{};
    if (patch) {
        AK_TRY(ensure_spare(ptr2, (size_t)(m->cap + 1) * 8));
        AK_TRY(ensure_spare(src2, (size_t)nnz_new * 4));
        AK_TRY(ensure_spare(aff2, (size_t)nnz_new * 4));
        AK_TRY(ensure_spare(w2, (size_t)nnz_new * 4));
        auto get = [&](int slot, size_t bytes) {
            return (uint32_t *)store_scratch(m, slot, bytes);
        };
        sc = InEdgeScratch{get(SCR_KEYS, (size_t)pairs * 4 + 16), get(SCR_VALS, (size_t)pairs * 4 + 16),
                           get(SCR_KEYS2, (size_t)pairs * 4 + 16), get(SCR_VALS2, (size_t)pairs * 4 + 16),
                           get(SCR_IN_ROWS, (size_t)n * 16),
                           get(SCR_MOVE, (size_t)(1 + move_words(nnz_old, pairs, n)) * 4),
                           get(SCR_TMP, tb), tb};
        if (!sc.keys || !sc.vals || !sc.keys2 || !sc.vals2 || !sc.rows || !sc.move || !sc.tmp)
            return fail(AKASHIC_ENOMEM, "update: out of device memory");
    }
    {
        // rows [first, first+n) must have no out-edges and no in-edges: checked on
        // the device, read back with the top-M's outcome, before anything changes
        PhaseScope ph(m, AKASHIC_PHASE_RELATE, st);
        CUDA_TRY(launch_check_new_rows(m->row_ptr.as<int64_t>(), m->in_ptr.as<int64_t>(),
                                       m->row_of.as<int32_t>(), first, n, m->status.as<int>(), st));
        int code = 0;
        akashic_status_t r = relate_top_m(ua, st, &ph.launches, &code);
        if (r != AKASHIC_OK) return fail(r, "update: relation GEMM / top-M failed");
        if (code != 0)
            return check_status(m, st, code == AKASHIC_EINVAL
                                           ? "update: rows [first, first+n) already have out-edges"
                                           : "update");
    }
    {
        PhaseScope ph(m, AKASHIC_PHASE_GRAPH, st);
        {
            PhaseScope pc(m, AKASHIC_PHASE_CSR_INSERT, st);
            akashic_status_t r = csr_insert(ua, m->row_ptr.as<int64_t>(), m->col.as<int32_t>(),
                                            m->aff.as<float>(), m->w.as<float>(), m->nnz,
                                            nrp.as<int64_t>(), ncol.as<int32_t>(),
                                            naff.as<float>(), m->w2.as<float>(),
                                            m->rstat.as<float2>(), touched, st, &pc.launches);
            ph.launches += pc.launches;
            if (r != AKASHIC_OK) return fail(r, "update: CSR insert failed");
        }
        PhaseScope pt(m, AKASHIC_PHASE_TRANSPOSE, st);
        if (patch) {
            // old lists moved, new edges placed, weights recomputed from the
            // logits (ak_inedges.cu)
            InEdgeUpdate u;
            u.n = m->n;
            u.nnz_new = nnz_new;
            u.in_ptr_old = m->in_ptr.as<int64_t>();
            u.in_src_old = m->in_src.as<int32_t>();
            u.in_aff_old = m->in_aff.as<float>();
            u.in_w_old = m->in_w.as<float>();
            u.touched = touched;
            u.in_ptr_new = ptr2.as<int64_t>();
            u.in_src_new = src2.as<int32_t>();
            u.in_aff_new = aff2.as<float>();
            u.in_w_new = w2.as<float>();
            u.nbr_ids = ua.nbr_ids;
            u.nbr_cos = ua.nbr_cos;
            u.scale = m->rel_scale;
            u.first = first;
            u.n_new = n;
            u.M = M;
            u.reciprocal = reciprocal != 0;
            u.row_bits = bits_for(m->n - 1);
            u.row_of = m->row_of.as<int32_t>();
            u.ext_of = m->ext_of.as<int32_t>();
            u.rstat = m->rstat.as<float2>();
            CUDA_TRY(launch_in_edges_update(u, sc, st, &pt.launches));
            swap_bufs(m->in_ptr, ptr2);
            swap_bufs(m->in_src, src2);
            swap_bufs(m->in_aff, aff2);
            swap_bufs(m->in_w, w2);
        }
        swap_bufs(m->row_ptr, nrp);
        swap_bufs(m->col, ncol);
        swap_bufs(m->aff, naff);
        swap_bufs(m->w, m->w2);
        m->nnz = nnz_new;
        if (patch) {
            pt.end();
            ph.launches += pt.launches;
            PhaseScope phub(m, AKASHIC_PHASE_HUB_PLAN, st);
            AK_TRY(build_split_plan(m, st));
        } else {
            AK_TRY(rebuild_in_edges(m, st));
        }
    }
    CUDA_TRY(cudaStreamSynchronize(st));
    return AKASHIC_OK;
}

static StreamScratch *scratch_for(akashic_mem *m, void *stream) {
    std::lock_guard<std::mutex> g(m->mu);
    auto it = m->scratch.find(stream);
    if (it != m->scratch.end()) return it->second;
    StreamScratch *s = new (std::nothrow) StreamScratch();
    if (s) m->scratch[stream] = s;
    return s;
}

static akashic_status_t retrieve_impl(akashic_mem *m, const uint16_t *q, int32_t B, int32_t k,
                                      float alpha, int32_t hops, const int32_t *q_ns,
                                      int32_t sort_by_time, int64_t *ids, float *scores,
                                      int32_t *page_ids, int32_t *n_pages, void *stream);

akashic_status_t akashic_mem_retrieve(akashic_mem_t *m, const uint16_t *q, int32_t B, int32_t k,
                                      float alpha, int32_t hops, int64_t *ids, float *scores,
                                      int32_t *page_ids, int32_t *n_pages, void *stream) {
    g_last_error.clear();
    return retrieve_impl(m, q, B, k, alpha, hops, nullptr, 0, ids, scores, page_ids, n_pages,
                         stream);
}

akashic_status_t akashic_mem_retrieve_scoped(akashic_mem_t *m, const uint16_t *q, int32_t B,
                                             int32_t k, float alpha, int32_t hops,
                                             const int32_t *q_ns, int32_t sort_by_time,
                                             int64_t *ids, float *scores, int32_t *page_ids,
                                             int32_t *n_pages, void *stream) {
    g_last_error.clear();
    return retrieve_impl(m, q, B, k, alpha, hops, q_ns, sort_by_time, ids, scores, page_ids,
                         n_pages, stream);
}

akashic_status_t akashic_mem_set_namespace(akashic_mem_t *m, int64_t first, int64_t n,
                                           const int32_t *ns, void *stream) {
    g_last_error.clear();
    if (!m) return fail(AKASHIC_EINVAL, "set_namespace: NULL store");
    if (first < 0 || n < 0 || first + n > m->n)
        return fail(AKASHIC_EINVAL, "set_namespace: range [%lld, %lld) outside the store of %lld",
                    (long long)first, (long long)(first + n), (long long)m->n);
    if (n == 0) return AKASHIC_OK;
    if (!ns) return fail(AKASHIC_EINVAL, "set_namespace: NULL ns");
    DeviceGuard g(m->device);
    CUDA_TRY(launch_scatter_by_row(ns, m->row_of.as<int32_t>(), first, n, m->ns_row.as<int32_t>(),
                                   (cudaStream_t)stream));
    return AKASHIC_OK;
}
akashic_status_t akashic_mem_delete(akashic_mem_t *m, const int64_t *ids, int64_t n,
                                    void *stream) {
    g_last_error.clear();
    if (!m) return fail(AKASHIC_EINVAL, "delete: NULL store");
    if (n < 0) return fail(AKASHIC_EINVAL, "delete: n < 0");
    if (n == 0) return AKASHIC_OK;
    if (!ids) return fail(AKASHIC_EINVAL, "delete: NULL ids");
    DeviceGuard g(m->device);
    Reclaim reclaim(m);
    cudaStream_t st = (cudaStream_t)stream;
    // check every ID first, so that a bad list changes nothing
    CUDA_TRY(launch_mark_dead(ids, n, m->n, m->row_of.as<int32_t>(), nullptr,
                              m->status.as<int>(), st));
    AK_TRY(check_status(m, st, "delete: chunk IDs must lie in [0, size)"));
    CUDA_TRY(launch_mark_dead(ids, n, m->n, m->row_of.as<int32_t>(), m->dead_row.as<int32_t>(),
                              m->status.as<int>(), st, m->page_of.as<int32_t>(),
                              m->page_live.as<int32_t>()));
    m->has_dead = true;
    const int64_t rows = m->n, nnz = m->nnz;
    if (nnz == 0) return AKASHIC_OK;
    // bitmaps of the deleted chunks and of the rows whose weights change, and
    // the compaction's scratch; what has to start at zero comes first
    const size_t rb = (size_t)ceil_div<int64_t>(rows, 32) * 4;
    const size_t eb = (size_t)ceil_div<int64_t>(nnz, 32) * 4;
    const size_t cb = (size_t)drop_words(nnz) * 4;
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t zero = 2 * up(rb) + 2 * up(eb);
    uint8_t *scr = (uint8_t *)store_scratch(m, SCR_DEL, zero + up(rb) + 2 * up(eb) + up(cb));
    if (!scr) return fail(AKASHIC_ENOMEM, "delete: out of device memory");
    uint32_t *dead_id = (uint32_t *)scr;
    uint32_t *touched = (uint32_t *)(scr + up(rb));
    uint32_t *drop = (uint32_t *)(scr + 2 * up(rb));
    uint32_t *drop_in = (uint32_t *)(scr + 2 * up(rb) + up(eb));
    uint32_t *dead_bits = (uint32_t *)(scr + zero);
    uint32_t *keep = (uint32_t *)(scr + zero + up(rb));
    int32_t *word_pos = (int32_t *)(scr + zero + up(rb) + up(eb));
    int32_t *counts = (int32_t *)(scr + zero + up(rb) + 2 * up(eb));
    AK_TRY(ensure_spare(m->rp2, (size_t)(m->cap + 1) * 8));
    AK_TRY(ensure_spare(m->col2, (size_t)nnz * 4));
    AK_TRY(ensure_spare(m->aff2, (size_t)nnz * 4));
    AK_TRY(ensure_spare(m->w2, (size_t)nnz * 4));
    AK_TRY(ensure_spare(m->in_ptr2, (size_t)(m->cap + 1) * 8));
    AK_TRY(ensure_spare(m->in_src2, (size_t)nnz * 4));
    AK_TRY(ensure_spare(m->in_aff2, (size_t)nnz * 4));
    AK_TRY(ensure_spare(m->in_w2, (size_t)nnz * 4));
    CUDA_TRY(cudaMemsetAsync(scr, 0, zero, st));
    CUDA_TRY(launch_dead_bits(m->dead_row.as<int32_t>(), m->ext_of.as<int32_t>(), rows, dead_bits,
                              dead_id, st));
    // out-edge CSR (rows are chunk IDs, targets chunk IDs)
    DropDead d{};
    d.n_rows = rows;
    d.nnz = nnz;
    d.ptr = m->row_ptr.as<int64_t>();
    d.tgt = m->col.as<int32_t>();
    d.val = m->aff.as<float>();
    d.w = m->w.as<float>();
    d.dead_bits = dead_id;
    d.ids = ids;
    d.n_ids = n;
    d.n_total = rows;
    d.drop_bits = drop;
    d.keep_bits = keep;
    d.word_pos = word_pos;
    d.counts = counts;
    d.tgt_out = m->col2.as<int32_t>();
    d.val_out = m->aff2.as<float>();
    d.w_out = m->w2.as<float>();
    CUDA_TRY(launch_drop_dead_edges(d, st));
    CUDA_TRY(launch_drop_row_ptr(d, m->rp2.as<int64_t>(), m->w2.as<float>(),
                                 m->rstat.as<float2>(), m->row_of.as<int32_t>(), touched, st));
    int64_t nnz_new = 0;
    CUDA_TRY(cudaMemcpyAsync(&nnz_new, m->rp2.as<int64_t>() + rows, 8, cudaMemcpyDeviceToHost, st));
    // in-edge transpose (rows are store rows, sources rows); the same edges go
    DropDead di = d;
    di.ptr = m->in_ptr.as<int64_t>();
    di.tgt = m->in_src.as<int32_t>();
    di.val = m->in_aff.as<float>();
    di.w = m->in_w.as<float>();
    di.dead_bits = dead_bits;
    di.own_row_of = m->row_of.as<int32_t>();
    di.touched = touched;
    di.ext_of = m->ext_of.as<int32_t>();
    di.rstat = m->rstat.as<float2>();
    di.drop_bits = drop_in;
    di.tgt_out = m->in_src2.as<int32_t>();
    di.val_out = m->in_aff2.as<float>();
    di.w_out = m->in_w2.as<float>();
    CUDA_TRY(launch_drop_dead_edges(di, st));
    CUDA_TRY(launch_drop_row_ptr(di, m->in_ptr2.as<int64_t>(), nullptr, nullptr, nullptr, nullptr,
                                 st));
    CUDA_TRY(cudaStreamSynchronize(st));
    m->nnz = nnz_new;
    swap_bufs(m->row_ptr, m->rp2);
    swap_bufs(m->col, m->col2);
    swap_bufs(m->aff, m->aff2);
    swap_bufs(m->w, m->w2);
    swap_bufs(m->in_ptr, m->in_ptr2);
    swap_bufs(m->in_src, m->in_src2);
    swap_bufs(m->in_aff, m->in_aff2);
    swap_bufs(m->in_w, m->in_w2);
    AK_TRY(build_split_plan(m, st));
    return check_status(m, st, "delete");
}
akashic_status_t akashic_mem_relocate(akashic_mem_t *m, const int64_t *S, int32_t n_req,
                                      int32_t s_len, float tau_assoc, void *stream) {
    g_last_error.clear();
    if (!m) return fail(AKASHIC_EINVAL, "relocate: NULL store");
    if (n_req < 0 || s_len < 1 || s_len > 64)
        return fail(AKASHIC_EINVAL, "relocate: need n_req >= 0 and 1 <= s_len <= 64");
    if (!(tau_assoc >= 0.f && tau_assoc <= 1.f))
        return fail(AKASHIC_EINVAL, "relocate: tau_assoc must lie in [0, 1]");
    if (n_req == 0) return AKASHIC_OK;
    if (!S) return fail(AKASHIC_EINVAL, "relocate: NULL S");
    DeviceGuard g(m->device);
    Reclaim reclaim(m);
    cudaStream_t st = (cudaStream_t)stream;
    PhaseScope ph(m, AKASHIC_PHASE_RELOCATE, st);
    const int64_t pairs = (int64_t)n_req * s_len * (s_len - 1) / 2;
    AK_TRY(mm_ensure_pairs(m, pairs, st, &ph.launches));
    AK_TRY(mm_ensure_pages(m, m->next_page + (int64_t)n_req * ceil_div<int64_t>(64, m->per_page) + 1,
                           st));
    int32_t *gb = (int32_t *)store_scratch(m, SCR_MM_G, (size_t)n_req * 64 * 4);
    int32_t *gn = (int32_t *)store_scratch(m, SCR_MM_GN, (size_t)n_req * 4);
    if (!gb || !gn) return fail(AKASHIC_ENOMEM, "relocate: out of device memory");
    const int32_t *dead = m->has_dead ? m->dead_row.as<int32_t>() : nullptr;
    const MmTables t = mm_tables(m);
    int64_t *result = m->mm_ctr.as<int64_t>() + 4;
    CUDA_TRY(launch_mm_count(S, n_req, s_len, m->n, m->row_of.as<int32_t>(), dead, t,
                             m->status.as<int>(), st));
    CUDA_TRY(launch_mm_relocate(S, n_req, s_len, m->n, m->row_of.as<int32_t>(), dead,
                                m->page_of.as<int32_t>(), t, tau_assoc, m->next_page, m->per_page,
                                gb, gn, m->status.as<int>(), result, st));
    ph.launches += 3;
    // everything the host needs in one read-back, the status word with it
    int64_t got[4] = {0, 0, 0, 0};
    CUDA_TRY(cudaMemcpyAsync(got, result, 32, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    if (got[3] != 0) AK_TRY(check_status(m, st, "relocate"));
    m->next_page = got[0];
    m->moves += got[1];
    m->co_pairs = got[2];
    return AKASHIC_OK;
}

akashic_status_t akashic_mem_compact_pages(akashic_mem_t *m, float theta, float tau_assoc,
                                           int64_t *released, void *stream) {
    g_last_error.clear();
    if (!m) return fail(AKASHIC_EINVAL, "compact: NULL store");
    if (!(theta > 0.f && theta <= 1.f))
        return fail(AKASHIC_EINVAL, "compact: theta must lie in (0, 1]");
    if (!(tau_assoc >= 0.f && tau_assoc <= 1.f))
        return fail(AKASHIC_EINVAL, "compact: tau_assoc must lie in [0, 1]");
    DeviceGuard g(m->device);
    Reclaim reclaim(m);
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t n = m->n, pages = m->next_page;
    if (released) *released = 0;
    if (n == 0) return AKASHIC_OK;
    // the directory first: pages to compact and the live chunks on them, with
    // the union of their groups, read back together
    int32_t *cand = (int32_t *)store_scratch(m, SCR_MM_CAND, (size_t)(pages + 1) * 4);
    uint32_t *moving = (uint32_t *)store_scratch(m, SCR_MM_MOVING, (size_t)ceil_div<int64_t>(n, 32) * 4);
    int32_t *parent = (int32_t *)store_scratch(m, SCR_MM_PARENT, (size_t)n * 4);
    int32_t *counts = (int32_t *)store_scratch(m, SCR_MM_COUNTS, (size_t)mm_words(n) * 4);
    uint32_t *ids = (uint32_t *)store_scratch(m, SCR_MM_IDS, (size_t)n * 4 + 16);
    uint32_t *nsk = (uint32_t *)store_scratch(m, SCR_MM_NSK, (size_t)n * 4 + 16);
    if (!cand || !moving || !parent || !counts || !ids || !nsk)
        return fail(AKASHIC_ENOMEM, "compact: out of device memory");
    PhaseScope ph(m, AKASHIC_PHASE_COMPACT, st);
    const MmTables t = mm_tables(m);
    const int32_t *dead = m->has_dead ? m->dead_row.as<int32_t>() : nullptr;
    const int32_t *row_of = m->row_of.as<int32_t>(), *ns_row = m->ns_row.as<int32_t>();
    CUDA_TRY(launch_mm_candidates(t, pages, theta, cand, st));
    CUDA_TRY(launch_mm_collect(t, n, row_of, dead, m->page_of.as<int32_t>(), ns_row, cand, moving,
                               parent, ids, nsk, counts, st));
    CUDA_TRY(launch_mm_union(t, moving, row_of, ns_row, tau_assoc, parent, m->status.as<int>(), st));
    ph.launches += (pages > 0) + 3;
    int64_t rc[2] = {0, 0};
    CUDA_TRY(cudaMemcpyAsync(rc, t.released, 16, cudaMemcpyDeviceToHost, st));
    AK_TRY(check_status(m, st, "compact"));
    const int64_t n_rel = rc[0], count = rc[1];
    if (n_rel == 0) return AKASHIC_OK;
    int64_t new_pages = 0;
    if (count > 0 && count <= mm_small_repack()) {
        // (a fresh page a chunk at most)
        AK_TRY(mm_ensure_pages(m, m->next_page + count + 1, st));
        int64_t *np = m->mm_ctr.as<int64_t>() + 3;
        CUDA_TRY(launch_mm_repack_small(mm_tables(m), pages, cand, ids, nsk, count, parent, row_of,
                                        m->page_of.as<int32_t>(), m->next_page, m->per_page, np,
                                        st));
        ph.launches += 2;
        CUDA_TRY(cudaMemcpyAsync(&new_pages, np, 8, cudaMemcpyDeviceToHost, st));
        CUDA_TRY(cudaStreamSynchronize(st));
        m->next_page += new_pages;
        m->moves += count;
        if (released) *released = n_rel;
        return AKASHIC_OK;
    }
    if (count > 0) {
        const size_t tb = (scan_tmp_bytes(count + 1) > radix_tmp_bytes(count)
                               ? scan_tmp_bytes(count + 1) : radix_tmp_bytes(count)) + 4096;
        uint32_t *root = (uint32_t *)store_scratch(m, SCR_MM_ROOT, (size_t)count * 4 + 16);
        uint32_t *k2 = (uint32_t *)store_scratch(m, SCR_MM_K2, (size_t)count * 4 + 16);
        uint32_t *v2 = (uint32_t *)store_scratch(m, SCR_MM_V2, (size_t)count * 4 + 16);
        // pages of each namespace's run, scanned into its base page
        int64_t *part = (int64_t *)store_scratch(m, SCR_MM_POS, (size_t)(count + 1) * 16);
        void *tmp = store_scratch(m, SCR_MM_TMP, tb);
        if (!root || !k2 || !v2 || !part || !tmp)
            return fail(AKASHIC_ENOMEM, "compact: out of device memory");
        int64_t *pos = part + count + 1;
        CUDA_TRY(launch_mm_roots(ids, count, parent, root, st));
        // order (namespace, group root, chunk ID): the list is in ID order;
        // stable sorts by root, then by namespace
        bool alt = false;
        CUDA_TRY(radix_sort_pairs(root, ids, k2, v2, count, 32, tmp, tb, st, &alt, &ph.launches));
        uint32_t *sid = alt ? v2 : ids, *spare_v = alt ? ids : v2;
        uint32_t *nk = alt ? root : k2;
        CUDA_TRY(launch_mm_ns_keys(sid, count, row_of, ns_row, nsk, st));
        bool alt2 = false;
        CUDA_TRY(radix_sort_pairs(nsk, sid, nk, spare_v, count, 32, tmp, tb, st, &alt2,
                                  &ph.launches));
        const uint32_t *order = alt2 ? spare_v : sid;
        const uint32_t *ns_sorted = alt2 ? nk : nsk;
        // every namespace starts on a fresh page (compaction never mixes
        // tenants or sessions)
        CUDA_TRY(launch_mm_part_pages(ns_sorted, count, m->per_page, part, st));
        CUDA_TRY(scan_exclusive(part, pos, count, tmp, tb, st, &ph.launches));
        CUDA_TRY(cudaMemcpyAsync(&new_pages, pos + count, 8, cudaMemcpyDeviceToHost, st));
        AK_TRY(check_status(m, st, "compact"));
        AK_TRY(mm_ensure_pages(m, m->next_page + new_pages + 1, st));
        CUDA_TRY(launch_mm_release_repack(mm_tables(m), pages, cand, order, ns_sorted, pos, count,
                                          row_of, m->page_of.as<int32_t>(), m->next_page,
                                          m->per_page, st));
        ph.launches += 3 + (pages > 0) + 1;
        m->next_page += new_pages;
        m->moves += count;
    } else {
        CUDA_TRY(launch_mm_release_repack(t, pages, cand, nullptr, nullptr, nullptr, 0, row_of,
                                          m->page_of.as<int32_t>(), m->next_page, m->per_page,
                                          st));
        ph.launches += 1;
    }
    if (released) *released = n_rel;
    return check_status(m, st, "compact");
}

akashic_status_t akashic_mem_page_stats(akashic_mem_t *m, int64_t *out) {
    g_last_error.clear();
    if (!m || !out) return fail(AKASHIC_EINVAL, "page_stats: NULL argument");
    DeviceGuard g(m->device);
    unsigned long long *d = (unsigned long long *)store_scratch(m, SCR_MM_TMP, 64);
    if (!d) return fail(AKASHIC_ENOMEM, "page_stats: out of device memory");
    CUDA_TRY(launch_mm_stats(mm_tables(m), m->next_page, d, 0));
    unsigned long long h[3] = {0, 0, 0};
    CUDA_TRY(cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost));
    out[0] = (int64_t)h[0];
    out[1] = (int64_t)h[1];
    out[2] = (int64_t)h[2];
    out[3] = m->appended + m->moves;
    out[4] = m->appended;
    return AKASHIC_OK;
}

akashic_status_t akashic_mem_export_pages(akashic_mem_t *m, int32_t *page_of, void *stream) {
    g_last_error.clear();
    if (!m || !page_of) return fail(AKASHIC_EINVAL, "export_pages: NULL argument");
    DeviceGuard g(m->device);
    CUDA_TRY(launch_by_id(m->page_of.as<int32_t>(), m->row_of.as<int32_t>(), m->n, page_of,
                          (cudaStream_t)stream));
    return AKASHIC_OK;
}
}  // extern "C"

// Orders `st` after every earlier table build (any stream); called with
// table_mu held, before the tables are read or extended.
static akashic_status_t wait_tables(akashic_mem *m, cudaStream_t st) {
    if (m->table_ev) CUDA_TRY(cudaStreamWaitEvent(st, m->table_ev, 0));
    return AKASHIC_OK;
}

// Records the end of a table build on `st` (table_mu held).
static akashic_status_t tables_built(akashic_mem *m, cudaStream_t st) {
    if (!m->table_ev) CUDA_TRY(cudaEventCreateWithFlags(&m->table_ev, cudaEventDisableTiming));
    CUDA_TRY(cudaEventRecord(m->table_ev, st));
    return AKASHIC_OK;
}

// Mass levels 0..H of the row bounds (level 0 all ones), extended as needed.
// Room for the largest hop count is taken at once, so extending the levels
// never moves a buffer that a retrieve on another stream may be reading.
// table_mu held.
static akashic_status_t ensure_mass(akashic_mem *m, const HopPlan &hp, int H, cudaStream_t st) {
    const int64_t n = m->n;
    AK_TRY(wait_tables(m, st));
    if (m->mass_n != n) m->mass_levels = -1;
    if (m->mass_levels >= H) return AKASHIC_OK;
    const size_t lv = (size_t)(AKASHIC_MAX_HOPS + 1) * n * 4;
    if (m->mass_levels < 0 || m->mass_up.cap < lv) {
        AK_TRY(ensure_spare(m->mass_up, lv));
        AK_TRY(ensure_spare(m->mass_dn, lv));
        AK_TRY(ensure_spare(m->mass_zero, (size_t)n * 4));
        AK_TRY(ensure_spare(m->mass_vu, (size_t)(m->n_split + 1) * 4));
        AK_TRY(ensure_spare(m->mass_vl, (size_t)(m->n_split + 1) * 4));
        CUDA_TRY(cudaMemsetAsync(m->mass_zero.p, 0, (size_t)n * 4, st));
        CUDA_TRY(launch_fill_f32(m->mass_up.as<float>(), n, 1.f, st));
        CUDA_TRY(launch_fill_f32(m->mass_dn.as<float>(), n, 1.f, st));
        m->mass_levels = 0;
        m->mass_n = n;
    }
    const cudaError_t e = launch_mass_levels(hp, m->mass_levels + 1, H, m->mass_up.as<float>(),
                                             m->mass_dn.as<float>(), m->mass_zero.as<float>(),
                                             m->mass_vu.as<float>(), m->mass_vl.as<float>(), st);
    m->mass_levels = -1;
    AK_TRY(tables_built(m, st));
    CUDA_TRY(e);
    m->mass_levels = H;
    return AKASHIC_OK;
}

// The candidate rows and their reach coefficients for H >= 2 hops (after the
// mass levels).  A level is never rewritten while the graph stays the same, so
// a call with another hop count only adds levels that no other call reads yet.
// Every buffer is taken before the first launch, and a build that has launched
// anything ends in tables_built: levels that are announced are always ordered
// before the calls of other streams.  table_mu held.
static akashic_status_t ensure_reach(akashic_mem *m, const HopPlan &hp, int H, cudaStream_t st) {
    const int64_t n = m->n;
    AK_TRY(wait_tables(m, st));
    if (m->reach_n != n) m->reach_levels = -1;
    if (m->reach_levels >= H) return AKASHIC_OK;
    const bool fresh = m->reach_levels < 1;
    if (fresh) {
        AK_TRY(m->reach_rows.ensure(REACH_T * 4));
        AK_TRY(m->reach_t.ensure(16));
        AK_TRY(m->reach_pick.ensure((size_t)reach_pick_words() * 8));
        AK_TRY(ensure_table(m->reach_map, (size_t)n * 4, (size_t)table_rows(m) * 4));
    }
    for (int t = fresh ? 0 : m->reach_levels; t < H; ++t)
        AK_TRY(ensure_table(m->reach_c[t], (size_t)n * REACH_T * 4,
                            (size_t)table_rows(m) * REACH_T * 4));
    ReachBuild rb{};
    rb.n = n;
    rb.mup = m->mass_up.as<float>();
    rb.in_ptr = hp.in_ptr;
    rb.in_src = hp.in_src;
    rb.in_w = hp.in_w;
    rb.row_ptr = m->row_ptr.as<int64_t>();
    rb.col = m->col.as<int32_t>();
    rb.row_of = m->row_of.as<int32_t>();
    rb.w = m->w.as<float>();
    rb.rows = m->reach_rows.as<int32_t>();
    rb.t_cnt = m->reach_t.as<int>();
    rb.map = m->reach_map.as<int32_t>();
    rb.pick = m->reach_pick.as<unsigned long long>();
    cudaError_t e = cudaSuccess;
    int levels = m->reach_levels;
    if (fresh) {
        e = launch_reach_pick(rb, m->reach_c[0].as<float>(), st);
        levels = 1;
        ++m->reach_build;
    }
    for (; e == cudaSuccess && levels < H; ++levels)
        e = launch_reach_level(rb, m->reach_c[levels - 1].as<float>(),
                               m->reach_c[levels].as<float>(), st);
    m->reach_levels = -1;
    AK_TRY(tables_built(m, st));
    CUDA_TRY(e);
    m->reach_levels = levels;
    m->reach_n = n;
    return AKASHIC_OK;
}

// All that a call of width bp and H hops keeps for its candidates: its stream's
// coefficients and partials, the store's tables.  polite: only while the device
// keeps as much free as this takes, else ENOMEM and nothing taken.  table_mu held.
static akashic_status_t take_tables(akashic_mem *m, StreamScratch *sc, const HopPlan &hp, int H,
                                    int bp, bool polite, cudaStream_t st) {
    const int64_t n = m->n, room = table_rows(m);
    const size_t parts =
        (size_t)(bp == 32 ? reach_fma_parts(n) : reach_parts()) * REACH_T * bp * 4;
    const auto coef = [&](int64_t rows) {
        return bp == 32 ? (size_t)rows * REACH_T * 4 : (size_t)reach_pad_rows(rows) * REACH_T * 2;
    };
    const auto sum = [](int64_t rows) { return (size_t)reach_sum_words(rows) * 8; };
    struct {
        DevBuf *b;
        size_t now, grown;
    } own[] = {{&sc->reach_part, parts, parts},
               {bp == 32 ? &sc->coef_f : &sc->coef_hi, coef(n), coef(room)},
               {bp == 32 ? &sc->cf_sum : &sc->coef_sum, sum(n), sum(room)},
               {&sc->coef_lo, bp == 32 ? 0 : coef(n), coef(room)}};
    if (polite) {
        size_t need = 0, left = 0, all = 0;
        for (const auto &o : own) need += o.now > o.b->cap ? o.grown : 0;
        for (int t = 0; t < H; ++t)
            if ((size_t)n * REACH_T * 4 > m->reach_c[t].cap) need += (size_t)room * REACH_T * 4;
        if (need > 0) {
            CUDA_TRY(cudaMemGetInfo(&left, &all));
            if (left < 2 * need) return AKASHIC_ENOMEM;
        }
    }
    for (const auto &o : own) AK_TRY(ensure_table(*o.b, o.now, o.grown));
    return ensure_reach(m, hp, H, st);
}

// A call that uses the tables, until it has queued all that reads them.
struct TableUse {
    akashic_mem *m = nullptr;
    void take(akashic_mem *of) {
        m = of;
        m->table_users.fetch_add(1);
    }
    ~TableUse() {
        if (m) m->table_users.fetch_sub(1);
    }
};

static ReachLevels reach_levels_of(const akashic_mem *m) {
    ReachLevels c{};
    for (int t = 0; t < REACH_MAX_H; ++t) c.level[t] = m->reach_c[t].as<float>();
    return c;
}

// The pinned words a stream's plans are read back through, and its marks.
static akashic_status_t plan_words(StreamScratch *sc, cudaStream_t st) {
    if (sc->plan_host) return AKASHIC_OK;
    constexpr size_t marks = StreamScratch::TRY_KEYS * sizeof(unsigned long long);
    AK_TRY(sc->tried.ensure(marks));
    CUDA_TRY(cudaMemsetAsync(sc->tried.p, 0, marks, st));
    CUDA_TRY(cudaMallocHost((void **)&sc->plan_host, 16 + marks));
    memset(sc->plan_host, 0, 16 + marks);
    sc->told = (unsigned long long *)(sc->plan_host + 4);
    return AKASHIC_OK;
}

static akashic_status_t retrieve_impl(akashic_mem *m, const uint16_t *q, int32_t B, int32_t k,
                                      float alpha, int32_t hops, const int32_t *q_ns,
                                      int32_t sort_by_time, int64_t *ids, float *scores,
                                      int32_t *page_ids, int32_t *n_pages, void *stream) {
    if (!m) return fail(AKASHIC_EINVAL, "retrieve: NULL store");
    if (!q || !ids || !scores) return fail(AKASHIC_EINVAL, "retrieve: NULL q/ids/scores");
    if (B < 1) return fail(AKASHIC_EINVAL, "retrieve: B < 1");
    if (k < 1 || k > 64) return fail(AKASHIC_EINVAL, "retrieve: k must be in [1, 64]");
    if (k > m->n) return fail(AKASHIC_EINVAL, "retrieve: k=%d exceeds the %lld chunks", k, (long long)m->n);
    if (hops < 0 || hops > AKASHIC_MAX_HOPS) return fail(AKASHIC_EINVAL, "retrieve: hops must be in [0, 16]");
    if (!(alpha >= 0.f) || !isfinite(alpha)) return fail(AKASHIC_EINVAL, "retrieve: alpha must be finite and >= 0");
    DeviceGuard g(m->device);
    Reclaim reclaim(m);
    cudaStream_t st = (cudaStream_t)stream;
    StreamScratch *sc = scratch_for(m, stream);
    if (!sc) return fail(AKASHIC_ENOMEM, "retrieve: host allocation failed");
    const int64_t n = m->n;
    const int eff_hops = (alpha > 0.f && m->nnz > 0) ? hops : 0;
    const int sms = device_sm_count();
    for (int32_t off = 0; off < B; off += 256) {
        const int b = B - off < 256 ? B - off : 256;
        int bp = 32;
        while (bp < b) bp <<= 1;
        const int64_t tiles = score_tiles(n);
        int zrows = 0;
        const SelectPlan sp = select_plan(n, bp, k, sms);
        AK_TRY(sc->qp.ensure((size_t)bp * m->dim * 2));
        AK_TRY(sc->shift.ensure((size_t)bp * 4));
        AK_TRY(ensure_spare(sc->u, (size_t)n * bp * 4));
        AK_TRY(ensure_spare(sc->zpart, (size_t)tiles * bp * 4));
        AK_TRY(ensure_spare(sc->cand, (size_t)sp.words * 8));
        if (eff_hops >= 1) AK_TRY(ensure_spare(sc->sa, (size_t)n * bp * 4));
        if (eff_hops >= 2) AK_TRY(ensure_spare(sc->sb, (size_t)n * bp * 4));
        if (eff_hops >= 1 && m->n_segs > 0) AK_TRY(ensure_spare(sc->partial, (size_t)m->n_segs * bp * 4));
        if (eff_hops >= 1) AK_TRY(sc->words.ensure(CW_COUNT * 4));
        // a small store: the hops in full, the selection from the slab (8192
        // chunks, 16 queries, two hops 163 -> 70 us), unless the candidates may
        // do with a host wait (RC_SYNC: 256 queries 74 us, 190 with the hops)
        const bool direct = m->fuse_filter && topk_direct(n);
        const bool reach_small =
            eff_hops == 2 && bp >= 128 && !q_ns && m->reach_on && m->n_split > 0;
        // row bounds, for the candidates and for the last hop (fused filter only)
        const bool bounds =
            eff_hops >= 1 && m->fuse_filter && m->hop_prune && (!direct || reach_small);
        const bool prune = bounds && !direct;
        if (bounds) {
            AK_TRY(ensure_spare(sc->rmax_u, (size_t)n * 4));
            AK_TRY(ensure_spare(sc->rmin_u, (size_t)n * 4));
            AK_TRY(ensure_spare(sc->skip_split, (size_t)(m->n_split + 1) * 4));
            AK_TRY(ensure_spare(sc->kept_rows, (size_t)n * 4));
            AK_TRY(ensure_spare(sc->kept_segs, (size_t)(m->n_segs + 1) * 4));
            AK_TRY(sc->pfloor.ensure(16));
        }
        unsigned int *ext = eff_hops >= 1 ? sc->words.as<unsigned int>() + CW_EXT : nullptr;
        int64_t *kept_count = (int64_t *)(sc->words.as<int32_t>() + CW_KEPT);
        const uint16_t *qb = q + (int64_t)off * m->dim;
        // namespace scope of this batch's queries (padding columns get -1)
        NsScope ns{};
        if (q_ns) {
            AK_TRY(sc->qns.ensure((size_t)bp * 4));
            CUDA_TRY(cudaMemsetAsync(sc->qns.p, 0xff, (size_t)bp * 4, st));
            CUDA_TRY(cudaMemcpyAsync(sc->qns.p, q_ns + off, (size_t)b * 4,
                                     cudaMemcpyDeviceToDevice, st));
            ns = NsScope{m->ns_row.as<int32_t>(), sc->qns.as<int32_t>(), nullptr};
        }
        if (m->has_dead) ns.dead = m->dead_row.as<int32_t>();
        // Without hops the top-k filter is fused into the score GEMM, which
        // then writes no slab: the bound comes from the score of every
        // stride-th row, computed first by the same kernel (same values).
        const SelectPlan sp2 = select_plan(sp.n_sample, bp, k, sms, 1);
        const bool dense_fused = eff_hops == 0 && m->fuse_filter && !direct &&
                                 sp2.off_tr == sp.off_tr &&
                                 sp2.words <= sp.words;
        unsigned long long *ws = sc->cand.as<unsigned long long>();
        ColumnRecompute rc{};
        HopPlan hp{};
        hp.split = m->split;
        hp.in_ptr = m->in_ptr.as<int64_t>();
        hp.in_src = m->in_src.as<int32_t>();
        hp.in_w = m->in_w.as<float>();
        hp.n = n;
        hp.n_split_rows = m->n_split;
        hp.split_row = m->split_row.as<int32_t>();
        hp.split_slot0 = m->split_slot0.as<int64_t>();
        hp.n_segs = m->n_segs;
        hp.seg_e0 = m->seg_e0.as<int64_t>();
        hp.seg_e1 = m->seg_e1.as<int64_t>();
        hp.seg_slot = m->seg_slot.as<int32_t>();
        hp.split_order = m->split_order.as<int32_t>();
        hp.slot_split = m->slot_split.as<int32_t>();
        // How a call with two to four hops gets its candidates' scores without
        // running the hops (each form's plan, on the device, may still send the
        // call through them):
        //   RC_SYNC  two hops, 65 queries and more: on the tensor cores; the host
        //            waits for the plan before it queues the hops (or not)
        //   RC_MMA   other hop counts, or 33 to 64 queries: the same, with the
        //            score in fp32 and the hops queued behind; their kernels
        //            return at once when the plan says the candidates suffice
        //            (which it does not for sharp temperatures: REACH_SPLIT_SHIFT)
        //   RC_FMA   at most 32 queries: in fp32 on the CUDA cores, then the hops
        //            likewise
        // The first builds the graph-only coefficients at once; they cost about
        // what the hops cost over 128 columns a level past the first, far less
        // than the hops of such a batch.  For the others they are built once the
        // hops have cost that much since the graph changed, and later where the
        // tables of the graphs before did not pay (table_turn), so that a graph
        // that changes every few calls soon costs no more than the hops.  One GB300,
        // hops -> candidates on a graph that stays: 1,048,576 chunks, 1 query, two
        // hops 1533 -> 440 us (the call that builds the tables 3439, the fourth after
        // a change); 262,147 chunks, 24 queries 384 -> 142 (913, the fourth); 262,144
        // chunks, 200 queries, three hops 1589 -> 237 (1593, the second; 564 in fp32).
        enum { RUN_HOPS, RC_SYNC, RC_MMA, RC_FMA } mode = RUN_HOPS;
        unsigned long long now = 0;   // this call's number, and where its key's mark
        int mark = 0;                 // stands (RC_MMA, RC_FMA)
        TableUse use;
        if (bounds) {
            std::lock_guard<std::mutex> lk(m->table_mu);
            Reclaim locked(nullptr);
            akashic_status_t r = ensure_mass(m, hp, eff_hops, st);
            if (r == AKASHIC_ENOMEM && release_tables_locked(m)) r = ensure_mass(m, hp, eff_hops, st);
            AK_TRY(r);
            const bool can = !q_ns && m->reach_on && eff_hops >= 2 && eff_hops <= REACH_MAX_H;
            // (no room for the tables: the hops run, as they would without, and the
            // stream does not ask again at this size)
            if (can && eff_hops == 2 && bp >= 128 && m->n_split > 0) {
                r = sc->no_room_sync_n == n ? AKASHIC_ENOMEM
                                            : take_tables(m, sc, hp, eff_hops, bp, false, st);
                if (r == AKASHIC_ENOMEM && sc->no_room_sync_n != n && release_tables_locked(m))
                    r = take_tables(m, sc, hp, eff_hops, bp, false, st);
                if (r == AKASHIC_OK) mode = RC_SYNC;
                else if (r == AKASHIC_ENOMEM) sc->no_room_sync_n = n;
                else return r;
            } else if (can && !direct && m->n_split >= k && sc->no_room_n != n) {
                const double work = (double)eff_hops * bp, cost = REACH_T * (eff_hops - 1) + 64;
                if (m->hop_work_n != n) table_turn(m);
                m->hop_work_n = n;
                bool go = m->reach_levels >= eff_hops && m->reach_n == n;
                const bool build = !go && m->hop_work >= cost * m->table_wait;
                if (!go && !build) m->hop_work += work;
                go = go || build;
                if (go) {
                    r = take_tables(m, sc, hp, eff_hops, bp, true, st);
                    if (r == AKASHIC_ENOMEM) sc->no_room_n = n;
                    else if (r != AKASHIC_OK) return r;
                    go = r == AKASHIC_OK;
                    if (go && build) m->table_cost += cost;
                }
                // where the candidates did not suffice, the next calls like it
                // run the hops alone (try_skips)
                if (go) {
                    AK_TRY(plan_words(sc, st));
                    StreamScratch::TryKey &t = sc->try_key(m->reach_build, n, alpha, eff_hops, k,
                                                           bp == 32 ? RC_FMA : RC_MMA);
                    mark = (int)(&t - sc->keys);
                    now = ((unsigned long long)t.number << 32) | t.calls++;
                    go = !try_skips(((volatile unsigned long long *)sc->told)[mark], now);
                }
                if (go) mode = bp == 32 ? RC_FMA : RC_MMA;
                if (go) m->table_saved += work;
            }
            g_last_error.clear();
            if (mode != RUN_HOPS) use.take(m);
        }
        // on the tensor cores the candidates' pass loads u - m as split bf16,
        // which the score GEMM writes in the bytes of the fp32 slab (hi [n][bp],
        // then lo [n][bp])
        const bool split_u = mode == RC_SYNC || mode == RC_MMA;
        // (the hops queued behind; the call's word says whether to skip the rest)
        const bool queued = mode == RC_MMA || mode == RC_FMA;
        const int32_t *skip = queued ? sc->words.as<int32_t>() + CW_SKIP : nullptr;
        uint16_t *u_hi = split_u ? sc->u.as<uint16_t>() : nullptr;
        uint16_t *u_lo = split_u ? u_hi + (size_t)n * bp : nullptr;
        auto score_fp32 = [&](int *launches, const int32_t *done) -> cudaError_t {
            return launch_score(m->emb.as<uint16_t>(), n, m->dim, sc->qp.as<uint16_t>(), bp,
                                sc->shift.as<float>(), m->tau, sc->u.as<float>(),
                                sc->zpart.as<float>(), m->status.as<int>(), st, launches, &zrows,
                                ns.dead, bounds ? sc->rmax_u.as<float>() : nullptr,
                                bounds ? sc->rmin_u.as<float>() : nullptr, b,
                                bounds ? ext : nullptr, done);
        };
        {
            PhaseScope ph(m, AKASHIC_PHASE_SCORE, st);
            // with the row bounds (never with the dense fused filter) the
            // score GEMM's epilogue reduces u's row extremes into the call's
            // words, which are zeroed here
            CUDA_TRY(launch_prep_queries(qb, b, bp, m->dim, m->tau, m->max_norm.as<float>(),
                                         sc->qp.as<uint16_t>(), sc->shift.as<float>(),
                                         m->status.as<int>(), st,
                                         sc->words.as<unsigned int>(),
                                         eff_hops >= 1 ? CW_COUNT : 0, CW_SKIP,
                                         queued ? sc->tried.as<unsigned long long>() + mark : nullptr,
                                         now));
            ph.launches += 1;
            if (split_u)
                CUDA_TRY(launch_score_split(m->emb.as<uint16_t>(), n, m->dim,
                                            sc->qp.as<uint16_t>(), bp, sc->shift.as<float>(),
                                            m->tau, u_hi, u_lo, sc->zpart.as<float>(),
                                            m->status.as<int>(), st, &ph.launches, &zrows, ns.dead,
                                            sc->rmax_u.as<float>(), sc->rmin_u.as<float>(), b,
                                            ext, skip));
            else if (!dense_fused)
                CUDA_TRY(score_fp32(&ph.launches, nullptr));
        }
        if (dense_fused) {
            {
                PhaseScope ps(m, AKASHIC_PHASE_SELECT, st);
                AK_TRY(ensure_spare(sc->samp, (size_t)sp.n_sample * bp * 4));
                AK_TRY(ensure_spare(sc->ext_s, (size_t)sp.n_sample * 4));
                AK_TRY(ensure_spare(sc->zsamp, (size_t)score_tiles(sp.n_sample) * bp * 4));
                CUDA_TRY(launch_ext_sample(m->ext_of.as<int32_t>(), sp.n_sample, sp.stride,
                                           sc->ext_s.as<int32_t>(), st));
                NsScope ns_samp{};
                if (q_ns) {
                    AK_TRY(ensure_spare(sc->ns_s, (size_t)sp.n_sample * 4));
                    CUDA_TRY(launch_ext_sample(m->ns_row.as<int32_t>(), sp.n_sample, sp.stride,
                                               sc->ns_s.as<int32_t>(), st));
                    ns_samp = NsScope{sc->ns_s.as<int32_t>(), sc->qns.as<int32_t>(), nullptr};
                }
                if (m->has_dead) {
                    AK_TRY(ensure_spare(sc->dead_s, (size_t)sp.n_sample * 4));
                    CUDA_TRY(launch_ext_sample(m->dead_row.as<int32_t>(), sp.n_sample, sp.stride,
                                               sc->dead_s.as<int32_t>(), st));
                    ns_samp.dead = sc->dead_s.as<int32_t>();
                }
                CUDA_TRY(launch_score_sample(m->emb.as<uint16_t>(), sp.n_sample, sp.stride, m->dim,
                                             sc->qp.as<uint16_t>(), bp, sc->shift.as<float>(),
                                             m->tau, sc->samp.as<float>(), sc->zsamp.as<float>(),
                                             m->status.as<int>(), st, &ps.launches));
                CUDA_TRY(launch_sample_bound(sp2, sc->samp.as<float>(), b, sc->ext_s.as<int32_t>(),
                                             ws, st, &ps.launches, 4u, ns_samp));
                ps.launches += 1;
            }
            PhaseScope ph(m, AKASHIC_PHASE_SCORE, st);
            CUDA_TRY(launch_score_filter(m->emb.as<uint16_t>(), n, m->dim, sc->qp.as<uint16_t>(),
                                         bp, b, sc->shift.as<float>(), m->tau,
                                         sc->zpart.as<float>(), m->ext_of.as<int32_t>(),
                                         ws + sp.off_bound, (unsigned int *)(ws + sp.off_cnt),
                                         ws + sp.off_buf, sp.cap, ns, m->status.as<int>(), st,
                                         &ph.launches, &zrows));
            rc.kind = 2;
            rc.emb = m->emb.as<uint16_t>();
            rc.qp = sc->qp.as<uint16_t>();
            rc.dim = m->dim;
            rc.tau = m->tau;
            rc.shift = sc->shift.as<float>();
            rc.dst = sc->u.as<float>();
        }
        const float *fin = sc->u.as<float>();
        bool reached = false;   // the buffers hold every candidate
        if (eff_hops >= 1) {
            float *bufs[2] = {sc->sa.as<float>(), sc->sb.as<float>()};
            rc.u = sc->u.as<float>();
            rc.in_ptr = hp.in_ptr;
            rc.in_src = hp.in_src;
            rc.in_w = hp.in_w;
            rc.alpha = alpha;
            // the row bounds of the last hop's output
            const RowBounds rb{sc->rmax_u.as<float>(), sc->rmin_u.as<float>(),
                               m->mass_up.as<float>(), m->mass_dn.as<float>(), ext, n, eff_hops,
                               alpha};
            // The hops without running them: when every row whose upper bound
            // reaches the floor (here the k-th largest lower bound) is a
            // candidate with reach coefficients, their final scores come from
            // one pass over u and they alone are the selection's candidates.
            bool reach_done = false;
            if (mode != RUN_HOPS) {
                {
                    PhaseScope ph(m, AKASHIC_PHASE_BOUND, st);
                    AK_TRY(plan_words(sc, st));
                    AK_TRY(sc->reach_plan.ensure(REACH_PLAN_INTS * 4));
                    ReachFlags rf{};
                    rf.u0 = rb.u0;
                    rf.l0 = rb.l0;
                    rf.mup = rb.mup;
                    rf.mdn = rb.mdn;
                    rf.ext = ext;
                    rf.n = n;
                    rf.H = eff_hops;
                    rf.alpha = alpha;
                    rf.rows = m->reach_rows.as<int32_t>();
                    rf.k = k;
                    rf.map = m->reach_map.as<int32_t>();
                    rf.t_cnt = m->reach_t.as<int>();
                    rf.ws = sc->words.as<int32_t>() + CW_REACH;
                    rf.plan = sc->reach_plan.as<int32_t>();
                    rf.skip = skip;
                    if (queued) {
                        rf.tried = sc->tried.as<unsigned long long>() + mark;
                        rf.told = sc->told + mark;
                        rf.again = now + TRY_AGAIN;
                    }
                    rf.shift = mode == RC_MMA ? sc->shift.as<float>() : nullptr;
                    rf.bp = bp;
                    CUDA_TRY(launch_reach_flags(rf, st, &ph.launches));
                    if (mode == RC_SYNC) {
                        if (!sc->plan_ev)
                            CUDA_TRY(cudaEventCreateWithFlags(&sc->plan_ev,
                                                              cudaEventDisableTiming));
                        CUDA_TRY(cudaMemcpyAsync(sc->plan_host, sc->reach_plan.p, 8,
                                                 cudaMemcpyDeviceToHost, st));
                        CUDA_TRY(cudaEventRecord(sc->plan_ev, st));
                    }
                }
                // The candidates' pass is queued before the host learns the
                // plan (its kernels return at once when the plan says the
                // hops run), so the GPU goes on while the host waits.  Every
                // candidate's packed coefficients are kept while the graph,
                // alpha and the hop count stay the same.
                PhaseScope ph(m, AKASHIC_PHASE_LAST_HOP, st);
                const int32_t *plan = sc->reach_plan.as<int32_t>();
                unsigned int *cnt = (unsigned int *)(ws + sp.off_cnt);
                if (mode == RC_FMA) {
                    if (sc->cf_build != m->reach_build || sc->cf_alpha != alpha ||
                        sc->cf_H != eff_hops || sc->cf_n != n) {
                        CUDA_TRY(launch_reach_combine(reach_levels_of(m), n, eff_hops, alpha,
                                                      sc->coef_f.as<float>(),
                                                      sc->cf_sum.as<double>(), st));
                        ph.launches += 2;
                        sc->cf_build = m->reach_build;
                        sc->cf_alpha = alpha;
                        sc->cf_H = eff_hops;
                        sc->cf_n = n;
                    }
                    CUDA_TRY(launch_reach_fma(sc->u.as<float>(), bp, b, n, sc->coef_f.as<float>(),
                                              sc->cf_sum.as<double>(), ext, plan,
                                              m->reach_rows.as<int32_t>(),
                                              m->ext_of.as<int32_t>(),
                                              sc->reach_part.as<float>(), cnt, ws + sp.off_buf,
                                              sp.cap, st, &ph.launches));
                } else {
                    if (sc->coef_build != m->reach_build || sc->coef_alpha != alpha ||
                        sc->coef_H != eff_hops || sc->coef_n != n) {
                        CUDA_TRY(launch_reach_pack(reach_levels_of(m), n, eff_hops, alpha,
                                                   sc->coef_hi.as<uint16_t>(),
                                                   sc->coef_lo.as<uint16_t>(),
                                                   sc->coef_sum.as<double>(), st));
                        ph.launches += 2;
                        sc->coef_build = m->reach_build;
                        sc->coef_alpha = alpha;
                        sc->coef_H = eff_hops;
                        sc->coef_n = n;
                    }
                    CUDA_TRY(launch_reach_scores(u_hi, u_lo, sc->shift.as<float>(), bp, b, n,
                                                 sc->coef_hi.as<uint16_t>(),
                                                 sc->coef_lo.as<uint16_t>(),
                                                 sc->coef_sum.as<double>(), plan,
                                                 m->reach_rows.as<int32_t>(),
                                                 m->ext_of.as<int32_t>(),
                                                 sc->reach_part.as<float>(), cnt, ws + sp.off_buf,
                                                 sp.cap, m->status.as<int>(), st, &ph.launches));
                }
                if (mode == RC_SYNC) {
                    ph.end();
                    CUDA_TRY(cudaEventSynchronize(sc->plan_ev));
                    reached = reach_done = sc->plan_host[0] == 1;
                    if (reach_done) rc = ColumnRecompute{};
                } else {
                    hp.done = plan;
                }
            }
            // the hops read u in fp32 (the same scores again)
            if (split_u && !reach_done) {
                PhaseScope ph(m, AKASHIC_PHASE_SCORE, st);
                CUDA_TRY(score_fp32(&ph.launches, hp.done));
            }
            for (int h = 0; h < eff_hops && !reach_done; ++h) {
                float *out = bufs[h & 1];
                const bool last = m->fuse_filter && !direct && h == eff_hops - 1;
                if (last) {
                    // Top-k filter fused into the last hop, its bound from the
                    // hop's own values on the row sample.
                    {
                        PhaseScope ps(m, AKASHIC_PHASE_SELECT, st);
                        CUDA_TRY(launch_hop_sample(hp, sp, sc->u.as<float>(), fin, alpha, ns,
                                                   (uint32_t *)(ws + sp.off_tr), st,
                                                   &ps.launches));
                        CUDA_TRY(launch_sample_bound(sp, nullptr, b, m->ext_of.as<int32_t>(), ws,
                                                     st, &ps.launches, 0u, ns, hp.done));
                    }
                    if (prune) {
                        PhaseScope ps(m, AKASHIC_PHASE_BOUND, st);
                        // floor: the filter bounds', raised without a namespace
                        // scope to the k-th largest lower bound of the heaviest
                        // split rows (where the top scores lie)
                        const int64_t n_lb = m->n_split < 1024 ? m->n_split : 1024;
                        AK_TRY(ensure_spare(sc->keep_scr, (size_t)keep_words(hp) * 4));
                        CUDA_TRY(launch_prune_floor(ws + sp.off_bound, b, rb,
                                                    q_ns ? nullptr : hp.split_row,
                                                    hp.split_order, n_lb, k,
                                                    sc->pfloor.as<float>(), hp.done, st));
                        // with a scope, each namespace of the batch gets its own
                        // floor (its rows can only be selected by its queries)
                        NsFloors nf{};
                        if (q_ns) {
                            AK_TRY(sc->nsf.ensure(4096));
                            int32_t *tags = sc->nsf.as<int32_t>();
                            float *tag_floor = (float *)(tags + PF_TAGS);
                            int *n_tags = (int *)(tag_floor + PF_TAGS);
                            CUDA_TRY(launch_ns_floors(ws + sp.off_bound, sc->qns.as<int32_t>(), b,
                                                      rb, m->ns_row.as<int32_t>(), hp.split_row,
                                                      hp.split_order, m->n_split, k, tags, n_tags,
                                                      tag_floor, st));
                            nf = NsFloors{m->ns_row.as<int32_t>(), tags, n_tags, tag_floor};
                            ps.launches += m->n_split > 0 ? 2 : 1;
                        }
                        CUDA_TRY(launch_keep(hp, rb, sc->pfloor.as<float>(), q_ns ? &nf : nullptr,
                                             sc->skip_split.as<int32_t>(),
                                             sc->kept_rows.as<int32_t>(),
                                             sc->kept_segs.as<int32_t>(), kept_count,
                                             sc->keep_scr.as<int32_t>(), st, &ps.launches));
                        ps.launches += 1;
                    }
                }
                const HopFilter flt{m->ext_of.as<int32_t>(), ws + sp.off_bound,
                                    (unsigned int *)(ws + sp.off_cnt), ws + sp.off_buf, sp.cap,
                                    ns};
                const HopBound hb{sc->skip_split.as<int32_t>(), sc->kept_rows.as<int32_t>(),
                                  kept_count, sc->kept_segs.as<int32_t>()};
                PhaseScope ph(m, last ? AKASHIC_PHASE_LAST_HOP : AKASHIC_PHASE_PROPAGATE, st);
                CUDA_TRY(launch_hop(hp, sc->u.as<float>(), fin, out, bp, alpha,
                                    sc->partial.as<float>(),
                                    sc->words.as<int>() + CW_QUEUE + 2 * h, last ? &flt : nullptr, st, &ph.launches,
                                    (last && prune) ? &hb : nullptr));
                if (last) {
                    rc.kind = 1;
                    rc.prev = fin;
                    rc.dst = out;
                }
                fin = out;
            }
        }
        {
            PhaseScope ph(m, AKASHIC_PHASE_SELECT, st);
            int32_t *pids = page_ids ? page_ids + (int64_t)off * k : nullptr;
            int32_t *npg = n_pages ? n_pages + off : nullptr;
            if (direct && !reached)
                CUDA_TRY(launch_topk_direct(fin, n, bp, b, k, sc->zpart.as<float>(), zrows,
                                            m->ext_of.as<int32_t>(), m->row_of.as<int32_t>(),
                                            m->page_of.as<int32_t>(), ids + (int64_t)off * k,
                                            scores + (int64_t)off * k, pids, npg,
                                            m->status.as<int>(), ns, sort_by_time, st,
                                            &ph.launches));
            else if ((eff_hops >= 1 && m->fuse_filter) || dense_fused)
                CUDA_TRY(launch_topk_merge(sp, fin, b, sc->cand.as<unsigned long long>(),
                                           sc->zpart.as<float>(), zrows, m->ext_of.as<int32_t>(),
                                           m->row_of.as<int32_t>(), m->page_of.as<int32_t>(),
                                           ids + (int64_t)off * k, scores + (int64_t)off * k,
                                           pids, npg, m->status.as<int>(), &rc, ns,
                                           sort_by_time, st, &ph.launches));
            else
                CUDA_TRY(launch_select(sp, fin, b, sc->cand.as<unsigned long long>(),
                                       sc->zpart.as<float>(), zrows, m->ext_of.as<int32_t>(),
                                       m->row_of.as<int32_t>(), m->page_of.as<int32_t>(),
                                       ids + (int64_t)off * k, scores + (int64_t)off * k, pids,
                                       npg, m->status.as<int>(), ns, sort_by_time, st,
                                       &ph.launches));
        }
    }
    return AKASHIC_OK;
}

extern "C" {

akashic_status_t akashic_mem_export_csr(akashic_mem_t *m, int64_t *n_rows, int64_t *nnz,
                                        int64_t *row_ptr, int32_t *col, float *aff, float *w,
                                        void *stream) {
    g_last_error.clear();
    if (!m) return fail(AKASHIC_EINVAL, "export: NULL store");
    if (n_rows) *n_rows = m->n;
    if (nnz) *nnz = m->nnz;
    if (!row_ptr && !col && !aff && !w) return AKASHIC_OK;
    DeviceGuard g(m->device);
    cudaStream_t st = (cudaStream_t)stream;
    if (row_ptr)
        CUDA_TRY(cudaMemcpyAsync(row_ptr, m->row_ptr.p, (size_t)(m->n + 1) * 8,
                                 cudaMemcpyDeviceToDevice, st));
    if (m->nnz > 0) {
        if (col) CUDA_TRY(cudaMemcpyAsync(col, m->col.p, (size_t)m->nnz * 4, cudaMemcpyDeviceToDevice, st));
        if (aff) CUDA_TRY(cudaMemcpyAsync(aff, m->aff.p, (size_t)m->nnz * 4, cudaMemcpyDeviceToDevice, st));
        if (w) CUDA_TRY(cudaMemcpyAsync(w, m->w.p, (size_t)m->nnz * 4, cudaMemcpyDeviceToDevice, st));
    }
    CUDA_TRY(cudaStreamSynchronize(st));
    return AKASHIC_OK;
}

akashic_status_t akashic_mem_set_profiling(akashic_mem_t *m, int32_t on) {
    if (!m) return fail(AKASHIC_EINVAL, "set_profiling: NULL store");
    m->prof = on != 0;
    return AKASHIC_OK;
}

akashic_status_t akashic_mem_phase_times(akashic_mem_t *m, float *ms, int32_t *launches) {
    if (!m) return fail(AKASHIC_EINVAL, "phase_times: NULL store");
    DeviceGuard g(m->device);
    std::vector<ProfRec> recs;
    {
        std::lock_guard<std::mutex> lk(m->mu);
        recs.swap(m->recs);
    }
    for (int p = 0; p < AKASHIC_PHASE_COUNT; ++p) {
        if (ms) ms[p] = 0.f;
        if (launches) launches[p] = 0;
    }
    akashic_status_t rc = AKASHIC_OK;
    for (auto &r : recs) {
        float t = 0.f;
        cudaError_t e = cudaEventSynchronize(r.b);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t, r.a, r.b);
        if (e != cudaSuccess) {
            cudaGetLastError();
            rc = fail(AKASHIC_ECUDA, "phase_times: %s", cudaGetErrorString(e));
        }
        if (r.phase >= 0 && r.phase < AKASHIC_PHASE_COUNT) {
            if (ms) ms[r.phase] += t;
            if (launches) launches[r.phase] += r.launches;
        }
    }
    std::lock_guard<std::mutex> lk(m->mu);
    for (auto &r : recs) {
        m->ev_pool.push_back(r.a);
        m->ev_pool.push_back(r.b);
    }
    return rc;
}

}  // extern "C"
