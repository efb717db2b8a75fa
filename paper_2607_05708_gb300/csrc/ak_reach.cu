// Scores of the top-k candidates for two to four hops, without the hops.
//
// Unrolling the hop recursion s^(h) = u + alpha R^T s^(h-1) (the relation
// propagation of §4.1, R_ki = w(k -> i)) gives, for a row j,
//   s^(H)_j = u_j + sum_{t=1..H} alpha^t sum_k C_t[k][j] u_k,
//   C_1[k][j] = w(k -> j),   C_t = R C_{t-1},
// with reach coefficients C_t that depend on the graph alone.  The row
// bounds of the last hop (ak_graph.cu) prove that only the rows whose
// upper bound reaches the top-k floor can be selected; when all of them lie
// in a small set of heavy candidate rows whose coefficients are kept, their
// final scores for every query come from one pass over the score slab u,
// and the hops are not run.  The selection is the same as the hops' up to
// scores that are equal within the two paths' roundings: sums in another order, and
// on the tensor cores coefficients and u as pairs of bf16 (16 bits; see
// REACH_SPLIT_SHIFT).
#include <cuda_bf16.h>

#include "ak_common.cuh"
#include "ak_sm100.cuh"

namespace ak {

// ------------------------------------------------------------------ graph-only
// Candidates: the REACH_T rows of largest upper mass mup[1] + mup[2],
// whatever the hop count (so that the levels of one hop count serve the others);
// ties to the lower row.  Mass counts, not in-degree: a row with few in-edges
// from chunks that link to little else outranks many hubs.  A histogram of the
// masses' upper bits gives a threshold that at least REACH_T rows reach, those
// rows are collected, and one CTA sorts them.  More than PICK_MAX of them (all
// within 3% of the last): no candidates, as the plan would hardly ever take
// them.
constexpr int PICK_SHIFT = 18, PICK_BINS = 1 << (31 - PICK_SHIFT), PICK_MAX = 4096;
__device__ __forceinline__ uint32_t mass_bits(const float *__restrict__ mup, int64_t n, int64_t r) {
    return __float_as_uint(mup[n + r] + mup[2 * n + r]);   // >= 0: ordered like the values
}

__global__ __launch_bounds__(256) void k_mass_hist(const float *__restrict__ mup, int64_t n,
                                                   int *__restrict__ hist) {
    __shared__ int h[PICK_BINS];
    for (int i = threadIdx.x; i < PICK_BINS; i += 256) h[i] = 0;
    __syncthreads();
    for (int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x; r < n; r += (int64_t)gridDim.x * 256)
        atomicAdd(&h[mass_bits(mup, n, r) >> PICK_SHIFT], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < PICK_BINS; i += 256)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// The lower edge of the highest bin with at least REACH_T rows in it and above
// (0 if there are fewer rows): every CTA finds it, then collects its rows.
__global__ __launch_bounds__(256) void k_mass_collect(const float *__restrict__ mup, int64_t n,
                                                      const int *__restrict__ hist,
                                                      unsigned long long *__restrict__ keys,
                                                      int *__restrict__ count) {
    __shared__ int sum[256];
    __shared__ int bin_s;
    constexpr int PER = PICK_BINS / 256;
    const int t = threadIdx.x;
    int mine = 0;                       // thread t: bins from the top, PER a thread
    for (int i = 0; i < PER; ++i) mine += hist[PICK_BINS - 1 - (t * PER + i)];
    sum[t] = mine;
    if (t == 0) bin_s = 0;
    __syncthreads();
    int above = 0;
    for (int i = 0; i < t; ++i) above += sum[i];
    if (above < REACH_T && above + mine >= REACH_T) {
        int b = PICK_BINS - 1 - t * PER;
        for (int i = 0; i < PER; ++i, --b) {
            above += hist[b];
            if (above >= REACH_T) break;
        }
        bin_s = b;
    }
    __syncthreads();
    // (rows without mass are nobody's candidates)
    const uint32_t lo = bin_s > 0 ? (uint32_t)bin_s << PICK_SHIFT : 1u;
    for (int64_t r = (int64_t)blockIdx.x * 256 + t; r < n; r += (int64_t)gridDim.x * 256) {
        const uint32_t m = mass_bits(mup, n, r);
        if (m < lo) continue;
        const int p = atomicAdd(count, 1);
        if (p < PICK_MAX)
            keys[p] = ((unsigned long long)m << 32) | (unsigned long long)(~(uint32_t)r);
    }
}

__global__ __launch_bounds__(1024) void k_reach_pick(const unsigned long long *__restrict__ keys,
                                                      const int *__restrict__ count,
                                                      int32_t *__restrict__ rows,
                                                      int *__restrict__ t_out) {
    __shared__ unsigned long long key[PICK_MAX];
    const int tid = threadIdx.x, m = *count;
    if (m > PICK_MAX) {
        if (tid == 0) *t_out = 0;
        return;
    }
    for (int i = tid; i < PICK_MAX; i += 1024) key[i] = i < m ? keys[i] : 0ull;
    __syncthreads();
    // descending bitonic sort
    for (int size = 2; size <= PICK_MAX; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = tid; i < PICK_MAX; i += 1024) {
                const int other = i ^ stride;
                if (other > i) {
                    const unsigned long long a = key[i], b = key[other];
                    const bool desc = (i & size) == 0;
                    if (desc ? a < b : a > b) {
                        key[i] = b;
                        key[other] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
    const int T = m < REACH_T ? m : REACH_T;
    if (tid < T) rows[tid] = (int32_t)~(uint32_t)(key[tid] & 0xffffffffull);
    if (tid == 0) *t_out = T;
}

__global__ void k_reach_map(const int32_t *__restrict__ rows, const int *__restrict__ t_cnt,
                            int32_t *__restrict__ map) {
    if ((int)threadIdx.x < *t_cnt) map[rows[threadIdx.x]] = (int32_t)threadIdx.x;
}

// C_1[k][t] = w(k -> rows[t]): the candidate's in-edges, C1_CTAS CTAs each (with
// one, a hub's 8 * 10^5 edges took 0.8 ms of a build on 1,048,576 chunks).
constexpr int C1_CTAS = 16;
__global__ void k_reach_c1(const int32_t *__restrict__ rows, const int *__restrict__ t_cnt,
                           const int64_t *__restrict__ in_ptr, const int32_t *__restrict__ in_src,
                           const float *__restrict__ in_w, float *__restrict__ C1) {
    const int t = blockIdx.x;
    if (t >= *t_cnt) return;
    const int64_t j = rows[t];
    for (int64_t e = in_ptr[j] + (int64_t)blockIdx.y * blockDim.x + threadIdx.x;
         e < in_ptr[j + 1]; e += (int64_t)gridDim.y * blockDim.x)
        C1[(int64_t)in_src[e] * REACH_T + t] = in_w[e];
}

// Cn[row(k)][:] = sum over k's out-edges (k -> i) of w * Cp[row(i)][:]: one
// warp per chunk ID k, four columns per lane (a float4), edges in CSR order.
__global__ void k_reach_spmm(const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                             const float *__restrict__ w, const int32_t *__restrict__ row_of,
                             int64_t n, const float *__restrict__ Cp, float *__restrict__ Cn) {
    static_assert(REACH_T == 128, "four columns per lane");
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n; k += nw) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int64_t e = row_ptr[k]; e < row_ptr[k + 1]; ++e) {
            const float we = w[e];
            const float4 c =
                reinterpret_cast<const float4 *>(Cp + (int64_t)row_of[col[e]] * REACH_T)[lane];
            a.x = fmaf(we, c.x, a.x);
            a.y = fmaf(we, c.y, a.y);
            a.z = fmaf(we, c.z, a.z);
            a.w = fmaf(we, c.w, a.w);
        }
        reinterpret_cast<float4 *>(Cn + (int64_t)row_of[k] * REACH_T)[lane] = a;
    }
}

int64_t reach_pick_words() { return PICK_MAX + (PICK_BINS + 2) / 2; }

cudaError_t launch_reach_pick(const ReachBuild &rb, float *C1, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(rb.map, 0xff, (size_t)rb.n * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(C1, 0, (size_t)rb.n * REACH_T * 4, st);
    if (e != cudaSuccess) return e;
    int *hist = (int *)(rb.pick + PICK_MAX);
    e = cudaMemsetAsync(hist, 0, (PICK_BINS + 1) * 4, st);
    if (e != cudaSuccess) return e;
    const int64_t want = ceil_div<int64_t>(rb.n, 1024), sms = device_sm_count();
    const unsigned g = (unsigned)(want < 2 * sms ? want : 2 * sms);
    k_mass_hist<<<g, 256, 0, st>>>(rb.mup, rb.n, hist);
    k_mass_collect<<<g, 256, 0, st>>>(rb.mup, rb.n, hist, rb.pick, hist + PICK_BINS);
    k_reach_pick<<<1, 1024, 0, st>>>(rb.pick, hist + PICK_BINS, rb.rows, rb.t_cnt);
    k_reach_map<<<1, REACH_T, 0, st>>>(rb.rows, rb.t_cnt, rb.map);
    k_reach_c1<<<dim3(REACH_T, C1_CTAS), 256, 0, st>>>(rb.rows, rb.t_cnt, rb.in_ptr, rb.in_src, rb.in_w, C1);
    return cudaGetLastError();
}

cudaError_t launch_reach_level(const ReachBuild &rb, const float *Cp, float *Cn, cudaStream_t st) {
    k_reach_spmm<<<device_sm_count() * 8, 256, 0, st>>>(rb.row_ptr, rb.col, rb.w, rb.row_of, rb.n,
                                                        Cp, Cn);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ per call
// The plan of a call, on the device: plan[0] = 1 when the candidates
// suffice (no other row reaches the floor, at least k of them do, and at
// least k candidates exist), else 0 and the hops run; plan[1] = nk, the
// flagged count; plan[2 .. 2 + nk) the flagged slots in ascending order;
// plan[REACH_PLAN_WIDE] = 1 when one of them is 64 or above.  Run by one
// CTA of at least REACH_T threads (every thread calls it).
__device__ void reach_build_plan(const int32_t *keep, int bad, int t_cnt, int k, int32_t *plan) {
    __shared__ int pre[REACH_T];
    const int t = threadIdx.x;
    const int f = t < REACH_T && keep[t] != 0 ? 1 : 0;
    if (t < REACH_T) pre[t] = f;
    __syncthreads();
    for (int o = 1; o < REACH_T; o <<= 1) {          // inclusive scan
        const int v = t < REACH_T && t >= o ? pre[t - o] : 0;
        __syncthreads();
        if (t < REACH_T) pre[t] += v;
        __syncthreads();
    }
    if (f) plan[2 + pre[t] - 1] = t;
    if (t == REACH_T - 1) {
        const int nk = pre[t];
        plan[1] = nk;
        plan[0] = (bad == 0 && nk >= k && t_cnt >= k) ? 1 : 0;
        // a flagged slot in the upper half: the candidates' pass loads all
        // 128 coefficient rows, else the first 64
        plan[REACH_PLAN_WIDE] = nk - pre[REACH_T / 2 - 1] > 0 ? 1 : 0;
    }
}

// The floor: the k-th largest lower bound over the candidates (each query's
// k-th largest final score reaches it: those k rows score at least their lb
// for every query); every CTA evaluates it, 128 bounds ranked against each
// other (a CTA of its own that sorted 1024 hubs' bounds took 10 us more a
// call).  Then the rows whose upper bound reaches it: a candidate's slot is
// flagged, any other row counted in bad; the last CTA to finish builds the
// plan.
__global__ __launch_bounds__(256) void k_reach_flags(const ReachFlags f) {
    __shared__ int last;
    __shared__ float floor_s;
    __shared__ unsigned int lb_s[REACH_T];
    griddep_wait();
    int32_t *keep = f.ws, *bad = f.ws + REACH_T, *done = f.ws + REACH_T + 1;
    const int t_cnt = *f.t_cnt, skip = f.skip ? f.skip[0] : 0;   // (one wait for both)
    if (skip == 1) {
        if (blockIdx.x == 0 && threadIdx.x == 0) f.plan[0] = 0;
        return;
    }
    {
        const int t = threadIdx.x;
        unsigned int lb = 0u;                            // (bounds are >= 0)
        if (t < t_cnt)
            lb = __float_as_uint(row_lower_bound(f.l0, f.mdn, f.n, f.H, f.alpha, ext_lmin(f.ext),
                                                 f.rows[t]));
        if (t < REACH_T) lb_s[t] = lb;
        if (t == 0) floor_s = 0.f;
        __syncthreads();
        if (t < t_cnt) {
            int rank = 0;
            for (int i = 0; i < t_cnt; ++i) rank += lb_s[i] > lb || (lb_s[i] == lb && i < t) ? 1 : 0;
            if (rank == f.k - 1) floor_s = __uint_as_float(lb);
        }
        __syncthreads();
    }
    const float floor_ = floor_s, umax = ext_umax(f.ext);
    int nb = 0;
    auto visit = [&](int64_t j, float ub) {
        if (ub >= floor_) {
            const int32_t t = f.map[j];
            if (t >= 0) keep[t] = 1;
            else ++nb;
        }
    };
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if ((f.n & 3) == 0) {
        // four rows a thread: 16-byte loads of u's row maxima and of each
        // mass level, the bound evaluated per row as row_upper_bound does
        const int64_t n4 = f.n >> 2;
        for (int64_t q = tid; q < n4; q += stride) {
            float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int t = f.H; t >= 1; --t) {
                const float4 m =
                    __ldg(reinterpret_cast<const float4 *>(f.mup + (int64_t)t * f.n) + q);
                c.x = f.alpha * (c.x + m.x);
                c.y = f.alpha * (c.y + m.y);
                c.z = f.alpha * (c.z + m.z);
                c.w = f.alpha * (c.w + m.w);
            }
            const float4 u = reinterpret_cast<const float4 *>(f.u0)[q];
            visit(4 * q, fmaf(umax, c.x, u.x) * (1.f + 1e-5f));
            visit(4 * q + 1, fmaf(umax, c.y, u.y) * (1.f + 1e-5f));
            visit(4 * q + 2, fmaf(umax, c.z, u.z) * (1.f + 1e-5f));
            visit(4 * q + 3, fmaf(umax, c.w, u.w) * (1.f + 1e-5f));
        }
    } else {
        for (int64_t j = tid; j < f.n; j += stride)
            visit(j, row_upper_bound(f.u0, f.mup, f.n, f.H, f.alpha, umax, j));
    }
    if (nb) atomicAdd(bad, nb);
    __threadfence();                                   // flags before the count
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();                                   // every CTA's flags are visible
    const volatile int32_t *vk = keep;
    __shared__ int32_t kf[REACH_T];
    if (threadIdx.x < REACH_T) kf[threadIdx.x] = vk[threadIdx.x];
    __syncthreads();
    // (a batch whose scores spread too far for 16 bits counts as a row too many)
    const bool sharp = f.shift && !(batch_shift(f.shift, f.bp) <= REACH_SPLIT_SHIFT);
    reach_build_plan(kf, *(volatile int *)bad + (sharp ? 1 : 0), t_cnt, f.k, f.plan);
    if (f.tried && threadIdx.x == REACH_T - 1 && f.plan[0] == 0) {   // (it wrote plan[0])
        *f.tried = f.again;
        *(volatile unsigned long long *)f.told = f.again;
    }
}

cudaError_t launch_reach_flags(const ReachFlags &f, cudaStream_t st, int *launches) {
    if (f.k < 1) return cudaErrorInvalidValue;
    // four rows per thread (one where n is not a multiple of 4): a few
    // independent loads per row, so the rows in flight set the rate; a
    // quarter of the CTAs also takes three quarters of the done counter's
    // atomics off the tail
    const int64_t g = ceil_div<int64_t>(f.n, (f.n & 3) == 0 ? 1024 : 256);
    cudaError_t e =
        launch_pdl(k_reach_flags, dim3((unsigned)(g > 0 ? g : 1)), dim3(256), 0, st, f);
    if (launches) *launches += 1;
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// ------------------------------------------------------------------ tensor-core terms
// partial[cta][i][b] = sum over the CTA's rows k of coef[k][i] u[k][b] for
// every candidate slot i, on tcgen05 with split-bf16 operands:
//   coef = A_hi + A_lo,  u = B_hi + B_lo  (each lo the bf16 rounding of the
//   rest, so hi + lo holds 16 significant bits),
//   coef u ~= A_hi B_hi + A_hi B_lo + A_lo B_hi,
// three MMAs per 16-row slice into an fp32 accumulator in TMEM (the
// dropped A_lo B_lo term is below 2^-16 of the product).  u stands for
// u - m here, m = batch_u_min: most of every u is the same constant, and
//   sum_k coef[k][i] u[k][b] = m S_i + sum_k coef[k][i] (u[k][b] - m)
// with S_i the coefficients' sum in 64 bits, so the products' and the
// accumulation's errors shrink with the terms.
//   A = the combined coefficients sum_t alpha^t C_t, packed by
//       k_reach_pack as [REACH_T slots][n_pad rows] bf16 (hi, lo), loaded
//       by TMA as K-major tiles [128 slots][64 rows] in the 128-byte swizzle;
//   B = u as the score GEMM wrote it, split bf16 [n rows][BP queries] (hi,
//       lo), loaded by TMA as MN-major tiles [64 rows][BP queries]: boxes of
//       64 rows x 64 queries in the 128-byte swizzle (128 bytes a row, the
//       16-byte chunk c of row r at c ^ (r % 8)), i.e. atoms of 8 rows x 64
//       queries, the BP / 64 boxes RM_BK * 128 bytes apart.
// D[slot][query] (M = 128 slots = TMEM lanes, N = BP queries = columns).
// The tensor core's accumulation of many positive terms drifts (each add
// into the fp32 accumulator rounds the same way, ~2^-25 an MMA), so an
// accumulator takes only RM_CHUNK stages (RM_CHUNK * 12 MMAs): two
// accumulators alternate, and the flush warps add each finished one to the
// CTA's sums, which they hold in registers, with ordinary round-to-nearest
// fp32 adds while the MMAs fill the other.  (Sums kept in memory cost so much
// per flush that an accumulator took 16 stages: scores 5.6e-6 off on 1,048,576
// chunks and 256 queries, 3.8e-8 with this and u - m.)  The operands' loads carry an L2 evict-first hint;
// slots 64 and above are flushed only when the plan is wide.
// Warps: 0 TMA producer (A and B), 1 MMA issuer, 2..9 flush (warp w reads
// TMEM lanes 32 (w % 4) .., column half (w - 2) / 4).  Both operands
// arrive by TMA, so the bytes in flight are the two stages' 192 KB of
// shared memory, not registers.  Each CTA takes a contiguous range of
// 64-row stages.
constexpr int RM_BK = 64;                // store rows (K) per stage
constexpr int RM_M = REACH_T;            // candidate slots (M)
constexpr int RM_STAGES = 2;
constexpr int RM_FLUSH_W = 8;            // flush warps
constexpr int RM_THREADS = 64 + 32 * RM_FLUSH_W;
constexpr int RM_CHUNK = 2;              // stages per accumulator

template <int BP>
struct RmCfg {
    static constexpr int A_BYTES = RM_M * RM_BK * 2;             // one of hi / lo
    static constexpr int B_BYTES = BP * RM_BK * 2;               // one of hi / lo
    static constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;
    static constexpr uint32_t LBO = RM_BK * 128;                 // between query atoms
    static constexpr uint32_t SBO = 8 * 128;                     // between 8-row groups
    static constexpr int SMEM = 1024 + RM_STAGES * STAGE_BYTES + 256;
    static constexpr int PARTS = RM_FLUSH_W / 4;     // column parts of a flush
    static constexpr int TMEM_COLS = 2 * BP; // two accumulators
    static_assert(BP == 64 || BP == 128 || BP == 256, "query widths 64, 128 and 256");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

template <int BP>
__global__ __launch_bounds__(RM_THREADS, 1) void k_reach_mma(
    const __grid_constant__ CUtensorMap tmAhi, const __grid_constant__ CUtensorMap tmAlo,
    const __grid_constant__ CUtensorMap tmAhi64, const __grid_constant__ CUtensorMap tmAlo64,
    const __grid_constant__ CUtensorMap tmBhi, const __grid_constant__ CUtensorMap tmBlo,
    int64_t n, const int32_t *__restrict__ plan, float *__restrict__ partial, int *status) {
    using C = RmCfg<BP>;
    griddep_wait();
    if (plan[0] == 0) return;                          // the hops run instead
    // every flagged slot below 64: only the first 64 coefficient rows are
    // loaded (rows 64..127 of the A tiles keep whatever they hold, and
    // the accumulator rows they feed are never read)
    const bool wide = plan[REACH_PLAN_WIDE] != 0;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + RM_STAGES * C::STAGE_BYTES);
    uint64_t *empty = full + RM_STAGES;               // the MMAs' commit
    uint64_t *dfull = empty + RM_STAGES;              // [2] accumulator complete
    uint64_t *dfree = dfull + 2;                      // [2] accumulator flushed (RM_FLUSH_W)
    uint32_t *tmem_slot = (uint32_t *)(dfree + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto a_hi = [&](int s) { return smem + s * C::STAGE_BYTES; };
    auto a_lo = [&](int s) { return smem + s * C::STAGE_BYTES + C::A_BYTES; };
    auto b_hi = [&](int s) { return smem + s * C::STAGE_BYTES + 2 * C::A_BYTES; };
    auto b_lo = [&](int s) { return smem + s * C::STAGE_BYTES + 2 * C::A_BYTES + C::B_BYTES; };

    const int64_t stages_total = (n + RM_BK - 1) / RM_BK;
    const int64_t per = (stages_total + gridDim.x - 1) / gridDim.x;
    const int64_t s0 = (int64_t)blockIdx.x * per;
    const int64_t s1 = s0 + per < stages_total ? s0 + per : stages_total;
    const int64_t ns = s1 > s0 ? s1 - s0 : 0;
    const int64_t n_chunks = (ns + RM_CHUNK - 1) / RM_CHUNK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < RM_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&dfull[a], 1);
            mbar_init(&dfree[a], RM_FLUSH_W);
        }
        mbar_fence_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, C::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (lane == 0 && ns > 0) {
            // ---------------- TMA producer: A hi / lo [128 slots][64 rows],
            // B hi / lo [64 rows][BP queries] as BP / 64 boxes each
            uint32_t stage = 0, phase = 0;
            int last_par[RM_STAGES];
            for (int s = 0; s < RM_STAGES; ++s) last_par[s] = -1;
            bool ok = true;
            // both operands are read once a call: evict them first, so that
            // they do not push the CTAs' partial rows out of L2
            const uint64_t pol = l2_evict_first_policy();
            for (int64_t t = 0; t < ns; ++t) {
                if (!mbar_wait_spin(&empty[stage], phase ^ 1u, status)) {
                    ok = false;
                    break;
                }
                mbar_expect_tx(&full[stage],
                               (wide ? 2 * C::A_BYTES : C::A_BYTES) + 2 * C::B_BYTES);
                const int kx = (int)((s0 + t) * RM_BK);
                tma_load_2d_hint(a_hi(stage), wide ? &tmAhi : &tmAhi64, &full[stage], kx, 0, pol);
                tma_load_2d_hint(a_lo(stage), wide ? &tmAlo : &tmAlo64, &full[stage], kx, 0, pol);
#pragma unroll
                for (int c = 0; c < BP / 64; ++c) {
                    tma_load_2d_hint(b_hi(stage) + c * C::LBO, &tmBhi, &full[stage], 64 * c, kx,
                                     pol);
                    tma_load_2d_hint(b_lo(stage) + c * C::LBO, &tmBlo, &full[stage], 64 * c, kx,
                                     pol);
                }
                last_par[stage] = (int)phase;
                if (++stage == RM_STAGES) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (!ok)   // let every copy this thread issued land before the CTA exits
                for (int s = 0; s < RM_STAGES; ++s)
                    if (last_par[s] >= 0) mbar_wait(&full[s], (uint32_t)last_par[s], status);
        }
    } else if (warp == 1) {
        if (lane == 0 && ns > 0) {
            // ---------------- MMA issuer: three products per 16-row slice
            const uint32_t idesc = idesc_bf16_m128(BP) | IDESC_B_MN_MAJOR;
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            for (int64_t t = 0; t < ns && ok; ++t) {
                const int64_t c = t / RM_CHUNK;
                const int acc = (int)(c & 1);
                const bool first = t % RM_CHUNK == 0;
                const bool last = t % RM_CHUNK == RM_CHUNK - 1 || t == ns - 1;
                // the accumulator is free once the flush warps emptied its
                // previous chunk (c - 2)
                if (first && !mbar_wait(&dfree[acc], (uint32_t)((c >> 1) & 1) ^ 1u, status)) break;
                if (!mbar_wait_spin(&full[stage], phase, status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem_base + (uint32_t)(acc * BP);
                const uint64_t ah = sdesc_sw128(smem_u32(a_hi(stage)));
                const uint64_t al = sdesc_sw128(smem_u32(a_lo(stage)));
                const uint64_t bh = sdesc_mn_sw128(smem_u32(b_hi(stage)), C::LBO, C::SBO);
                const uint64_t bl = sdesc_mn_sw128(smem_u32(b_lo(stage)), C::LBO, C::SBO);
#pragma unroll
                for (int k = 0; k < RM_BK / 16; ++k) {
                    // A: 16 K values = 32 bytes further along the row; B: two
                    // 8-row groups further down
                    const uint64_t ao = (uint64_t)(2 * k), bo = (uint64_t)(2 * C::SBO * k) >> 4;
                    umma_bf16(d, ah + ao, bh + bo, idesc, (first && k == 0) ? 0u : 1u);
                    umma_bf16(d, ah + ao, bl + bo, idesc, 1u);
                    umma_bf16(d, al + ao, bh + bo, idesc, 1u);
                }
                umma_commit(&empty[stage]);
                if (last) umma_commit(&dfull[acc]);
                if (++stage == RM_STAGES) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    } else {
        // ---------------- flush warps: each finished accumulator into the
        // warp's share of the CTA's sums (registers), written at the end
        const int fw = warp - 2;
        const int q = warp & 3;                       // TMEM lanes 32 q ..
        const int part = fw >> 2;                     // column part
        const int slot = q * 32 + lane;
        constexpr int PW = BP / C::PARTS;             // columns of a part
        // slots 64..127 are read only when the plan is wide
        const bool live = wide || q < 2;
        float sum[PW];
#pragma unroll
        for (int i = 0; i < PW; ++i) sum[i] = 0.f;
        for (int64_t c = 0; c < n_chunks; ++c) {
            const int acc = (int)(c & 1);
            int f_ok = lane == 0 ? (mbar_wait(&dfull[acc], (uint32_t)((c >> 1) & 1), status) ? 1 : 0)
                                 : 0;
            f_ok = __shfl_sync(0xffffffffu, f_ok, 0);
            if (!f_ok) break;
            tc_fence_after();
            if (live) {
#pragma unroll
                for (int ch = 0; ch < PW / 32; ++ch) {
                    uint32_t r[32];
                    tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) +
                                  (uint32_t)(acc * BP + part * PW + ch * 32),
                              r);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) sum[ch * 32 + i] += __uint_as_float(r[i]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dfree[acc]);
        }
        if (live) {
            float *o = partial + ((int64_t)blockIdx.x * REACH_T + slot) * BP + part * PW;
#pragma unroll
            for (int i = 0; i < PW; i += 4)
                *reinterpret_cast<float4 *>(o + i) =
                    make_float4(sum[i], sum[i + 1], sum[i + 2], sum[i + 3]);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem_base, C::TMEM_COLS);
}

// coef_hi / coef_lo [REACH_T][n_pad] bf16: row i = candidate slot i's
// combined coefficient sum_t alpha^t C_t[k][i] (Horner over t) split into
// hi + lo, zero for k >= n.  One CTA per 64 rows k: the rows' slots are
// read contiguously (coalesced), transposed through shared memory and
// written along k (coalesced).  part[cta][i]: the rows' sums in 64 bits.
__global__ __launch_bounds__(256) void k_reach_pack(const ReachLevels C, int64_t n,
                                                    int64_t n_pad, int H, float alpha,
                                                    uint16_t *__restrict__ hi,
                                                    uint16_t *__restrict__ lo,
                                                    double *__restrict__ part) {
    __shared__ float tile[64][REACH_T + 1];
    const int64_t k0 = (int64_t)blockIdx.x * 64;
    for (int x = threadIdx.x; x < 64 * REACH_T; x += blockDim.x) {
        const int kk = x / REACH_T, i = x % REACH_T;
        const int64_t k = k0 + kk;
        float c = 0.f;
        if (k < n) {
            const int64_t at = k * REACH_T + i;
            for (int t = H; t >= 1; --t) c = alpha * (c + C.level[t - 1][at]);
        }
        tile[kk][i] = c;
    }
    __syncthreads();
    if (threadIdx.x < REACH_T) {
        double s = 0.0;
        for (int kk = 0; kk < 64; ++kk) s += (double)tile[kk][threadIdx.x];
        part[(int64_t)blockIdx.x * REACH_T + threadIdx.x] = s;
    }
    for (int x = threadIdx.x; x < 32 * REACH_T; x += blockDim.x) {
        const int i = x / 32, kk = 2 * (x % 32);
        const int64_t k = k0 + kk;
        uint32_t l;
        const uint32_t h = split_bf16_pair(tile[kk][i], tile[kk + 1][i], l);
        *reinterpret_cast<uint32_t *>(hi + (int64_t)i * n_pad + k) = h;
        *reinterpret_cast<uint32_t *>(lo + (int64_t)i * n_pad + k) = l;
    }
}


// Final score of each flagged candidate for each real query column: its u
// plus the CTAs' partials, appended as a filter key (score bits, ~chunk ID)
// to the column's buffer; the buffer then holds exactly them.  bp / Q
// blocks per candidate slot of the plan, each on Q query columns (blocks
// past nk, and every block when the plan says the hops run, return at
// once): thread t takes column t % Q of its block's and every G-th
// partial from t / Q on (coalesced rows of the partials), and the groups
// are added in group order (the same order on every run).
// F32: u is fp32 in `u` (32 query columns a block) and the partials are of
// u - Lmin; else u - m is split bf16 in u_hi, u_lo (64 columns), m = batch_u_min.
template <bool F32>
__global__ __launch_bounds__(1024) void k_reach_emit(const float *__restrict__ u,
                                                     const uint16_t *__restrict__ u_hi,
                                                     const uint16_t *__restrict__ u_lo, int bp, int B,
                                                     const float *__restrict__ partial,
                                                     int n_parts, const int32_t *__restrict__ plan,
                                                     const int32_t *__restrict__ rows,
                                                     const int32_t *__restrict__ ext_of,
                                                     unsigned int *__restrict__ cnt,
                                                     unsigned long long *__restrict__ buf,
                                                     int64_t cap, const double *__restrict__ sums,
                                                     const unsigned int *__restrict__ ext,
                                                     const float *__restrict__ shift) {
    constexpr int Q = F32 ? 32 : 64, G = 1024 / Q;
    __shared__ float red[1024];
    griddep_wait();
    if (plan[0] == 0) return;
    const int nk = plan[1];
    const int qb_n = bp / Q;
    const int i = blockIdx.x / qb_n;
    if (i >= nk) return;
    const int slot = plan[2 + i];
    const int b = (blockIdx.x % qb_n) * Q + threadIdx.x % Q;
    const int g = threadIdx.x / Q;
    float acc = 0.f;
    if (!F32 || b < B) {   // (the fp32 pass writes the real columns only)
#pragma unroll 4
        for (int p = g; p < n_parts; p += G) acc += partial[((int64_t)p * REACH_T + slot) * bp + b];
    }
    red[threadIdx.x] = acc;
    const float m = F32 ? ext_lmin(ext) : batch_u_min(shift, bp);
    __syncthreads();
    if (g == 0 && b < B) {
        float sum = red[threadIdx.x];
        for (int h = 1; h < G; ++h) sum += red[h * Q + threadIdx.x];
        const int64_t j = rows[slot];
        // the partials are of u - m; in the split form so is u itself
        const double uj = F32 ? (double)u[j * bp + b]
                              : (double)__bfloat162float(__ushort_as_bfloat16(u_hi[j * bp + b])) +
                                    (double)__bfloat162float(__ushort_as_bfloat16(u_lo[j * bp + b])) +
                                    (double)m;
        const float s = (float)(uj + ((double)m * sums[slot] + (double)sum));
        buf[(int64_t)b * cap + i] = ((unsigned long long)__float_as_uint(s) << 32) |
                                    (unsigned long long)(~(uint32_t)ext_of[j]);
        if (i == 0) cnt[b] = (unsigned int)nk;
    }
}

int reach_parts() { return device_sm_count(); }

int64_t reach_pad_rows(int64_t n) { return (n + RM_BK - 1) / RM_BK * RM_BK; }


// sum[i] = the column sums' parts part[p][i], p < n_parts, in a fixed order.
__global__ __launch_bounds__(256) void k_reach_colsum(const double *__restrict__ part,
                                                      int64_t n_parts, double *__restrict__ sum) {
    __shared__ double red[256];
    double s = 0.0;
    for (int64_t p = threadIdx.x; p < n_parts; p += 256) s += part[p * REACH_T + blockIdx.x];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) sum[blockIdx.x] = red[0];
}

static int combine_ctas() { return device_sm_count() * 8; }
int64_t reach_sum_words(int64_t n) {
    const int64_t tiles = reach_pad_rows(n) / 64;
    return (int64_t)REACH_T * (1 + (tiles > combine_ctas() ? tiles : combine_ctas()));
}

cudaError_t launch_reach_pack(const ReachLevels &C, int64_t n, int H, float alpha,
                              uint16_t *coef_hi, uint16_t *coef_lo, double *sums,
                              cudaStream_t st) {
    const int64_t n_pad = reach_pad_rows(n);
    if (n_pad <= 0) return cudaSuccess;
    k_reach_pack<<<(unsigned)(n_pad / 64), 256, 0, st>>>(C, n, n_pad, H, alpha, coef_hi, coef_lo,
                                                         sums + REACH_T);
    k_reach_colsum<<<REACH_T, 256, 0, st>>>(sums + REACH_T, n_pad / 64, sums);
    return cudaGetLastError();
}

template <int BP>
static cudaError_t reach_mma_bp(const uint16_t *coef_hi, const uint16_t *coef_lo,
                                const uint16_t *u_hi, const uint16_t *u_lo, int64_t n,
                                const int32_t *plan, float *partial, int parts, int *status,
                                cudaStream_t st) {
    using C = RmCfg<BP>;
    static bool attr[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_reach_mma<BP>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
        if (e != cudaSuccess) return e;
        attr[dev] = true;
    }
    const int64_t n_pad = reach_pad_rows(n);
    CUtensorMap thi, tlo, thi64, tlo64;
    cudaError_t e = make_tmap_2d(&thi, coef_hi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                                 (uint64_t)n_pad, RM_M, (uint64_t)n_pad * 2, RM_BK, RM_M);
    if (e == cudaSuccess)
        e = make_tmap_2d(&tlo, coef_lo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)n_pad, RM_M,
                         (uint64_t)n_pad * 2, RM_BK, RM_M);
    if (e == cudaSuccess)
        e = make_tmap_2d(&thi64, coef_hi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)n_pad,
                         RM_M, (uint64_t)n_pad * 2, RM_BK, RM_M / 2);
    if (e == cudaSuccess)
        e = make_tmap_2d(&tlo64, coef_lo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)n_pad,
                         RM_M, (uint64_t)n_pad * 2, RM_BK, RM_M / 2);
    CUtensorMap tbh, tbl;
    if (e == cudaSuccess)
        e = make_tmap_2d(&tbh, u_hi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, BP, (uint64_t)n,
                         (uint64_t)BP * 2, 64, RM_BK);
    if (e == cudaSuccess)
        e = make_tmap_2d(&tbl, u_lo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, BP, (uint64_t)n,
                         (uint64_t)BP * 2, 64, RM_BK);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_reach_mma<BP>, dim3(parts), dim3(RM_THREADS), C::SMEM, st, thi, tlo, thi64,
                      tlo64, tbh, tbl, n, plan, partial, status);
}

cudaError_t launch_reach_scores(const uint16_t *u_hi, const uint16_t *u_lo, const float *shift,
                                int bp, int B, int64_t n, const uint16_t *coef_hi,
                                const uint16_t *coef_lo, const double *sums, const int32_t *plan,
                                const int32_t *rows, const int32_t *ext_of, float *partial,
                                unsigned int *cnt, unsigned long long *buf, int64_t cap,
                                int *status, cudaStream_t st, int *launches) {
    const int parts = reach_parts();
    cudaError_t e = cudaErrorInvalidValue;
    if (n <= 0) return e;
    switch (bp) {
    case 64: e = reach_mma_bp<64>(coef_hi, coef_lo, u_hi, u_lo, n, plan, partial, parts, status, st); break;
    case 128: e = reach_mma_bp<128>(coef_hi, coef_lo, u_hi, u_lo, n, plan, partial, parts, status, st); break;
    case 256: e = reach_mma_bp<256>(coef_hi, coef_lo, u_hi, u_lo, n, plan, partial, parts, status, st); break;
    }
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_reach_emit<false>, dim3(REACH_T * (bp / 64)), dim3(1024), 0, st,
                   (const float *)nullptr, u_hi, u_lo, bp, B, (const float *)partial, parts, plan,
                   rows, ext_of, cnt, buf, cap, sums, (const unsigned int *)nullptr, shift);
    if (launches) *launches += 2;
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// ------------------------------------------------------------------ fp32 terms
// The same partial sums in fp32 on the CUDA cores, for at most 32 queries (the
// tensor cores' tiles have 64 columns, and a slab of 64 would cost more than
// the FMAs):
//   sum_k coef[k][i] u[k][b] = m S_i + sum_k coef[k][i] (u[k][b] - m)
// with m = Lmin, the smallest u of any live row and real query: u - m is exact
// where u <= 2 m, every term stays >= 0, and the terms are as much smaller as u
// is flat, and the sums' rounding with them.  (Plain sums of nearly equal
// terms all round the same way: three hops on 262,144 chunks were 1.4e-6 off,
// 3e-8 so, 2.8e-7 the hops.)
// Bound by the loads for few queries (64 coefficients and the query columns a
// row: 268 MB at 1,048,576 chunks) and by the FMAs and shared loads towards 32:
// n * 64 * columns of them, 96 or 128 where flagged slots lie there.  The hops
// gather nnz columns a hop instead, an order of magnitude more, from L2.
// A warp works alone: it takes groups of RF_ROWS rows, copies their
// coefficients and query columns into its own ring of RF_STAGES stages
// (cp.async), and keeps an ST-slot x CT-column tile of sums in registers, a
// lane's part SPL slots x CPL columns: SPL * CPL FMAs a row for (SPL + CPL) / 4
// 16-byte shared loads.  The eight warps' tiles, then the CTAs' partials, are
// added in a fixed order.
constexpr int RF_ROWS = 8, RF_STAGES = 4, RF_WARPS = 8;

template <int ST, int CT>
struct RfCfg {
    static constexpr int SPL = ST * CT == 512 ? 4 : 8;
    static constexpr int SG = ST / SPL, CG = 32 / SG;           // lanes over slots, columns
    static constexpr int CPL = CT / CG;
    static constexpr int STAGE = RF_ROWS * (ST + CT);           // floats a stage
    static constexpr int SMEM = RF_WARPS * RF_STAGES * STAGE * 4;
    static_assert(SPL % 4 == 0 && CPL % 4 == 0 && SG * CG == 32, "16-byte shared loads");
    static_assert(RF_WARPS * ST * CT * 4 <= SMEM, "the tiles' sum reuses the rings");
};

__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(valid ? 16 : 0)
                 : "memory");
}

template <int ST, int CT>
__global__ __launch_bounds__(RF_WARPS * 32, 2) void k_reach_fma(
    const float *__restrict__ u, int bp, int64_t n, const float *__restrict__ coef, int slot0,
    const int32_t *__restrict__ plan, const unsigned int *__restrict__ ext,
    float *__restrict__ partial) {
    using C = RfCfg<ST, CT>;
    extern __shared__ float4 rf_smem[];
    float *smem = reinterpret_cast<float *>(rf_smem);
    griddep_wait();
    if (plan[0] == 0) return;
    const int s0 = slot0 + (int)blockIdx.y * ST;       // slots s0 .. s0 + ST - 1
    if (plan[1 + plan[1]] < s0) return;                // the last flagged slot is below
    const float m = ext_lmin(ext);
    const int c0 = blockIdx.z * CT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sg = lane % C::SG, cg = lane / C::SG;
    float *ring = smem + warp * RF_STAGES * C::STAGE;
    const int64_t groups = (n + RF_ROWS - 1) / RF_ROWS;
    const int64_t per = (groups + gridDim.x - 1) / gridDim.x;
    const int64_t g0 = (int64_t)blockIdx.x * per + warp;
    const int64_t g1 = min((int64_t)(blockIdx.x + 1) * per, groups);
    auto load = [&](int64_t g, int stage) {
        float *cs = ring + stage * C::STAGE, *us = cs + RF_ROWS * ST;
#pragma unroll
        for (int i = 0; i < RF_ROWS * ST / 128; ++i) {
            const int c = lane + 32 * i, r = c / (ST / 4);
            const int64_t row = g * RF_ROWS + r;
            const bool ok = row < n;
            cp_async16(cs + c * 4, coef + (ok ? row : 0) * REACH_T + s0 + (c % (ST / 4)) * 4, ok);
        }
#pragma unroll
        for (int i = 0; i < (RF_ROWS * CT / 4 + 31) / 32; ++i) {
            const int c = lane + 32 * i, r = c / (CT / 4);
            const int64_t row = g * RF_ROWS + r;
            const bool ok = row < n;
            if (RF_ROWS * CT / 4 >= 32 || c < RF_ROWS * CT / 4)
                cp_async16(us + c * 4, u + (ok ? row : 0) * bp + c0 + (c % (CT / 4)) * 4, ok);
        }
    };
    float acc[C::SPL][C::CPL];
#pragma unroll
    for (int i = 0; i < C::SPL; ++i)
#pragma unroll
        for (int j = 0; j < C::CPL; ++j) acc[i][j] = 0.f;
    int64_t gl = g0;                                   // next group to load
#pragma unroll
    for (int s = 0; s < RF_STAGES - 1; ++s, gl += RF_WARPS) {
        if (gl < g1) load(gl, s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int stage = 0, next = RF_STAGES - 1;
    for (int64_t g = g0; g < g1; g += RF_WARPS, gl += RF_WARPS) {
        if (gl < g1) load(gl, next);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group %0;" ::"n"(RF_STAGES - 1) : "memory");
        __syncwarp();
        const float *cs = ring + stage * C::STAGE, *us = cs + RF_ROWS * ST;
#pragma unroll
        for (int r = 0; r < RF_ROWS; ++r) {
            float a[C::SPL], x[C::CPL];
#pragma unroll
            for (int i = 0; i < C::SPL / 4; ++i)
                *reinterpret_cast<float4 *>(a + 4 * i) =
                    *reinterpret_cast<const float4 *>(cs + r * ST + (i * C::SG + sg) * 4);
#pragma unroll
            for (int j = 0; j < C::CPL / 4; ++j)
                *reinterpret_cast<float4 *>(x + 4 * j) =
                    *reinterpret_cast<const float4 *>(us + r * CT + (j * C::CG + cg) * 4);
#pragma unroll
            for (int j = 0; j < C::CPL; ++j) x[j] -= m;   // (rows past n have coefficient 0)
#pragma unroll
            for (int i = 0; i < C::SPL; ++i)
#pragma unroll
                for (int j = 0; j < C::CPL; ++j) acc[i][j] = fmaf(a[i], x[j], acc[i][j]);
        }
        __syncwarp();   // the stage is free for the next round's copies
        if (++stage == RF_STAGES) stage = 0;
        if (++next == RF_STAGES) next = 0;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // the warps' tiles through shared memory, added in warp order
    float *mine = smem + warp * ST * CT;
#pragma unroll
    for (int i = 0; i < C::SPL; ++i)
#pragma unroll
        for (int j = 0; j < C::CPL; j += 4)
            *reinterpret_cast<float4 *>(mine + ((i / 4 * C::SG + sg) * 4 + i % 4) * CT +
                                        (j / 4 * C::CG + cg) * 4) =
                make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
    __syncthreads();
    for (int x = threadIdx.x; x < ST * CT; x += RF_WARPS * 32) {
        float s = smem[x];
#pragma unroll
        for (int w = 1; w < RF_WARPS; ++w) s += smem[w * ST * CT + x];
        partial[((int64_t)blockIdx.x * REACH_T + s0 + x / CT) * bp + c0 + x % CT] = s;
    }
}

// coef[k][i] = sum_t alpha^t C_t[k][i] (Horner over t), fp32, and its column
// sums in 64 bits: each CTA's in part[cta][i], added by k_reach_colsum.  128
// threads a row.
__global__ __launch_bounds__(256) void k_reach_combine(const ReachLevels C, int64_t n, int H,
                                                       float alpha, float *__restrict__ coef,
                                                       double *__restrict__ part) {
    __shared__ double half[REACH_T];
    const int i = threadIdx.x % REACH_T, h = threadIdx.x / REACH_T;
    double s = 0.0;
    for (int64_t k = (int64_t)blockIdx.x * 2 + h; k < n; k += (int64_t)gridDim.x * 2) {
        float c = 0.f;
        for (int t = H; t >= 1; --t) c = alpha * (c + C.level[t - 1][k * REACH_T + i]);
        coef[k * REACH_T + i] = c;
        s += (double)c;
    }
    if (h == 1) half[i] = s;
    __syncthreads();
    if (h == 0) part[(int64_t)blockIdx.x * REACH_T + i] = s + half[i];
}
cudaError_t launch_reach_combine(const ReachLevels &C, int64_t n, int H, float alpha, float *coef,
                                 double *sums, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_reach_combine<<<combine_ctas(), 256, 0, st>>>(C, n, H, alpha, coef, sums + REACH_T);
    k_reach_colsum<<<REACH_T, 256, 0, st>>>(sums + REACH_T, combine_ctas(), sums);
    return cudaGetLastError();
}

// CTAs along the rows: two an SM, at least a group of rows a warp.
int reach_fma_parts(int64_t n) {
    const int64_t most = ceil_div<int64_t>(n, RF_ROWS * RF_WARPS), want = 2 * device_sm_count();
    return (int)(want < most ? want : most);
}

template <int ST, int CT>
static cudaError_t reach_fma_tile(const float *u, int bp, int B, int64_t n, const float *coef,
                                  int slot0, const int32_t *plan, const unsigned int *ext,
                                  float *partial, int parts, cudaStream_t st) {
    static bool attr[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_reach_fma<ST, CT>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             RfCfg<ST, CT>::SMEM);
        if (e != cudaSuccess) return e;
        attr[dev] = true;
    }
    const int slots = slot0 == 0 ? 64 : REACH_T - slot0;
    return launch_pdl(k_reach_fma<ST, CT>, dim3(parts, slots / ST, (B + CT - 1) / CT),
                      dim3(RF_WARPS * 32), RfCfg<ST, CT>::SMEM, st, u, bp, n, coef, slot0, plan,
                      ext, partial);
}

// Slots 0..63, then the two groups of 32 above (CTAs of a group without a
// flagged slot return at once).
cudaError_t launch_reach_fma(const float *u, int bp, int B, int64_t n, const float *coef,
                             const double *sums, const unsigned int *ext, const int32_t *plan,
                             const int32_t *rows, const int32_t *ext_of, float *partial,
                             unsigned int *cnt, unsigned long long *buf, int64_t cap,
                             cudaStream_t st, int *launches) {
    if (n <= 0 || B < 1 || B > 32 || bp != 32) return cudaErrorInvalidValue;
    const int parts = reach_fma_parts(n);
    cudaError_t e;
#define RF_TILE(ST, CT, S0) reach_fma_tile<ST, CT>(u, bp, B, n, coef, S0, plan, ext, partial, parts, st)
    if (B <= 8) e = RF_TILE(64, 8, 0);
    else if (B <= 16) e = RF_TILE(64, 16, 0);
    else e = RF_TILE(64, 32, 0);
    if (e == cudaSuccess) e = B <= 16 ? RF_TILE(32, 16, 64) : RF_TILE(32, 32, 64);
#undef RF_TILE
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_reach_emit<true>, dim3(REACH_T * (bp / 32)), dim3(1024), 0, st, u,
                   (const uint16_t *)nullptr, (const uint16_t *)nullptr, bp, B,
                   (const float *)partial, parts, plan, rows, ext_of, cnt, buf, cap, sums, ext,
                   (const float *)nullptr);
    if (launches) *launches += 3;
    return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace ak
