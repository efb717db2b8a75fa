// Relation graph on the device: prefix sums, a stable LSD radix sort, the
// in-edge transpose in store-row space, relation weights, the page-order
// layout of appended chunks, and the propagation hop (a2) that
// spreads scores along cross-chunk relations (arXiv 2607.05708, §4.1:
// related chunks are recovered together).
#include "ak_common.cuh"

namespace ak {

static int sm_count_cached() {
    static int cached[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (!cached[dev]) {
        int v = 0;
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        cached[dev] = v > 0 ? v : 1;
    }
    return cached[dev];
}
int device_sm_count() { return sm_count_cached(); }

// ================================================================== ordered tiles
// groups[g] = the sum of the counts of tiles 1024 g .. (see tile_base).
__global__ __launch_bounds__(256) void k_tile_groups(int32_t *__restrict__ counts, int64_t tiles) {
    griddep_wait();
    __shared__ int part[8];
    const int64_t t0 = (int64_t)blockIdx.x * TILE_GROUP;
    int s = 0;
#pragma unroll
    for (int q = 0; q < TILE_GROUP / 256; ++q) {
        const int64_t t = t0 + q * 256 + threadIdx.x;
        s += t < tiles ? counts[t] : 0;
    }
    s = (int)__reduce_add_sync(0xffffffffu, (unsigned)s);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s += part[w];
        counts[tiles + blockIdx.x] = s;
    }
}

cudaError_t launch_tile_groups(int32_t *counts, int64_t tiles, cudaStream_t st, int *launches) {
    if (tiles <= TILE_FLAT) return cudaSuccess;
    if (launches) *launches += 1;
    return launch_pdl(k_tile_groups, dim3((unsigned)ceil_div<int64_t>(tiles, TILE_GROUP)),
                      dim3(256), 0, st, counts, tiles);
}

// ================================================================== scan
constexpr int SCAN_THREADS = 256, SCAN_ITEMS = 8;
static_assert(SCAN_TILE == SCAN_THREADS * SCAN_ITEMS, "a tile is one CTA's share");

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Each CTA scans one tile of SCAN_TILE values (exclusive) and emits the
// tile total.
__global__ __launch_bounds__(SCAN_THREADS) void k_scan_tile(const int64_t *__restrict__ in,
                                                            int64_t *__restrict__ out, int64_t n,
                                                            int64_t *__restrict__ tile_sum) {
    __shared__ int64_t wsum[SCAN_THREADS / 32];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int64_t v[SCAN_ITEMS];
    int64_t run = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int64_t idx = base + i;
        v[i] = idx < n ? in[idx] : 0;
        run += v[i];
    }
    int64_t incl = warp_incl_scan(run);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t s = lane < SCAN_THREADS / 32 ? wsum[lane] : 0;
        s = warp_incl_scan(s);
        if (lane < SCAN_THREADS / 32) wsum[lane] = s;
    }
    __syncthreads();
    int64_t excl = incl - run + (warp > 0 ? wsum[warp - 1] : 0);
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int64_t idx = base + i;
        if (idx < n) out[idx] = excl;
        excl += v[i];
    }
    if (threadIdx.x == SCAN_THREADS - 1) tile_sum[blockIdx.x] = excl;
}

__global__ void k_scan_add(int64_t *__restrict__ out, int64_t n,
                           const int64_t *__restrict__ tile_off) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < n) out[idx] += tile_off[idx / SCAN_TILE];
}

__global__ void k_scan_total(const int64_t *__restrict__ in, int64_t *__restrict__ out,
                             int64_t n) {
    // out[n] = out[n-1] + in[n-1]  (n >= 1), else 0
    out[n] = n > 0 ? out[n - 1] + in[n - 1] : 0;
}

// Flat form, for at most SCAN_FLAT_TILES tiles: the tile sums, then each CTA
// adds up the sums of the tiles before it and scans its own tile; the last
// CTA writes the total.  Two launches (one for a single tile).
constexpr int64_t SCAN_FLAT_TILES = 1024;

__device__ __forceinline__ int64_t block_sum_scan(int64_t v, int64_t *wsum) {
    // the CTA's sum of v, on every thread (wsum: SCAN_THREADS / 32 slots)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) wsum[warp] = v;
    __syncthreads();
    int64_t s = 0;
#pragma unroll
    for (int w = 0; w < SCAN_THREADS / 32; ++w) s += wsum[w];
    return s;
}

__global__ __launch_bounds__(SCAN_THREADS) void k_scan_reduce(const int64_t *__restrict__ in,
                                                              int64_t n,
                                                              int64_t *__restrict__ tile_sum) {
    griddep_wait();
    __shared__ int64_t wsum[SCAN_THREADS / 32];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t idx = base + i * SCAN_THREADS + threadIdx.x;
        if (idx < n) s += in[idx];
    }
    s = block_sum_scan(s, wsum);
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = s;
}

__global__ __launch_bounds__(SCAN_THREADS) void k_scan_down(const int64_t *__restrict__ in,
                                                            int64_t *__restrict__ out, int64_t n,
                                                            const int64_t *__restrict__ tile_sum) {
    griddep_wait();
    __shared__ int64_t wsum[SCAN_THREADS / 32];
    int64_t pre = 0;
    for (int64_t t = threadIdx.x; t < (int64_t)blockIdx.x; t += SCAN_THREADS) pre += tile_sum[t];
    pre = block_sum_scan(pre, wsum);
    __syncthreads();   // wsum is reused below
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    int64_t v[SCAN_ITEMS];
    int64_t run = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t idx = base + i;
        v[i] = idx < n ? in[idx] : 0;
        run += v[i];
    }
    const int64_t incl = warp_incl_scan(run);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int64_t excl = pre + incl - run;
    for (int w = 0; w < warp; ++w) excl += wsum[w];
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t idx = base + i;
        if (idx < n) out[idx] = excl;
        excl += v[i];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == SCAN_THREADS - 1) out[n] = excl;
}

static cudaError_t scan_rec(const int64_t *in, int64_t *out, int64_t n, int64_t *tmp,
                            cudaStream_t st, int *launches) {
    if (n <= 0) return cudaSuccess;
    int64_t tiles = ceil_div<int64_t>(n, SCAN_TILE);
    int64_t *sums = tmp, *offs = tmp + tiles;
    k_scan_tile<<<(unsigned)tiles, SCAN_THREADS, 0, st>>>(in, out, n, sums);
    if (launches) *launches += 1;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || tiles == 1) return e;
    e = scan_rec(sums, offs, tiles, tmp + 2 * tiles + 2, st, launches);
    if (e != cudaSuccess) return e;
    k_scan_add<<<(unsigned)ceil_div<int64_t>(n, 256), 256, 0, st>>>(out, n, offs);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

cudaError_t scan_exclusive(const int64_t *in, int64_t *out, int64_t n, void *tmp,
                           size_t tmp_bytes, cudaStream_t st, int *launches) {
    if (tmp_bytes < scan_tmp_bytes(n)) return cudaErrorInvalidValue;
    const int64_t tiles = ceil_div<int64_t>(n, SCAN_TILE);
    if (n > 0 && tiles <= SCAN_FLAT_TILES) {
        int64_t *sums = (int64_t *)tmp;
        if (tiles > 1) launch_pdl(k_scan_reduce, dim3((unsigned)tiles), dim3(SCAN_THREADS), 0, st,
                                  in, n, sums);
        launch_pdl(k_scan_down, dim3((unsigned)tiles), dim3(SCAN_THREADS), 0, st, in, out, n, sums);
        if (launches) *launches += tiles > 1 ? 2 : 1;
        return cudaGetLastError();
    }
    cudaError_t e = scan_rec(in, out, n, (int64_t *)tmp, st, launches);
    if (e != cudaSuccess) return e;
    k_scan_total<<<1, 1, 0, st>>>(in, out, n);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

// ================================================================== radix sort
// Stable LSD radix sort of (uint32 key, uint32 value) pairs, 8 bits a pass.
// Per pass: tile histograms (digit-major), one exclusive scan, then a stable
// scatter in which each warp ranks its keys round by round with
// __match_any_sync and the warps of a tile are combined in order.
constexpr int RS_THREADS = 256, RS_ITEMS = 16;
static_assert(RS_TILE == RS_THREADS * RS_ITEMS, "a tile is one CTA's share");
constexpr int RS_WARPS = RS_THREADS / 32, RS_PER_WARP = RS_TILE / RS_WARPS;

__global__ __launch_bounds__(RS_THREADS) void k_rs_hist(const uint32_t *__restrict__ keys,
                                                        int64_t n, int shift, uint32_t mask,
                                                        int64_t n_tiles,
                                                        int64_t *__restrict__ hist) {
    __shared__ int h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    for (int i = threadIdx.x; i < RS_TILE; i += RS_THREADS) {
        int64_t idx = base + i;
        if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & mask], 1);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * n_tiles + blockIdx.x] = h[threadIdx.x];
}

// Rank the warp's 32 * ITEMS keys of the tile stably by digit: loc[r] is
// the key's rank among the warp's keys of its digit, cnt[warp][d] the
// warp's count of digit d; then pre[w][d] = the counts of digit d in the
// warps before w (one thread a digit).  Keys at or past n get no digit.
template <int ITEMS>
__device__ __forceinline__ void rs_rank(const uint32_t *__restrict__ keys,
                                        const uint32_t *__restrict__ vals, int64_t n,
                                        int64_t base, int shift, uint32_t mask,
                                        uint32_t (&k)[ITEMS], uint32_t (&v)[ITEMS],
                                        int (&loc)[ITEMS], int (*cnt)[256], int (*pre)[256]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = lane; d < 256; d += 32) cnt[warp][d] = 0;
    __syncwarp();
    const unsigned lt = (1u << lane) - 1u;
    // every load first, then the ranking (whose rounds depend on each other)
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t idx = base + r * 32 + lane;
        k[r] = idx < n ? keys[idx] : 0u;
        v[r] = idx < n ? vals[idx] : 0u;
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        int64_t idx = base + r * 32 + lane;
        bool ok = idx < n;
        uint32_t d = ok ? ((k[r] >> shift) & mask) : 0x100u;   // 0x100: no digit
        unsigned peers = __match_any_sync(0xffffffffu, d);
        int leader = __ffs(peers) - 1;
        int c = ok ? cnt[warp][d] : 0;
        loc[r] = c + __popc(peers & lt);
        __syncwarp();
        if (ok && lane == leader) cnt[warp][d] = c + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {
        int d = threadIdx.x;   // RS_THREADS == 256 digits
        int run = 0;
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) {
            pre[w][d] = run;
            run += cnt[w][d];
        }
    }
    __syncthreads();
}

__global__ __launch_bounds__(RS_THREADS) void k_rs_scatter(
    const uint32_t *__restrict__ keys, const uint32_t *__restrict__ vals, int64_t n, int shift,
    uint32_t mask, int64_t n_tiles, const int64_t *__restrict__ offs, uint32_t *__restrict__ okeys,
    uint32_t *__restrict__ ovals) {
    __shared__ int cnt[RS_WARPS][256];
    __shared__ int pre[RS_WARPS][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * RS_TILE + (int64_t)warp * RS_PER_WARP;
    uint32_t k[RS_ITEMS], v[RS_ITEMS];
    int loc[RS_ITEMS];
    rs_rank<RS_ITEMS>(keys, vals, n, base, shift, mask, k, v, loc, cnt, pre);
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        int64_t idx = base + r * 32 + lane;
        if (idx < n) {
            uint32_t d = (k[r] >> shift) & mask;
            int64_t pos = offs[(int64_t)d * n_tiles + blockIdx.x] + pre[warp][d] + loc[r];
            okeys[pos] = k[r];
            ovals[pos] = v[r];
        }
    }
}

// Small sorts (at most RS_SMALL_TILES tiles of RS_SMALL_TILE keys: four a
// thread, so that a sort of ~100k pairs still spreads over ~100 CTAs) take
// one launch a pass after a first histogram launch.  Histograms are int32,
// digit-major [256][n_tiles].
// Each scatter CTA derives its own offsets from the pass's histograms (the
// totals of the smaller digits plus its digit's counts in the tiles before
// it) and counts the next pass's digit of every key it places into the next
// histograms, by destination tile.  Three histogram buffers rotate: pass p
// reads H[p % 3], counts into H[(p+1) % 3] (zero by then) and zeroes its
// column of H[(p+2) % 3], which pass p-1 read and pass p+1 counts into.
constexpr int RS_SMALL_ITEMS = 4;
static_assert(RS_SMALL_TILE == RS_THREADS * RS_SMALL_ITEMS, "a tile is one CTA's share");

__global__ __launch_bounds__(RS_THREADS) void k_rs_hist32(const uint32_t *__restrict__ keys,
                                                          int64_t n, int shift, uint32_t mask,
                                                          int n_tiles, int *__restrict__ hist,
                                                          int *__restrict__ zero1,
                                                          int *__restrict__ zero2) {
    griddep_wait();
    __shared__ int h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_SMALL_TILE;
    for (int i = threadIdx.x; i < RS_SMALL_TILE; i += RS_THREADS) {
        int64_t idx = base + i;
        if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & mask], 1);
    }
    __syncthreads();
    const int64_t at = (int64_t)threadIdx.x * n_tiles + blockIdx.x;
    hist[at] = h[threadIdx.x];
    zero1[at] = 0;
    zero2[at] = 0;
}

__global__ __launch_bounds__(RS_THREADS) void k_rs_scatter_small(
    const uint32_t *__restrict__ keys, const uint32_t *__restrict__ vals, int64_t n, int shift,
    uint32_t mask, int n_tiles, const int *__restrict__ hcur, int *__restrict__ hnext,
    int shift_next, uint32_t mask_next, int *__restrict__ hzero, uint32_t *__restrict__ okeys,
    uint32_t *__restrict__ ovals) {
    griddep_wait();
    __shared__ int cnt[RS_WARPS][256];
    __shared__ int pre[RS_WARPS][256];
    __shared__ int off_s[256];
    __shared__ int wtot[RS_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    {
        // thread d: digit d's total and its count in the tiles before this one
        const int d = threadIdx.x;
        const int *row = hcur + (int64_t)d * n_tiles;
        int tot = 0, before = 0;
#pragma unroll 16
        for (int t = 0; t < n_tiles; ++t) {
            const int c = row[t];
            tot += c;
            before += t < (int)blockIdx.x ? c : 0;
        }
        int incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) wtot[warp] = incl;
        __syncthreads();
        int wpre = 0;
        for (int w = 0; w < warp; ++w) wpre += wtot[w];
        off_s[d] = wpre + incl - tot + before;
        if (hzero) hzero[(int64_t)d * n_tiles + blockIdx.x] = 0;
    }
    const int64_t base =
        (int64_t)blockIdx.x * RS_SMALL_TILE + (int64_t)warp * (32 * RS_SMALL_ITEMS);
    uint32_t k[RS_SMALL_ITEMS], v[RS_SMALL_ITEMS];
    int loc[RS_SMALL_ITEMS];
    rs_rank<RS_SMALL_ITEMS>(keys, vals, n, base, shift, mask, k, v, loc, cnt, pre);   // syncs the CTA
#pragma unroll
    for (int r = 0; r < RS_SMALL_ITEMS; ++r) {
        const int64_t idx = base + r * 32 + lane;
        const bool ok = idx < n;
        const uint32_t d = (k[r] >> shift) & mask;
        const int pos = ok ? off_s[d] + pre[warp][d] + loc[r] : 0;
        if (ok) {
            okeys[pos] = k[r];
            ovals[pos] = v[r];
        }
        if (hnext) {
            // one atomic per distinct (next digit, destination tile) of the
            // warp's round: a high digit has few values, whose counters
            // would otherwise take the whole round's atomics each
            const uint32_t slot =
                ok ? ((k[r] >> shift_next) & mask_next) * (uint32_t)n_tiles +
                         (uint32_t)(pos / RS_SMALL_TILE)
                   : 0xffffffffu;
            const unsigned peers = __match_any_sync(0xffffffffu, slot);
            if (ok && lane == __ffs(peers) - 1) atomicAdd(&hnext[slot], (int)__popc(peers));
        }
    }
}

// At most RS_ONE pairs: every thread counts the keys before its own (smaller
// ones, and equal ones at an earlier place) and writes its pair there, in one
// launch spread over n / 128 CTAs.  A radix sort's launches cost ~4 us each
// whatever their size: 1280 pairs of 18 bits 19 -> 11 us (19 with a bitonic
// network in one CTA).
constexpr int64_t RS_ONE = 2048;
__global__ __launch_bounds__(128) void k_sort_one(const uint32_t *__restrict__ keys,
                                                  const uint32_t *__restrict__ vals, int n,
                                                  uint32_t mask, uint32_t *__restrict__ okeys,
                                                  uint32_t *__restrict__ ovals) {
    griddep_wait();
    __shared__ uint4 x4[RS_ONE / 4];
    uint32_t *x = reinterpret_cast<uint32_t *>(x4);
    for (int i = threadIdx.x; i < ((n + 3) & ~3); i += 128) x[i] = i < n ? keys[i] & mask : ~0u;
    __syncthreads();
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= n) return;
    const uint32_t mine = x[i];
    int rank = 0;
    for (int j = 0; j < n; j += 4) {
        const uint4 k = x4[j >> 2];
        rank += k.x < mine || (k.x == mine && j < i) ? 1 : 0;
        rank += k.y < mine || (k.y == mine && j + 1 < i) ? 1 : 0;
        rank += k.z < mine || (k.z == mine && j + 2 < i) ? 1 : 0;
        rank += k.w < mine || (k.w == mine && j + 3 < i) ? 1 : 0;
    }
    okeys[rank] = keys[i];
    ovals[rank] = vals[i];
}

cudaError_t radix_sort_pairs(uint32_t *keys, uint32_t *vals, uint32_t *keys_alt,
                             uint32_t *vals_alt, int64_t n, int bits, void *tmp,
                             size_t tmp_bytes, cudaStream_t st, bool *result_in_alt,
                             int *launches) {
    *result_in_alt = false;
    if (n <= 1 || bits <= 0) return cudaSuccess;
    if (tmp_bytes < radix_tmp_bytes(n)) return cudaErrorInvalidValue;
    if (n <= RS_ONE) {
        launch_pdl(k_sort_one, dim3((unsigned)ceil_div<int64_t>(n, 128)), dim3(128), 0, st, keys,
                   vals, (int)n, bits >= 32 ? 0xffffffffu : (1u << bits) - 1u, keys_alt, vals_alt);
        if (launches) *launches += 1;
        *result_in_alt = true;
        return cudaGetLastError();
    }
    const int64_t n_tiles = ceil_div<int64_t>(n, RS_TILE);
    const int64_t m = 256 * n_tiles;
    int64_t *hist = (int64_t *)tmp;
    int64_t *offs = hist + m;
    void *stmp = (void *)(offs + m + 1);
    size_t stmp_bytes = tmp_bytes - (size_t)(2 * m + 1) * sizeof(int64_t);
    uint32_t *ki = keys, *vi = vals, *ko = keys_alt, *vo = vals_alt;
    const int64_t s_tiles = ceil_div<int64_t>(n, RS_SMALL_TILE);
    if (s_tiles <= RS_SMALL_TILES) {
        const int64_t ms = 256 * s_tiles;
        int *h[3] = {(int *)tmp, (int *)tmp + ms, (int *)tmp + 2 * ms};
        const int nt = (int)s_tiles;
        launch_pdl(k_rs_hist32, dim3(nt), dim3(RS_THREADS), 0, st, ki, n, 0,
                   bits < 8 ? (1u << bits) - 1u : 0xffu, nt, h[0], h[1], h[2]);
        if (launches) *launches += 1;
        for (int p = 0, sh = 0; sh < bits; ++p, sh += 8) {
            const int nb = bits - sh < 8 ? bits - sh : 8;
            const int shn = sh + 8;
            const int nbn = bits - shn < 8 ? bits - shn : 8;
            launch_pdl(k_rs_scatter_small, dim3(nt), dim3(RS_THREADS), 0, st, ki, vi, n, sh,
                       (1u << nb) - 1u, nt, h[p % 3], shn < bits ? h[(p + 1) % 3] : nullptr, shn,
                       shn < bits ? (1u << nbn) - 1u : 0u, p >= 1 ? h[(p + 2) % 3] : nullptr, ko,
                       vo);
            if (launches) *launches += 1;
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            uint32_t *t;
            t = ki; ki = ko; ko = t;
            t = vi; vi = vo; vo = t;
            *result_in_alt = !*result_in_alt;
        }
        return cudaSuccess;
    }
    for (int sh = 0; sh < bits; sh += 8) {
        int nb = bits - sh < 8 ? bits - sh : 8;
        uint32_t mask = (1u << nb) - 1u;
        k_rs_hist<<<(unsigned)n_tiles, RS_THREADS, 0, st>>>(ki, n, sh, mask, n_tiles, hist);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        e = scan_exclusive(hist, offs, m, stmp, stmp_bytes, st, launches);
        if (e != cudaSuccess) return e;
        k_rs_scatter<<<(unsigned)n_tiles, RS_THREADS, 0, st>>>(ki, vi, n, sh, mask, n_tiles, offs,
                                                                ko, vo);
        if (launches) *launches += 2;
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        uint32_t *t;
        t = ki; ki = ko; ko = t;
        t = vi; vi = vo; vo = t;
        *result_in_alt = !*result_in_alt;
    }
    return cudaSuccess;
}

// ================================================================== CSR helpers
// One warp per row: src[e] = global row id for every edge of the row, and the
// row is checked: targets in [0, n_total), never the row itself, strictly
// ascending.  row_ptr is relative (offsets into col), rows are local; the
// global id of local row r is row_base + r; edge e is written at out_off + e.
__global__ void k_edge_src_check(const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                 int64_t n_rows, int64_t row_base, int64_t n_total,
                                 int32_t *__restrict__ src, int *status) {
    const int lane = threadIdx.x & 31;
    int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t p0 = row_ptr[0];
    for (; r < n_rows; r += stride) {
        int64_t a = row_ptr[r], b = row_ptr[r + 1];
        if (b < a) {
            if (lane == 0) set_status(status, AKASHIC_EDEVICE);
            continue;
        }
        const int64_t gid = row_base + r;
        for (int64_t e = a + lane; e < b; e += 32) {
            int32_t c = col[e];
            bool bad = c < 0 || (int64_t)c >= n_total || (int64_t)c == gid ||
                       (e > a && col[e - 1] >= c);
            if (bad) set_status(status, AKASHIC_EDEVICE);
            if (src) src[e - p0] = (int32_t)gid;
        }
    }
}

cudaError_t launch_edge_src_check(const int64_t *row_ptr, const int32_t *col, int64_t n_rows,
                                  int64_t row_base, int64_t n_total, int32_t *src, int *status,
                                  cudaStream_t st) {
    if (n_rows <= 0) return cudaSuccess;
    int64_t warps = n_rows < (int64_t)device_sm_count() * 64 ? n_rows : (int64_t)device_sm_count() * 64;
    k_edge_src_check<<<(unsigned)ceil_div<int64_t>(warps * 32, 256), 256, 0, st>>>(
        row_ptr, col, n_rows, row_base, n_total, src, status);
    return cudaGetLastError();
}

// Relation weights: w = softmax of each row's edge logits.  Eight lanes per
// row and four rows per warp step (rows are short: 32 edges plus the
// reciprocal ones), so a warp keeps four rows' loads in flight; a row of up
// to 64 edges is read once and kept in registers.
constexpr int RSM_LANES = 8, RSM_KEEP = 8;
__global__ void k_row_softmax(const int64_t *__restrict__ row_ptr, const float *__restrict__ aff,
                              float *__restrict__ w, int64_t n_rows, float2 *__restrict__ rstat) {
    constexpr int L = RSM_LANES, R = 32 / RSM_LANES;
    const int lane = threadIdx.x & 31, sub = lane % L, grp = lane / L;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // the next step's row bounds are loaded while this step's rows are
    // processed (they head each step's chain of dependent loads)
    int64_t r0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * R;
    int64_t na = 0, nb = 0;
    if (r0 + grp < n_rows) {
        na = row_ptr[r0 + grp];
        nb = row_ptr[r0 + grp + 1];
    }
    for (; r0 < n_rows; r0 += nw * R) {
        const int64_t r = r0 + grp;
        const int64_t a = na, b = nb;
        const int64_t rn = r + nw * R;
        na = rn < n_rows ? row_ptr[rn] : 0;
        nb = rn < n_rows ? row_ptr[rn + 1] : 0;
        float v[RSM_KEEP];
        float m = -INFINITY;
#pragma unroll
        for (int t = 0; t < RSM_KEEP; ++t) {
            const int64_t e = a + sub + t * L;
            v[t] = e < b ? aff[e] : -INFINITY;
            m = fmaxf(m, v[t]);
        }
        for (int64_t e = a + sub + RSM_KEEP * L; e < b; e += L) m = fmaxf(m, aff[e]);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < RSM_KEEP; ++t)
            if (a + sub + t * L < b) s += expf(v[t] - m);
        for (int64_t e = a + sub + RSM_KEEP * L; e < b; e += L) s += expf(aff[e] - m);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (b > a) {
            const float2 stat = make_float2(m, 1.f / s);
            if (rstat && sub == 0) rstat[r] = stat;
#pragma unroll
            for (int t = 0; t < RSM_KEEP; ++t) {
                const int64_t e = a + sub + t * L;
                if (e < b) w[e] = row_softmax_weight(v[t], stat);
            }
            for (int64_t e = a + sub + RSM_KEEP * L; e < b; e += L)
                w[e] = row_softmax_weight(aff[e], stat);
        }
    }
}

cudaError_t launch_row_softmax(const int64_t *row_ptr, const float *aff, float *w, int64_t n_rows,
                               float2 *rstat, cudaStream_t st) {
    if (n_rows <= 0) return cudaSuccess;
    const int64_t want = ceil_div<int64_t>(n_rows, 32 / RSM_LANES);
    const int64_t warps = want < (int64_t)device_sm_count() * 64 ? want : (int64_t)device_sm_count() * 64;
    k_row_softmax<<<(unsigned)ceil_div<int64_t>(warps * 32, 256), 256, 0, st>>>(row_ptr, aff, w,
                                                                              n_rows, rstat);
    return cudaGetLastError();
}

// In-degree of every store row (targets mapped from chunk IDs to rows).
__global__ void k_in_degree(const int32_t *__restrict__ col, const int32_t *__restrict__ row_of,
                            int64_t nnz, unsigned long long *__restrict__ deg) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&deg[row_of[col[e]]], 1ull);
}

cudaError_t launch_in_degree(const int32_t *col, const int32_t *row_of, int64_t nnz, int64_t *deg,
                             cudaStream_t st) {
    if (nnz <= 0) return cudaSuccess;
    int grid = (int)(nnz / 256 + 1 < (int64_t)device_sm_count() * 16 ? nnz / 256 + 1
                                                                     : device_sm_count() * 16);
    k_in_degree<<<grid, 256, 0, st>>>(col, row_of, nnz, (unsigned long long *)deg);
    return cudaGetLastError();
}

// keys[i] = row_of[ids[sel ? sel[i] : i]]: chunk IDs (of edge sources or
// targets) mapped to store rows, optionally through a permutation.
__global__ void k_map_keys(const uint32_t *__restrict__ sel, const int32_t *__restrict__ ids,
                           const int32_t *__restrict__ row_of, uint32_t *__restrict__ keys,
                           int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = (uint32_t)row_of[ids[sel ? sel[i] : (uint32_t)i]];
}

cudaError_t launch_map_keys(const uint32_t *sel, const int32_t *ids, const int32_t *row_of,
                            uint32_t *keys, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_map_keys<<<device_sm_count() * 8, 256, 0, st>>>(sel, ids, row_of, keys, n);
    return cudaGetLastError();
}

__global__ void k_iota_u32(uint32_t *__restrict__ v, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        v[i] = (uint32_t)i;
}

cudaError_t launch_iota(uint32_t *v, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_iota_u32<<<device_sm_count() * 8, 256, 0, st>>>(v, n);
    return cudaGetLastError();
}

__global__ void k_gather_in(const uint32_t *__restrict__ order, const int32_t *__restrict__ src,
                            const int32_t *__restrict__ row_of, const float *__restrict__ w,
                            const float *__restrict__ aff, int32_t *__restrict__ in_src,
                            float *__restrict__ in_w, float *__restrict__ in_aff, int64_t nnz) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz;
         p += (int64_t)gridDim.x * blockDim.x) {
        uint32_t e = order[p];
        in_src[p] = row_of[src[e]];
        in_w[p] = w[e];
        in_aff[p] = aff[e];
    }
}

cudaError_t launch_gather_in(const uint32_t *order, const int32_t *src, const int32_t *row_of,
                             const float *w, const float *aff, int32_t *in_src, float *in_w,
                             float *in_aff, int64_t nnz, cudaStream_t st) {
    if (nnz <= 0) return cudaSuccess;
    k_gather_in<<<device_sm_count() * 8, 256, 0, st>>>(order, src, row_of, w, aff, in_src, in_w,
                                                       in_aff, nnz);
    return cudaGetLastError();
}

// Lay out one append batch in page order: row first+i of the store takes
// chunk first+order[i] (embedding row, page, ID maps).  One warp per row.
__global__ void k_batch_layout(const uint32_t *__restrict__ order, int64_t first, int64_t n,
                               int dim, const uint16_t *__restrict__ emb_in,
                               uint16_t *__restrict__ emb, const int32_t *__restrict__ page_in,
                               int64_t first_page, int per_page, int32_t *__restrict__ page_row,
                               int32_t *__restrict__ ext_of, int32_t *__restrict__ row_of) {
    griddep_wait();
    const int lane = threadIdx.x & 31;
    int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int words = dim / 8;   // 16-byte words per row (dim is a multiple of 64)
    for (; i < n; i += stride) {
        const int64_t o = order ? (int64_t)order[i] : i;
        const uint4 *src = (const uint4 *)(emb_in + o * dim);
        uint4 *dst = (uint4 *)(emb + (first + i) * dim);
        for (int t = lane; t < words; t += 32) dst[t] = src[t];
        if (lane == 0) {
            ext_of[first + i] = (int32_t)(first + o);
            row_of[first + o] = (int32_t)(first + i);
            page_row[first + i] = page_in ? page_in[o] : (int32_t)(first_page + o / per_page);
        }
    }
}

cudaError_t launch_batch_layout(const uint32_t *order, int64_t first, int64_t n, int dim,
                                const uint16_t *emb_in, uint16_t *emb, const int32_t *page_in,
                                int64_t first_page, int per_page, int32_t *page_row,
                                int32_t *ext_of, int32_t *row_of, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    launch_pdl(k_batch_layout, dim3((unsigned)(device_sm_count() * 8)), dim3(256), 0, st, order,
               first, n, dim, emb_in, emb, page_in, first_page, per_page, page_row, ext_of, row_of);
    return cudaGetLastError();
}

// out[row_of[first + i]] = in[i] for i < n (per-chunk values into row order).
__global__ void k_scatter_by_row(const int32_t *__restrict__ in, const int32_t *__restrict__ row_of,
                                 int64_t first, int64_t n, int32_t *__restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[row_of[first + i]] = in[i];
}

cudaError_t launch_scatter_by_row(const int32_t *in, const int32_t *row_of, int64_t first,
                                  int64_t n, int32_t *out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_scatter_by_row<<<device_sm_count() * 2, 256, 0, st>>>(in, row_of, first, n, out);
    return cudaGetLastError();
}

// Split plan.  A row with more than SPLIT_T in-edges is cut at every source
// window boundary (sources are sorted within a row, so the cut points are
// found by binary search) and then every SEG_LEN edges.
__device__ __forceinline__ int64_t lower_bound_src(const int32_t *__restrict__ src, int64_t lo,
                                                   int64_t hi, int64_t key) {
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int64_t)src[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// A hub row (more than split_t in-edges, sorted by source row) cut by one
// warp: lane l takes source windows w0 + l, w0 + l + 32, ...; a window starts
// where a binary search finds its first source and ends where the next lane's
// starts, and its segments (at most seg_len edges each) are numbered by a scan
// across the lanes in window order; emit(segment, first edge, end, window) for
// each.  Returns the row's segment count (on every lane).
template <typename Emit>
__device__ int64_t warp_segments(const SplitParams &sp, const int32_t *__restrict__ in_src,
                                 int64_t a, int64_t b, Emit emit) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = (int64_t)in_src[a] / sp.win_rows, w1 = (int64_t)in_src[b - 1] / sp.win_rows;
    int64_t base = 0;
    for (int64_t wb = w0; wb <= w1; wb += 32) {
        const int64_t w = wb + lane;
        const int64_t lo = w == w0 ? a : (w <= w1 ? lower_bound_src(in_src, a, b, w * sp.win_rows) : b);
        int64_t hi = __shfl_down_sync(0xffffffffu, lo, 1);
        if (lane == 31) hi = w < w1 ? lower_bound_src(in_src, lo, b, (w + 1) * sp.win_rows) : b;
        const int64_t cnt = w <= w1 ? (hi - lo + sp.seg_len - 1) / sp.seg_len : 0;
        int64_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        for (int64_t t = 0; t < cnt; ++t) {
            const int64_t e = lo + t * sp.seg_len;
            emit(base + incl - cnt + t, e, e + sp.seg_len < hi ? e + sp.seg_len : hi, w);
        }
        base += __shfl_sync(0xffffffffu, incl, 31);
    }
    return base;
}

// The hub rows (more than split_t in-edges) in row order, and their number, in
// ordered tiles (tile_base).
constexpr int HEAVY_TILE = 1024;
template <bool WRITE>
__global__ __launch_bounds__(256) void k_heavy_rows(const int64_t *__restrict__ in_ptr, int64_t n,
                                                    int64_t split_t, int32_t *__restrict__ rows,
                                                    int64_t *__restrict__ n_rows,
                                                    int32_t *__restrict__ counts) {
    griddep_wait();
    const int t = threadIdx.x;
    const int64_t tile = blockIdx.x;
    if (WRITE && counts[tile] == 0 && tile != gridDim.x - 1) return;
    unsigned bal[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t i = tile * HEAVY_TILE + q * 256 + t;
        bal[q] = __ballot_sync(0xffffffffu, i < n && in_ptr[i + 1] - in_ptr[i] > split_t);
    }
    int places[4];
    const int own = tile_places(bal, places);
    if constexpr (!WRITE) {
        if (t == 0) counts[tile] = own;
    } else {
        const int64_t base = tile_base(counts, 0, tile);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if ((bal[q] >> (t & 31)) & 1u)
                rows[base + places[q]] = (int32_t)(tile * HEAVY_TILE + q * 256 + t);
        if (t == 0 && tile == gridDim.x - 1) *n_rows = base + own;
    }
}

// Segment count of every hub row, a warp a row (0 past them, for the scan).  (A
// warp that walked 32 rows of the store and cut the hubs among them one after
// another took 56 us at 524,288 chunks, as a cut is a chain of ~20 dependent
// loads.)
__global__ __launch_bounds__(256) void k_hub_segs(SplitParams sp,
                                                  const int64_t *__restrict__ in_ptr,
                                                  const int32_t *__restrict__ in_src,
                                                  const int32_t *__restrict__ rows,
                                                  const int64_t *__restrict__ n_rows,
                                                  int64_t max_hubs, int64_t *__restrict__ nseg) {
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t n = *n_rows, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = gt >> 5; i < n; i += nw) {
        const int64_t r = rows[i];
        const int64_t c = warp_segments(sp, in_src, in_ptr[r], in_ptr[r + 1],
                                        [](int64_t, int64_t, int64_t, int64_t) {});
        if (lane == 0) nseg[i] = c;
    }
    for (int64_t i = n + gt; i < max_hubs; i += nw * 32) nseg[i] = 0;
}

// The plan of every hub row, a warp each: its segments with their window and
// their owner, and the row's place by segment count (key n_segs - count, so
// that ascending keys are heaviest first).
__global__ void k_hub_fill(SplitParams sp, const int64_t *__restrict__ in_ptr,
                           const int32_t *__restrict__ in_src, const int32_t *__restrict__ rows,
                           const int64_t *__restrict__ slot0, int64_t n_rows, int64_t n_segs,
                           int32_t *__restrict__ split_row, int64_t *__restrict__ split_slot0,
                           int64_t *__restrict__ seg_e0, int64_t *__restrict__ seg_e1,
                           uint32_t *__restrict__ seg_win, uint32_t *__restrict__ seg_id,
                           int32_t *__restrict__ slot_split, uint32_t *__restrict__ row_key,
                           uint32_t *__restrict__ row_id) {
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n_rows; i += nw) {
        const int64_t r = rows[i], slot = slot0[i];
        const int64_t cnt = warp_segments(
            sp, in_src, in_ptr[r], in_ptr[r + 1], [&](int64_t s, int64_t e0, int64_t e1, int64_t w) {
                seg_e0[slot + s] = e0;
                seg_e1[slot + s] = e1;
                seg_win[slot + s] = (uint32_t)w;
                seg_id[slot + s] = (uint32_t)(slot + s);
                slot_split[slot + s] = (int32_t)i;
            });
        if (lane == 0) {
            split_row[i] = (int32_t)r;
            split_slot0[i] = slot;
            if (i == n_rows - 1) split_slot0[n_rows] = n_segs;
            row_key[i] = (uint32_t)(n_segs - cnt);
            row_id[i] = (uint32_t)i;
        }
    }
}

__global__ void k_seg_permute(const uint32_t *__restrict__ order, const int64_t *__restrict__ e0,
                              const int64_t *__restrict__ e1, int64_t n_segs,
                              int64_t *__restrict__ e0s, int64_t *__restrict__ e1s,
                              int32_t *__restrict__ slot) {
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_segs;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t o = order[i];
        e0s[i] = e0[o];
        e1s[i] = e1[o];
        slot[i] = (int32_t)o;
    }
}

int64_t hub_plan_words(int64_t n, int64_t max_hubs) {
    return ceil_div<int64_t>(tile_words(ceil_div<int64_t>(n, HEAVY_TILE)), 2) + max_hubs +
           (int64_t)(scan_tmp_bytes(max_hubs) / 8) + 1;
}

cudaError_t launch_hub_count(const SplitParams &sp, const int64_t *in_ptr, const int32_t *in_src,
                             int64_t n, int64_t max_hubs, int32_t *rows, int64_t *slot0,
                             int64_t *counts, int64_t *scratch, cudaStream_t st) {
    const int64_t tiles = ceil_div<int64_t>(n, HEAVY_TILE);
    if (n <= 0 || max_hubs <= 0) {
        cudaError_t e = cudaMemsetAsync(counts, 0, 8, st);
        return e == cudaSuccess ? cudaMemsetAsync(slot0 + (max_hubs > 0 ? max_hubs : 0), 0, 8, st) : e;
    }
    int32_t *tc = (int32_t *)scratch;
    int64_t *nseg = scratch + ceil_div<int64_t>(tile_words(tiles), 2);
    launch_pdl(k_heavy_rows<false>, dim3((unsigned)tiles), dim3(256), 0, st, in_ptr, n, sp.split_t,
               rows, counts, tc);
    cudaError_t e = launch_tile_groups(tc, tiles, st);
    if (e != cudaSuccess) return e;
    launch_pdl(k_heavy_rows<true>, dim3((unsigned)tiles), dim3(256), 0, st, in_ptr, n, sp.split_t,
               rows, counts, tc);
    const int64_t want = ceil_div<int64_t>(max_hubs, 8), cap = (int64_t)device_sm_count() * 8;
    launch_pdl(k_hub_segs, dim3((unsigned)(want < cap ? want : cap)), dim3(256), 0, st, sp, in_ptr,
               in_src, rows, counts, max_hubs, nseg);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return scan_exclusive(nseg, slot0, max_hubs, nseg + max_hubs, scan_tmp_bytes(max_hubs), st);
}

cudaError_t launch_hub_fill(const SplitParams &sp, const int64_t *in_ptr, const int32_t *in_src,
                            const int32_t *rows, const int64_t *slot0, int64_t n_rows,
                            int64_t n_segs, int32_t *split_row, int64_t *split_slot0,
                            int64_t *seg_e0, int64_t *seg_e1, uint32_t *seg_win, uint32_t *seg_id,
                            int32_t *slot_split, uint32_t *row_key, uint32_t *row_id,
                            cudaStream_t st) {
    if (n_rows <= 0) return cudaSuccess;
    const int64_t want = ceil_div<int64_t>(n_rows, 4), cap = (int64_t)device_sm_count() * 16;
    launch_pdl(k_hub_fill, dim3((unsigned)(want < cap ? want : cap)), dim3(128), 0, st, sp, in_ptr,
               in_src, rows, slot0, n_rows, n_segs, split_row, split_slot0, seg_e0, seg_e1,
               seg_win, seg_id, slot_split, row_key, row_id);
    return cudaGetLastError();
}

cudaError_t launch_seg_permute(const uint32_t *order, const int64_t *e0, const int64_t *e1,
                               int64_t n_segs, int64_t *e0s, int64_t *e1s, int32_t *slot,
                               cudaStream_t st) {
    if (n_segs <= 0) return cudaSuccess;
    launch_pdl(k_seg_permute, dim3((unsigned)(device_sm_count() * 2)), dim3(256), 0, st, order, e0,
               e1, n_segs, e0s, e1s, slot);
    return cudaGetLastError();
}

// ================================================================== propagation hop
// out[j,:] = u[j,:] + alpha * sum_{i->j} w_ij in[i,:], gathered over the
// in-edge CSR, one warp per destination row.  A row holds BP fp32 values
// (BP/4 float4).  For BP >= 128 each lane owns BP/128 float4 of the row; for
// smaller BP the warp splits into 32/(BP/4) lane groups that take
// alternate edges and are summed at the end.  Rows with more than split_t
// in-edges are skipped here and handled by window segments + fixup.
// L2 policy for the hop: gathered source rows are re-read ~32 times (once
// per out-edge of the source), so they are loaded with an evict-last
// policy; everything read or written once (graph arrays, u, the output
// slab, partial sums) streams with evict-first (.cs) accesses so that it
// does not push gathered rows out of L2.
__device__ __forceinline__ uint64_t l2_keep_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ float4 ld_keep(const float4 *p, uint64_t pol) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float4 ld_stream(const float4 *p) { return __ldcs(p); }
__device__ __forceinline__ void st_stream(float4 *p, float4 v) { __stcs(p, v); }
__device__ __forceinline__ int32_t ld_stream(const int32_t *p) { return __ldcs(p); }
__device__ __forceinline__ float ld_stream(const float *p) { return __ldcs(p); }

template <int BP>
struct HopShape {
    static constexpr int F = BP / 4;                       // float4 per row
    static constexpr int G = F >= 32 ? 1 : 32 / F;         // edge groups per warp
    static constexpr int V = F >= 32 ? F / 32 : 1;         // float4 per lane
    static constexpr int LW = F >= 32 ? 32 : F;            // lanes per group
};

template <int BP, int WIDTH = 1>
__device__ __forceinline__ void hop_accumulate(const int32_t *__restrict__ in_src,
                                               const float *__restrict__ in_w, int64_t e0,
                                               int64_t e1, const float4 *__restrict__ in4,
                                               float4 (&acc)[HopShape<BP>::V]) {
    using S = HopShape<BP>;
    // gathers in flight: UN edges x V float4 (WIDTH times more in the wide
    // variant, which runs fewer warps)
    constexpr int UN = WIDTH * (8 / S::V > 0 ? 8 / S::V : 1);
    const int lane = threadIdx.x & 31;
    const int g = lane / S::LW, sub = lane % S::LW;
    const uint64_t pol = l2_keep_policy();
#pragma unroll
    for (int v = 0; v < S::V; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    // the next batch's (source, weight) pairs are loaded while this batch gathers
    int32_t s_n = 0;
    float w_n = 0.f;
    if (e0 + lane < e1) {
        s_n = ld_stream(in_src + e0 + lane);
        w_n = ld_stream(in_w + e0 + lane);
    }
    for (int64_t eb = e0; eb < e1; eb += 32) {
        const int cnt = (int)(e1 - eb < 32 ? e1 - eb : 32);
        const int32_t s_l = s_n;
        const float w_l = w_n;
        if (eb + 32 + lane < e1) {
            s_n = ld_stream(in_src + eb + 32 + lane);
            w_n = ld_stream(in_w + eb + 32 + lane);
        }
        int t = 0;
        for (; t + UN * S::G <= cnt; t += UN * S::G) {
            int32_t sq[UN];
            float wq[UN];
#pragma unroll
            for (int q = 0; q < UN; ++q) {
                sq[q] = __shfl_sync(0xffffffffu, s_l, t + q * S::G + g);
                wq[q] = __shfl_sync(0xffffffffu, w_l, t + q * S::G + g);
            }
            float4 x[UN][S::V];
#pragma unroll
            for (int q = 0; q < UN; ++q)
#pragma unroll
                for (int v = 0; v < S::V; ++v)
                    x[q][v] = ld_keep(in4 + (int64_t)sq[q] * S::F + sub + 32 * v, pol);
#pragma unroll
            for (int q = 0; q < UN; ++q)
#pragma unroll
                for (int v = 0; v < S::V; ++v) {
                    acc[v].x = fmaf(wq[q], x[q][v].x, acc[v].x);
                    acc[v].y = fmaf(wq[q], x[q][v].y, acc[v].y);
                    acc[v].z = fmaf(wq[q], x[q][v].z, acc[v].z);
                    acc[v].w = fmaf(wq[q], x[q][v].w, acc[v].w);
                }
        }
        for (; t < cnt; t += S::G) {
            const int idx = t + g;
            int32_t sv = __shfl_sync(0xffffffffu, s_l, idx < 32 ? idx : 31);
            float wv = __shfl_sync(0xffffffffu, w_l, idx < 32 ? idx : 31);
            if (idx < cnt) {
#pragma unroll
                for (int v = 0; v < S::V; ++v) {
                    float4 x = ld_keep(in4 + (int64_t)sv * S::F + sub + 32 * v, pol);
                    acc[v].x = fmaf(wv, x.x, acc[v].x);
                    acc[v].y = fmaf(wv, x.y, acc[v].y);
                    acc[v].z = fmaf(wv, x.z, acc[v].z);
                    acc[v].w = fmaf(wv, x.w, acc[v].w);
                }
            }
        }
    }
    if (S::G > 1) {
#pragma unroll
        for (int o = S::LW; o < 32; o <<= 1) {
#pragma unroll
            for (int v = 0; v < S::V; ++v) {
                acc[v].x += __shfl_xor_sync(0xffffffffu, acc[v].x, o);
                acc[v].y += __shfl_xor_sync(0xffffffffu, acc[v].y, o);
                acc[v].z += __shfl_xor_sync(0xffffffffu, acc[v].z, o);
                acc[v].w += __shfl_xor_sync(0xffffffffu, acc[v].w, o);
            }
        }
    }
}

// ------------------------------------------------------------------ row bounds
// Scalar bounds on the hops' fp32 values, one pair per row: U[j] is at least
// and L[j] at most every real query column's value of s^(h)_j.  Level 0 is
// u's row maximum / minimum (from the score step); level h follows the hop
// s^(h)_j = fma(alpha, sum_{i->j} w_ij s^(h-1)_i, u_j) with the sums of
// w * U and w * L over the row's in-edges (w, s >= 0), widened for rounding by
// n, the terms one after another in either sum: the row's in-edges where it is
// kept whole, else a segment's edges and the row's segments (what the hop adds
// in sequence; the bound's own sums add a 32nd of a segment, then the
// segments).  The hop's sum takes at most 2n + 10 roundings on any term's path
// and the bound's own sum at most n + 5, so exp(+-x), x = 3.25 (n + 8) 2^-24,
// covers both (with 1 + x + x^2 >= exp(x) and 1 - x <= exp(-x) for 0 <= x <=
// 1), and a factor 1 -+ 4e-6 (~67 ulp) covers the final rounding of the hop
// and of evaluating the bound in fp32.  (n = the in-degree widened a hub of
// 2 * 10^5 in-edges by 4% a level, as much as u itself varies.)
__device__ __forceinline__ float bound_x(int64_t n) {
    return 3.25f * (float)(n + 8) * 5.9604645e-8f;
}
__device__ __forceinline__ float bound_up(float u0, float v, int64_t n, float alpha) {
    const float x = bound_x(n);
    if (!(x <= 1.f)) return INFINITY;
    return fmaf(alpha * v, 1.f + x + x * x, u0) * (1.f + 4e-6f);
}
__device__ __forceinline__ float bound_dn(float l0, float v, int64_t n, float alpha) {
    const float x = bound_x(n);
    const float g = x < 1.f ? 1.f - x : 0.f;
    return fmaf(alpha * v, g, l0) * (1.f - 4e-6f);
}

// The sums of w * U[source] and w * L[source] over in-edges e0..e1, by a
// group of LN lanes (lane `sl` of the group), four edges in flight per lane;
// every lane of the group returns them.
template <int LN>
__device__ __forceinline__ void bound_sums(const int32_t *__restrict__ in_src,
                                           const float *__restrict__ in_w, int64_t e0, int64_t e1,
                                           const float *__restrict__ U, const float *__restrict__ L,
                                           int sl, float &vu, float &vl) {
    vu = 0.f;
    vl = 0.f;
    for (int64_t eb = e0 + sl; eb < e1; eb += 4 * LN) {
        int32_t s[4];
        float w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t e = eb + LN * q;
            s[q] = e < e1 ? __ldcs(in_src + e) : 0;
            w[q] = e < e1 ? __ldcs(in_w + e) : 0.f;
        }
        float a[4], c[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool in = eb + LN * q < e1;
            a[q] = in ? __ldg(U + s[q]) : 0.f;
            c[q] = in ? __ldg(L + s[q]) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            vu = fmaf(w[q], a[q], vu);
            vl = fmaf(w[q], c[q], vl);
        }
    }
#pragma unroll
    for (int off = LN / 2; off > 0; off >>= 1) {
        vu += __shfl_xor_sync(0xffffffffu, vu, off);
        vl += __shfl_xor_sync(0xffffffffu, vl, off);
    }
}

// One level for the rows kept whole: four lanes per row, eight rows per warp.
constexpr int BND_LANES = 4;
__global__ void k_bound_rows(const int64_t *__restrict__ in_ptr, const int32_t *__restrict__ in_src,
                             const float *__restrict__ in_w, int64_t n, int64_t split_t,
                             const float *__restrict__ u0, const float *__restrict__ l0,
                             const float *__restrict__ Up, const float *__restrict__ Lp,
                             float alpha, float *__restrict__ Un, float *__restrict__ Ln) {
    constexpr int R = 32 / BND_LANES;
    const int lane = threadIdx.x & 31, sl = lane % BND_LANES, grp = lane / BND_LANES;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * R; r0 < n;
         r0 += nw * R) {
        const int64_t j = r0 + grp;
        int64_t e0 = 0, e1 = 0;
        if (j < n) {
            e0 = in_ptr[j];
            e1 = in_ptr[j + 1];
        }
        const bool whole = j < n && e1 - e0 <= split_t;
        float vu, vl;
        bound_sums<BND_LANES>(in_src, in_w, e0, whole ? e1 : e0, Up, Lp, sl, vu, vl);
        if (whole && sl == 0) {
            Un[j] = bound_up(u0[j], vu, e1 - e0, alpha);
            Ln[j] = bound_dn(l0[j], vl, e1 - e0, alpha);
        }
    }
}

// Split rows: one warp per segment, its sums added into the owning row's
// totals (the order of the additions does not change the bound: every
// term is >= 0 and a term's path stays within a segment's edges + the row's
// segments + 5 roundings) ...
__global__ void k_seg_bound(const int64_t *__restrict__ seg_e0, const int64_t *__restrict__ seg_e1,
                            const int32_t *__restrict__ seg_slot, int64_t n_segs,
                            const int32_t *__restrict__ slot_split,
                            const int32_t *__restrict__ in_src, const float *__restrict__ in_w,
                            const float *__restrict__ Up, const float *__restrict__ Lp,
                            float *__restrict__ split_vu, float *__restrict__ split_vl) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < n_segs; s += nw) {
        float vu, vl;
        bound_sums<32>(in_src, in_w, seg_e0[s], seg_e1[s], Up, Lp, lane, vu, vl);
        if (lane == 0) {
            const int32_t r = slot_split[seg_slot[s]];
            atomicAdd(split_vu + r, vu);
            atomicAdd(split_vl + r, vl);
        }
    }
}

// ... then each split row's bounds.
__global__ void k_split_bound(const int64_t *__restrict__ in_ptr, int64_t n_split,
                              const int32_t *__restrict__ split_row,
                              const int64_t *__restrict__ split_slot0, int64_t seg_len,
                              const float *__restrict__ u0, const float *__restrict__ l0,
                              const float *__restrict__ split_vu, const float *__restrict__ split_vl,
                              float alpha, float *__restrict__ Un, float *__restrict__ Ln) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_split;
         r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = split_row[r];
        const int64_t edges = in_ptr[j + 1] - in_ptr[j];
        const int64_t path = seg_len + (split_slot0[r + 1] - split_slot0[r]);
        const int64_t n = edges < path ? edges : path;
        Un[j] = bound_up(u0[j], split_vu[r], n, alpha);
        Ln[j] = bound_dn(l0[j], split_vl[r], n, alpha);
    }
}

__global__ void k_fill_f32(float *__restrict__ v, int64_t n, float x) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        v[i] = x;
}

cudaError_t launch_fill_f32(float *v, int64_t n, float x, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_fill_f32<<<device_sm_count() * 2, 256, 0, st>>>(v, n, x);
    return cudaGetLastError();
}

cudaError_t launch_mass_levels(const HopPlan &p, int t0, int t1, float *mup, float *mdn,
                               const float *zeros, float *split_vu, float *split_vl,
                               cudaStream_t st) {
    const int sms = device_sm_count();
    const int64_t n = p.n;
    for (int t = t0; t <= t1; ++t) {
        const float *Up = mup + (int64_t)(t - 1) * n, *Lp = mdn + (int64_t)(t - 1) * n;
        float *Un = mup + (int64_t)t * n, *Ln = mdn + (int64_t)t * n;
        const int64_t want = ceil_div<int64_t>(n, 32);
        const int g = (int)(want < (int64_t)sms * 8 ? (want < 1 ? 1 : want) : (int64_t)sms * 8);
        k_bound_rows<<<g, 256, 0, st>>>(p.in_ptr, p.in_src, p.in_w, n, p.split.split_t, zeros,
                                         zeros, Up, Lp, 1.f, Un, Ln);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (p.n_split_rows > 0) {
            e = cudaMemsetAsync(split_vu, 0, (size_t)p.n_split_rows * 4, st);
            if (e == cudaSuccess) e = cudaMemsetAsync(split_vl, 0, (size_t)p.n_split_rows * 4, st);
            if (e != cudaSuccess) return e;
            const int64_t ws = ceil_div<int64_t>(p.n_segs, 8);
            const int gs = (int)(ws < (int64_t)sms * 8 ? (ws < 1 ? 1 : ws) : (int64_t)sms * 8);
            k_seg_bound<<<gs, 256, 0, st>>>(p.seg_e0, p.seg_e1, p.seg_slot, p.n_segs,
                                            p.slot_split, p.in_src, p.in_w, Up, Lp, split_vu,
                                            split_vl);
            const int64_t wr = ceil_div<int64_t>(p.n_split_rows, 256);
            const int gr = (int)(wr < (int64_t)sms * 2 ? wr : (int64_t)sms * 2);
            k_split_bound<<<gr, 256, 0, st>>>(p.in_ptr, p.n_split_rows, p.split_row, p.split_slot0,
                                              p.split.seg_len, zeros, zeros,
                                              split_vu, split_vl, 1.f, Un, Ln);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

// Last hop, after the floor: the rows kept whole whose upper bound reaches
// their floor (kept_rows), the split rows that do not (split_skip), and the
// segments of the split rows that do (kept_segs), over rows, split rows and
// segments, in ordered tiles (tile_base): both lists are in row order and in
// window-major order, the order that keeps gathered source rows in L2 (in the
// order of the tiles' finish the last hop took 363 instead of 317 us on 500,009
// chunks, 100 scoped queries).  The bounds are evaluated
// here: no per-row arrays are
// written (eleven launches did this; with the floor 102 -> 60 us there, 34 ->
// 11 us on 4096 chunks).
constexpr int KEEP_TILE = 1024;
// k_keep_mark tests (a bit an item in bits, a count a tile), k_keep_list writes
// the lists.
__global__ __launch_bounds__(256) void k_keep_mark(const RowBounds rb,
                                                   const float *__restrict__ floor_p,
                                                   const NsFloors nf,
                                                   const int64_t *__restrict__ in_ptr,
                                                   int64_t split_t, int64_t n_split,
                                                   const int32_t *__restrict__ split_row,
                                                   int64_t n_segs,
                                                   const int32_t *__restrict__ seg_slot,
                                                   const int32_t *__restrict__ slot_split,
                                                   int32_t *__restrict__ split_skip,
                                                   int32_t *__restrict__ counts,
                                                   uint32_t *__restrict__ bits,
                                                   const int32_t *__restrict__ done) {
    __shared__ int own;
    __shared__ int32_t tag_s[PF_TAGS];
    __shared__ float tag_floor_s[PF_TAGS];
    griddep_wait();
    if (done && done[0] == 1) return;
    const int t = threadIdx.x;
    const float floor_ = *floor_p, umax = ext_umax(rb.ext);
    int n_tags = 0;
    if (nf.ns_row) {
        n_tags = *nf.n_tags;
        for (int i = t; i < n_tags; i += 256) {
            tag_s[i] = nf.tags[i];
            tag_floor_s[i] = nf.tag_floor[i];
        }
        __syncthreads();
    }
    auto reaches = [&](int64_t j) {
        const float ub = row_upper_bound(rb.u0, rb.mup, rb.n, rb.H, rb.alpha, umax, j);
        if (!(ub >= floor_)) return false;
        if (!nf.ns_row) return true;
        const int32_t tag = nf.ns_row[j];
        int lo = 0, hi = n_tags;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (tag_s[mid] < tag) lo = mid + 1;
            else hi = mid;
        }
        return lo < n_tags && tag_s[lo] == tag && ub >= tag_floor_s[lo];
    };
    // tiles of rows, of segments, of split rows
    const int64_t row_tiles = (rb.n + KEEP_TILE - 1) / KEEP_TILE;
    const int64_t seg_tiles = (n_segs + KEEP_TILE - 1) / KEEP_TILE;
    const int64_t tile = blockIdx.x;
    if (tile >= row_tiles + seg_tiles) {
        for (int q = 0; q < KEEP_TILE / 256; ++q) {
            const int64_t r = (tile - row_tiles - seg_tiles) * KEEP_TILE + q * 256 + t;
            if (r < n_split) split_skip[r] = reaches(split_row[r]) ? 0 : 1;
        }
        return;
    }
    if (t == 0) own = 0;
    __syncthreads();
    const bool rows = tile < row_tiles;
    const int64_t i0 = (rows ? tile : tile - row_tiles) * KEEP_TILE;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t i = i0 + q * 256 + t;
        bool k = false;
        if (rows) k = i < rb.n && reaches(i) && in_ptr[i + 1] - in_ptr[i] <= split_t;
        else k = i < n_segs && reaches(split_row[slot_split[seg_slot[i]]]);
        const unsigned bal = __ballot_sync(0xffffffffu, k);
        if ((t & 31) == 0) {
            bits[tile * 32 + q * 8 + (t >> 5)] = bal;
            if (bal) atomicAdd(&own, __popc(bal));
        }
    }
    __syncthreads();
    if (t == 0) counts[tile] = own;
}

__global__ __launch_bounds__(256) void k_keep_list(int64_t row_tiles, int64_t seg_tiles,
                                                   const int32_t *__restrict__ counts,
                                                   const uint32_t *__restrict__ bits,
                                                   int32_t *__restrict__ kept_rows,
                                                   int32_t *__restrict__ kept_segs,
                                                   int64_t *__restrict__ kept_count,
                                                   const int32_t *__restrict__ done) {
    griddep_wait();
    if (done && done[0] == 1) return;
    const int t = threadIdx.x;
    const int64_t tile = blockIdx.x;
    const bool rows = tile < row_tiles;
    const bool last = tile == (rows ? row_tiles : row_tiles + seg_tiles) - 1;
    const int own = counts[tile];
    if (own == 0 && !last) return;   // nothing to write, no total to tell
    const int64_t base = tile_base(counts, rows ? 0 : row_tiles, tile);
    if (last && t == 0) kept_count[rows ? 0 : 1] = base + own;
    if (own == 0) return;
    unsigned bal[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) bal[q] = bits[tile * 32 + q * 8 + (t >> 5)];
    int places[4];
    tile_places(bal, places);
    int32_t *out = rows ? kept_rows : kept_segs;
    const int64_t i0 = (rows ? tile : tile - row_tiles) * KEEP_TILE;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if ((bal[q] >> (t & 31)) & 1u) out[base + places[q]] = (int32_t)(i0 + q * 256 + t);
}

static int64_t keep_tiles(const HopPlan &p) {
    return ceil_div<int64_t>(p.n, KEEP_TILE) + ceil_div<int64_t>(p.n_segs, KEEP_TILE);
}
int64_t keep_words(const HopPlan &p) {
    return tile_words(keep_tiles(p)) + keep_tiles(p) * (KEEP_TILE / 32);
}

cudaError_t launch_keep(const HopPlan &p, const RowBounds &rb, const float *floor_p,
                        const NsFloors *nf, int32_t *split_skip, int32_t *kept_rows,
                        int32_t *kept_segs, int64_t *kept_count, int32_t *words, cudaStream_t st,
                        int *launches) {
    static_assert(KEEP_TILE == 1024, "tile_places");
    const int64_t tiles = keep_tiles(p), row_tiles = ceil_div<int64_t>(p.n, KEEP_TILE);
    const NsFloors f = nf ? *nf : NsFloors{};
    uint32_t *bits = (uint32_t *)(words + tile_words(tiles));
    cudaError_t e = launch_pdl(
        k_keep_mark, dim3((unsigned)(tiles + ceil_div<int64_t>(p.n_split_rows, KEEP_TILE))),
        dim3(256), 0, st, rb, floor_p, f, p.in_ptr, p.split.split_t, p.n_split_rows, p.split_row,
        p.n_segs, p.seg_slot, p.slot_split, split_skip, words, bits, p.done);
    if (e == cudaSuccess) e = launch_tile_groups(words, tiles, st, launches);
    if (e == cudaSuccess)
        e = launch_pdl(k_keep_list, dim3((unsigned)tiles), dim3(256), 0, st, row_tiles,
                       tiles - row_tiles, (const int32_t *)words, (const uint32_t *)bits, kept_rows,
                       kept_segs, kept_count, p.done);
    if (launches) *launches += 2;
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// A split row: out = u + alpha * (sum of its partial slots a..b-1), summed
// by one warp in slot order (lane groups take alternate slots and are
// added in group order), so the result does not depend on scheduling.
// Filter epilogue: lane `sub` holds columns (sub + 32 v) * 4 + 0..3 of row j.
// thr[BP] holds the column bounds and thr_hi[BP/4] their upper words (the
// score bits), four columns per uint4 so that a lane's test is one
// conflict-free shared load and four 32-bit compares; only a value whose
// bits reach the bound's (rare: ~ a few k per column) takes the 64-bit
// compare and the append.
template <int BP>
__device__ __noinline__ void hop_filter_row(const HopFilter &f, const unsigned long long *thr,
                                           const uint4 *thr_hi, int sub, int64_t j, uint32_t id,
                                           const float4 (&o)[HopShape<BP>::V]) {
#pragma unroll
    for (int v = 0; v < HopShape<BP>::V; ++v) {
        const uint4 h = thr_hi[sub + 32 * v];
        const uint32_t x[4] = {__float_as_uint(o[v].x), __float_as_uint(o[v].y),
                               __float_as_uint(o[v].z), __float_as_uint(o[v].w)};
        const uint32_t hh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (x[e] >= hh[e]) {
                const int c = (sub + 32 * v) * 4 + e;
                const unsigned long long key =
                    ((unsigned long long)x[e] << 32) | (unsigned long long)(~id);
                if (key >= thr[c] && in_scope(f.ns, j, c)) {
                    const unsigned int p = atomicAdd(&f.cnt[c], 1u);
                    if ((int64_t)p < f.cap) f.buf[(int64_t)c * f.cap + p] = key;
                }
            }
        }
    }
}

// Kept out of line: any inlined test here slowed the whole row loop of the
// hop by ~5% (measured), while a call per row costs ~2%.
template <int BP, bool FILTER>
__device__ __forceinline__ void hop_emit(const HopFilter &f, const unsigned long long *thr,
                                         const uint4 *thr_hi, int sub, int64_t j, uint32_t id,
                                         const float4 (&o)[HopShape<BP>::V]) {
    if constexpr (FILTER) hop_filter_row<BP>(f, thr, thr_hi, sub, j, id, o);
}

template <int BP, bool FILTER, int WIDTH = 1>
__device__ __forceinline__ void hop_fixup_row(int64_t j, int64_t a, int64_t b,
                                              const float4 *__restrict__ part4,
                                              const float4 *__restrict__ u4,
                                              float4 *__restrict__ out4, float alpha,
                                              const HopFilter &f,
                                              const unsigned long long *thr,
                                              const uint4 *thr_hi) {
    using S = HopShape<BP>;
    constexpr int P = WIDTH * (8 / S::V > 0 ? 8 / S::V : 1);   // slots in flight per lane group
    const int lane = threadIdx.x & 31;
    const int g = lane / S::LW, sub = lane % S::LW;
    const uint32_t id = FILTER ? (uint32_t)f.ext_of[j] : 0u;
    float4 acc[S::V];
#pragma unroll
    for (int v = 0; v < S::V; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t t = a; t < b; t += P * S::G) {
        float4 x[P][S::V];
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const int64_t sl = t + q * S::G + g;
#pragma unroll
            for (int v = 0; v < S::V; ++v)
                x[q][v] = sl < b ? ld_stream(part4 + sl * S::F + sub + 32 * v)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
            for (int v = 0; v < S::V; ++v) {
                acc[v].x += x[q][v].x; acc[v].y += x[q][v].y;
                acc[v].z += x[q][v].z; acc[v].w += x[q][v].w;
            }
    }
    if (S::G > 1) {
#pragma unroll
        for (int o = S::LW; o < 32; o <<= 1)
#pragma unroll
            for (int v = 0; v < S::V; ++v) {
                acc[v].x += __shfl_xor_sync(0xffffffffu, acc[v].x, o);
                acc[v].y += __shfl_xor_sync(0xffffffffu, acc[v].y, o);
                acc[v].z += __shfl_xor_sync(0xffffffffu, acc[v].z, o);
                acc[v].w += __shfl_xor_sync(0xffffffffu, acc[v].w, o);
            }
    }
    if (lane < S::LW) {
        float4 o[S::V];
#pragma unroll
        for (int v = 0; v < S::V; ++v) {
            o[v] = ld_stream(u4 + j * S::F + sub + 32 * v);
            o[v].x = fmaf(alpha, acc[v].x, o[v].x);
            o[v].y = fmaf(alpha, acc[v].y, o[v].y);
            o[v].z = fmaf(alpha, acc[v].z, o[v].z);
            o[v].w = fmaf(alpha, acc[v].w, o[v].w);
            if constexpr (!FILTER) st_stream(out4 + j * S::F + sub + 32 * v, o[v]);
        }
        hop_emit<BP, FILTER>(f, thr, thr_hi, sub, j, id, o);
    }
}

// With the filter (the last hop) the output slab is not written: the
// selection needs only the keys the filter appends (a query whose buffer
// overflows gets its column recomputed by the merge).
//
// One queue: first the split rows (their segment partials are complete,
// the segment kernel ran before), heaviest first, one warp each; then the
// rows kept whole, ROWS_PER_GRAB consecutive rows per claim (load
// balance), with the group's row pointers read at once and each row's u
// load issued before its gathers.
// WIDTH 2 (the pruned last hop, few work items): twice the loads in flight
// per warp, two CTAs per SM.
template <int BP, bool FILTER, int WIDTH = 1>
__global__ __launch_bounds__(256, WIDTH > 1 ? 2 : 3) void k_hop_rows(const int64_t *__restrict__ in_ptr,
                                                  const int32_t *__restrict__ in_src,
                                                  const float *__restrict__ in_w, int64_t n,
                                                  const float4 *__restrict__ u4,
                                                  const float4 *__restrict__ in4,
                                                  float4 *__restrict__ out4, float alpha,
                                                  int64_t split_t, int64_t n_split,
                                                  const int32_t *__restrict__ split_order,
                                                  const int32_t *__restrict__ split_row,
                                                  const int64_t *__restrict__ split_slot0,
                                                  const float4 *__restrict__ part4,
                                                  HopFilter f,
                                                  const int32_t *__restrict__ split_skip,
                                                  const int32_t *__restrict__ kept_rows,
                                                  const int64_t *__restrict__ kept_count,
                                                  int *__restrict__ queue,
                                                  const int32_t *__restrict__ done) {
    using S = HopShape<BP>;
    griddep_wait();
    if (done && done[0] == 1) return;
    const int lane = threadIdx.x & 31;
    const int sub = lane % S::LW;
    // with the skip (last hop), the rows kept whole that reach the floor
    // come as a compact list; a claim takes ROWS_PER_GRAB rows either way
    const bool listed = FILTER && kept_rows != nullptr;
    const int64_t n_items = listed ? *kept_count : n;
    // (with fewer claims than warps, fewer rows a claim: a row is a chain of
    // dependent loads, and eight in a row left most warps idle on a short
    // list: last hop 314 -> 194 us on 500,009 chunks and 100 scoped queries)
    const int64_t per = n_items / ((int64_t)gridDim.x * (blockDim.x >> 5));
    const int64_t grab = per >= ROWS_PER_GRAB ? ROWS_PER_GRAB : (per < 1 ? 1 : per);
    const int64_t groups = (n_items + grab - 1) / grab;
    __shared__ unsigned long long thr[FILTER ? BP : 1];
    __shared__ uint4 thr_hi[FILTER ? BP / 4 : 1];
    // last hop: rows whose bound stays below the floor append nothing
    const bool prune = FILTER && split_skip != nullptr;
    if constexpr (FILTER) {
        for (int c = threadIdx.x; c < BP; c += blockDim.x) {
            const unsigned long long t = f.bound[c];
            thr[c] = t;
            reinterpret_cast<uint32_t *>(thr_hi)[c] = (uint32_t)(t >> 32);
        }
        __syncthreads();
    }
    while (true) {
        int64_t it = 0;
        if (lane == 0) it = atomicAdd(queue, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n_split + groups) break;
        if (it < n_split) {
            const int32_t r = split_order[it];
            if (prune && split_skip[r]) continue;
            hop_fixup_row<BP, FILTER, WIDTH>(split_row[r], split_slot0[r], split_slot0[r + 1], part4,
                                      u4, out4, alpha, f, thr, thr_hi);
            continue;
        }
        // lane r: the claim's r-th row (consecutive rows, or listed ones),
        // its edge range; `todo`: the rows kept whole
        const int64_t i0 = (it - n_split) * grab;
        const int nr = (int)(n_items - i0 < grab ? n_items - i0 : grab);
        int64_t myrow = 0, p0 = 0, p1 = 0;
        if (lane < nr) {
            myrow = listed ? (int64_t)kept_rows[i0 + lane] : i0 + lane;
            p0 = in_ptr[myrow];
            p1 = in_ptr[myrow + 1];
        }
        const bool want = lane < nr && p1 - p0 <= split_t;
        unsigned todo = __ballot_sync(0xffffffffu, want);
        int32_t ids = 0;
        if (FILTER && want) ids = f.ext_of[myrow];
#pragma unroll 1
        while (todo) {
            const int r = __ffs(todo) - 1;
            todo &= todo - 1;
            const int64_t e0 = __shfl_sync(0xffffffffu, p0, r);
            const int64_t e1 = __shfl_sync(0xffffffffu, p1, r);
            const uint32_t id = FILTER ? (uint32_t)__shfl_sync(0xffffffffu, ids, r) : 0u;
            const int64_t j = __shfl_sync(0xffffffffu, myrow, r);
            float4 b[S::V];
            if (lane < S::LW) {
#pragma unroll
                for (int v = 0; v < S::V; ++v) b[v] = ld_stream(u4 + j * S::F + sub + 32 * v);
            }
            float4 acc[S::V];
            hop_accumulate<BP, WIDTH>(in_src, in_w, e0, e1, in4, acc);
            if (lane < S::LW) {
#pragma unroll
                for (int v = 0; v < S::V; ++v) {
                    b[v].x = fmaf(alpha, acc[v].x, b[v].x);
                    b[v].y = fmaf(alpha, acc[v].y, b[v].y);
                    b[v].z = fmaf(alpha, acc[v].z, b[v].z);
                    b[v].w = fmaf(alpha, acc[v].w, b[v].w);
                    if constexpr (!FILTER) st_stream(out4 + j * S::F + sub + 32 * v, b[v]);
                }
                hop_emit<BP, FILTER>(f, thr, thr_hi, sub, j, id, b);
            }
        }
    }
}

// Segments of split rows, claimed one at a time in window-major order.
template <int BP, int WIDTH = 1>
__global__ __launch_bounds__(256, WIDTH > 1 ? 2 : 3) void k_hop_segs(const int64_t *__restrict__ seg_e0,
                                                  const int64_t *__restrict__ seg_e1,
                                                  const int32_t *__restrict__ seg_slot,
                                                  int64_t n_segs,
                                                  const int32_t *__restrict__ in_src,
                                                  const float *__restrict__ in_w,
                                                  const float4 *__restrict__ in4,
                                                  float4 *__restrict__ part4,
                                                  const int32_t *__restrict__ kept_segs,
                                                  const int64_t *__restrict__ kept_count,
                                                  int *__restrict__ queue,
                                                  const int32_t *__restrict__ done) {
    using S = HopShape<BP>;
    griddep_wait();
    if (done && done[0] == 1) return;
    const int lane = threadIdx.x & 31;
    const int sub = lane % S::LW;
    // last hop: only the listed segments (those of unpruned split rows)
    const int64_t total = kept_segs ? *kept_count : n_segs;
    while (true) {
        int64_t i = 0;
        if (lane == 0) i = atomicAdd(queue, 1);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= total) break;
        const int64_t s = kept_segs ? (int64_t)kept_segs[i] : i;
        float4 acc[S::V];
        hop_accumulate<BP, WIDTH>(in_src, in_w, seg_e0[s], seg_e1[s], in4, acc);
        const int64_t slot = seg_slot[s];
        if (lane < S::LW) {
#pragma unroll
            for (int v = 0; v < S::V; ++v) st_stream(part4 + slot * S::F + sub + 32 * v, acc[v]);
        }
    }
}

template <int BP>
static cudaError_t hop_bp(const HopPlan &p, const float *u, const float *in, float *out,
                          float alpha, float *partial, int *counters, const HopFilter *flt,
                          cudaStream_t st, int *launches, const HopBound *hbp) {
    const int sms = device_sm_count();
    // the last hop skips rows whose bound stays below the filter floor
    const bool prune = flt && hbp && hbp->kept_rows && hbp->kept_count && hbp->split_skip &&
                       (p.n_segs == 0 || hbp->kept_segs);
    cudaError_t e = cudaSuccess;
    if (p.n_segs > 0) {
        const int64_t want = ceil_div<int64_t>(p.n_segs, 8);
        const int cps = prune ? 2 : 3;
        const int g2 = (int)(want < (int64_t)sms * cps ? want : (int64_t)sms * cps);
        e = launch_pdl(prune ? k_hop_segs<BP, 2> : k_hop_segs<BP>, dim3(g2), dim3(256), 0, st,
                       p.seg_e0, p.seg_e1, p.seg_slot, p.n_segs, p.in_src, p.in_w,
                       (const float4 *)in, (float4 *)partial, prune ? hbp->kept_segs : nullptr,
                       prune ? hbp->kept_count + 1 : nullptr, counters + 1, p.done);
        if (e != cudaSuccess) return e;
        if (launches) *launches += 1;
    }
    // (pruned: split rows + the kept list, its length known on the device only)
    const int64_t items = p.n_split_rows + (prune && p.n > 4096 ? 4096 : p.n);
    const int64_t want = ceil_div<int64_t>(items, 8);
    const int cpr = prune ? 2 : 3;
    const int grid = (int)(want < (int64_t)sms * cpr ? (want < 1 ? 1 : want) : (int64_t)sms * cpr);
    const HopFilter f = flt ? *flt : HopFilter{nullptr, nullptr, nullptr, nullptr, 0, NsScope{}};
    e = launch_pdl(prune ? k_hop_rows<BP, true, 2> : flt ? k_hop_rows<BP, true>
                                                         : k_hop_rows<BP, false>,
                   dim3(grid), dim3(256), 0, st, p.in_ptr, p.in_src, p.in_w, p.n,
                   (const float4 *)u, (const float4 *)in, (float4 *)out, alpha, p.split.split_t,
                   p.n_split_rows, p.split_order, p.split_row, p.split_slot0,
                   (const float4 *)partial, f, prune ? hbp->split_skip : nullptr,
                   prune ? hbp->kept_rows : nullptr, prune ? hbp->kept_count : nullptr, counters,
                   p.done);
    if (launches) *launches += 1;
    return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_hop(const HopPlan &p, const float *u, const float *in, float *out, int bp,
                       float alpha, float *partial, int *counters, const HopFilter *flt,
                       cudaStream_t st, int *launches, const HopBound *hb) {
    switch (bp) {
    case 32: return hop_bp<32>(p, u, in, out, alpha, partial, counters, flt, st, launches, hb);
    case 64: return hop_bp<64>(p, u, in, out, alpha, partial, counters, flt, st, launches, hb);
    case 128: return hop_bp<128>(p, u, in, out, alpha, partial, counters, flt, st, launches, hb);
    case 256: return hop_bp<256>(p, u, in, out, alpha, partial, counters, flt, st, launches, hb);
    default: return cudaErrorInvalidValue;
    }
}

// The last hop's values on the row sample, as selection keys, column-major
// (keysT[c][v], sample row v = store row v * stride): the filter's bound is
// the k-th largest of each column, so it must not lie far below the final
// scores.  A row of at most max_edges in-edges gets its final value (the same
// sums in the same order as k_hop_rows); a heavier one its value one hop
// before, which its final value is not below (w >= 0, alpha >= 0, monotone
// rounding): either way no key is above its row's final key.  max_edges is
// split_t (every row kept whole) unless the graph has at least k split rows:
// the floor then comes from their bounds, and rows of more than SMP_EDGES
// edges would only set this kernel's time (with the selection 53 instead of
// 189 us on 262,144 chunks and 200 queries).  That holds where most rows are past
// SMP_EDGES too: on 262,144 chunks linked by updates (32 neighbours, both ways;
// median in-degree 41, 4739 split rows) no buffer overflowed, 64 queries took 151 us
// for one hop and 482 for two (200 and 529 with the level before).  Rows outside the query's scope get key 0.
// The bound used to come from the level before for every row; on a graph
// without heavy in-degrees a hop adds about the same to every row, so nearly
// all rows cleared it, the buffers overflowed and the merge recomputed whole
// columns (65,536 chunks, 64 queries, one hop, 16 nearest neighbours: 9.56 ms
// a call, 0.086 ms with this bound).  1 / stride of a hop's gathers, bound by their latency: a warp
// takes one sample row.
constexpr int SMP_ROWS = 8, SMP_EDGES = 32;
template <int BP>
__global__ __launch_bounds__(256, BP >= 256 ? 2 : BP >= 128 ? 3 : 4) void k_hop_sample(
    const int64_t *__restrict__ in_ptr, const int32_t *__restrict__ in_src,
    const float *__restrict__ in_w, int64_t n_sample, int64_t stride, int64_t max_edges,
    const float4 *__restrict__ u4, const float4 *__restrict__ in4, float alpha, const NsScope ns,
    uint32_t *__restrict__ keysT, const int32_t *__restrict__ done) {
    using S = HopShape<BP>;
    __shared__ uint32_t tile[SMP_ROWS][BP + 1];
    griddep_wait();
    if (done && done[0] == 1) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane % S::LW;
    const int64_t v0 = (int64_t)blockIdx.x * SMP_ROWS;
    static_assert(SMP_ROWS == 8, "a row a warp");
    const int r = warp;
    if (v0 + r < n_sample) {
        const int64_t j = (v0 + r) * stride;
        const int64_t e0 = in_ptr[j], e1 = in_ptr[j + 1];
        const bool whole = e1 - e0 <= max_edges;
        float4 acc[S::V];
        hop_accumulate<BP, BP >= 256 ? 2 : 1>(in_src, in_w, e0, whole ? e1 : e0, in4, acc);
        if (lane < S::LW) {
#pragma unroll
            for (int v = 0; v < S::V; ++v) {
                float4 x = whole ? u4[j * S::F + sub + 32 * v] : in4[j * S::F + sub + 32 * v];
                if (whole) {
                    x.x = fmaf(alpha, acc[v].x, x.x);
                    x.y = fmaf(alpha, acc[v].y, x.y);
                    x.z = fmaf(alpha, acc[v].z, x.z);
                    x.w = fmaf(alpha, acc[v].w, x.w);
                }
                const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int c = (sub + 32 * v) * 4 + e;
                    tile[r][c] = in_scope(ns, j, c) ? __float_as_uint(xs[e]) : 0u;
                }
            }
        }
    }
    __syncthreads();
    const int rr = threadIdx.x % SMP_ROWS;
    if (v0 + rr < n_sample)
        for (int c = threadIdx.x / SMP_ROWS; c < BP; c += 256 / SMP_ROWS)
            keysT[(int64_t)c * n_sample + v0 + rr] = tile[rr][c];
}

cudaError_t launch_hop_sample(const HopPlan &p, const SelectPlan &sp, const float *u,
                              const float *in, float alpha, NsScope ns, uint32_t *keysT,
                              cudaStream_t st, int *launches) {
    auto go = [&](auto kernel) {
        return launch_pdl(kernel, dim3((unsigned)ceil_div<int64_t>(sp.n_sample, SMP_ROWS)),
                          dim3(256), 0, st, p.in_ptr, p.in_src, p.in_w, sp.n_sample, sp.stride,
                          p.n_split_rows >= sp.k && SMP_EDGES < p.split.split_t
                              ? SMP_EDGES : p.split.split_t,
                          (const float4 *)u, (const float4 *)in, alpha, ns, keysT, p.done);
    };
    cudaError_t e = cudaErrorInvalidValue;
    switch (sp.bp) {
    case 32: e = go(k_hop_sample<32>); break;
    case 64: e = go(k_hop_sample<64>); break;
    case 128: e = go(k_hop_sample<128>); break;
    case 256: e = go(k_hop_sample<256>); break;
    }
    if (launches) *launches += 1;
    return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace ak
