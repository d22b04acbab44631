// rs_scan_sort.cu -- device-wide exclusive scan and stable LSD radix sort.
//
// Scan: one launch.  Up to SCAN_SMALL elements one block loops over them;
// above, tiles of SCAN_TILE elements in one pass: each tile publishes its sum,
// looks back over its predecessors' (rs_lookback) and publishes its prefix
// (decoupled look-back: Merrill & Garland 2016; per digit in a radix sort:
// Adinets & Merrill 2022).
// Sort: 8-bit digits.  Up to SORT_SMALL keys one block does all passes in
// shared memory.  Above, one launch counts the digits of every pass, and each
// pass is one launch over tiles of 4096 keys that finds each digit's place by
// looking back, so a pass reads and writes the data once.
#include <algorithm>
#include <cstdlib>

#include "rs_internal.cuh"

namespace {

// tries for a predecessor's word in a look-back (-1 by the injected fault
// wait_<tag>: as if no predecessor ever came)
int wait_limit(const char *tag)
{
    if (!getenv("RS_FAULT")) return RS_SPIN_LIMIT;
    return rs_fault((std::string("wait_") + tag).c_str()) ? -1 : RS_SPIN_LIMIT;
}

constexpr int SCAN_THREADS = 512;
constexpr int SCAN_ITEMS = 8;
constexpr int64_t SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;
constexpr int64_t SCAN_SMALL = 4 * SCAN_TILE;  // one block: 8 us; two launches with the look-back: 9

template <typename T>
__device__ __forceinline__ void scan_load(const T *data, int64_t base, int64_t n, T (&v)[SCAN_ITEMS], T &s)
{
    s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        v[j] = (base + j < n) ? data[base + j] : T(0);
        s += v[j];
    }
}

template <typename T>
__device__ __forceinline__ void scan_store(T *data, int64_t base, int64_t n, const T (&v)[SCAN_ITEMS], T run)
{
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        if (base + j < n) data[base + j] = run;
        run += v[j];
    }
}

template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_small(T *data, int64_t n, T *total)
{
    T carry = 0;
    for (int64_t t0 = 0; t0 < n; t0 += SCAN_TILE) {
        const int64_t base = t0 + (int64_t)threadIdx.x * SCAN_ITEMS;
        T v[SCAN_ITEMS], s, tot;
        scan_load(data, base, n, v, s);
        const T run = rs_block_scan<SCAN_THREADS>(s, tot);
        scan_store(data, base, n, v, (T)(carry + run));
        carry += tot;
    }
    if (total && threadIdx.x == 0) *total = carry;
}

template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_lookback(T *data, int64_t n, T *total, RsLookback lb,
                                                                 rs_dev_status *st)
{
    const int64_t tile = rs_next_tile(lb);
    const int64_t base = tile * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    T v[SCAN_ITEMS], s, tot;
    scan_load(data, base, n, v, s);
    const T run = rs_block_scan<SCAN_THREADS>(s, tot);
    const T before = (T)rs_lookback(lb, tile, (unsigned long long)tot, st);
    scan_store(data, base, n, v, (T)(before + run));
    if (total && threadIdx.x == 0 && (tile + 1) * SCAN_TILE >= n) *total = before + tot;
}

template <typename T>
rs_status scan_top(rs_ctx *ctx, T *data, int64_t n, T *total, const char *tag)
{
    if (n <= 0) {
        if (total) RS_CUDA(ctx, cudaMemsetAsync(total, 0, sizeof(T), ctx->stream));
        return RS_OK;
    }
    if (n <= SCAN_SMALL) {
        RS_LAUNCH(ctx, "scan_small", k_scan_small<T>, 1, SCAN_THREADS, 0, data, n, total);
        return RS_OK;
    }
    const int64_t tiles = ceil_div(n, SCAN_TILE);
    RsLookback lb;
    RS_TRY(rs_lookback_init(ctx, tiles, &lb, tag));
    RS_LAUNCH(ctx, "scan", k_scan_lookback<T>, tiles, SCAN_THREADS, 0, data, n, total, lb, ctx->d_status);
    return RS_OK;
}

// ---------------------------------------------------------------------------
// radix sort
// ---------------------------------------------------------------------------
constexpr int RADIX_BITS = 8;
constexpr int RADIX = 1 << RADIX_BITS;
// Tiles of 4096 keys: 16 a digit on average, a whole line of 64-bit keys.  A
// pass is bound by instruction issue (200 warp instructions per 32 keys, most
// of them the ranking and the two placements): 0.31 ms for 33M 64-bit keys
// with 32-bit values, 2.6 TB/s; with tiles of 2048 and match.any in place of
// eight ballots 0.34.  Counting, scanning and scattering each pass by itself
// took 0.38, and 12 launches a pass group instead of 2 + passes.
constexpr int SORT_THREADS = 512;
constexpr int SORT_ITEMS = 8;
constexpr int64_t SORT_TILE = SORT_THREADS * SORT_ITEMS;
static_assert(SORT_TILE == RS_SORT_TILE, "tile size shared with the fixed-scratch entry point");
static_assert(SORT_THREADS >= RADIX, "each digit has a thread");
constexpr int HIST_THREADS = 256;
constexpr int SMALL_SORT_THREADS = 1024;
constexpr int64_t SORT_SMALL = SMALL_SORT_THREADS * SORT_ITEMS;

// Stable ranks of a block's keys within their digits, a warp's keys being
// consecutive rows of 32: rank[j] counts the equal digits before row j's key
// in its warp; wcnt (a counter per warp and digit, cleared here) ends with the
// warps' totals.
template <typename K, typename C>
__device__ __forceinline__ void sort_rank(const K (&key)[SORT_ITEMS], int64_t wbase, int64_t n, int shift, C *wcnt,
                                          uint32_t (&rank)[SORT_ITEMS])
{
    const int lane = lane_id();
    const uint32_t lt = (1u << lane) - 1u;
    for (int d = lane; d < RADIX; d += 32) wcnt[d] = 0;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < SORT_ITEMS; j++) {
        const bool ok = wbase + j * 32 + lane < n;
        const uint32_t d = (uint32_t)(key[j] >> shift) & (RADIX - 1);
        uint32_t peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
        for (int b = 0; b < RADIX_BITS; b++) {
            const uint32_t m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
            peers &= ((d >> b) & 1u) ? m : ~m;
        }
        const uint32_t before = ok ? wcnt[d] : 0u;
        __syncwarp();
        if (ok && (peers & lt) == 0) wcnt[d] = (C)(before + __popc(peers));
        __syncwarp();
        rank[j] = before + __popc(peers & lt);
    }
}

// the warps' counts of digit d to their starts within the digit; returns the total
template <int WARPS, typename C>
__device__ __forceinline__ uint32_t sort_warp_starts(C (*wcnt)[RADIX], int d)
{
    uint32_t c[WARPS], tot = 0;
#pragma unroll
    for (int w = 0; w < WARPS; w++) c[w] = wcnt[w][d];
#pragma unroll
    for (int w = 0; w < WARPS; w++) {
        wcnt[w][d] = (C)tot;
        tot += c[w];
    }
    return tot;
}

// digit counts of every pass (rows that share a digit, as the high digits of
// sorted or clustered keys do, add once).  HIST_ROWS keys a thread are in
// flight, and a block takes no more than that many while the blocks fill the
// chip: with a sort tile a block, one load at a time, the latency of 16 loads
// in a row was the time (15 sorts of up to 0.5M keys: 223 -> 123 us).
constexpr int HIST_ROWS = 4;

template <typename K>
__global__ void __launch_bounds__(HIST_THREADS) k_sort_hist(const K *keys, int64_t n, int passes, uint32_t *hist,
                                                            int64_t per_block)
{
    extern __shared__ uint32_t h[];
    for (int d = threadIdx.x; d < passes * RADIX; d += HIST_THREADS) h[d] = 0;
    __syncthreads();
    const int64_t b0 = (int64_t)blockIdx.x * per_block;
    const int64_t b1 = min(n, b0 + per_block);
    for (int64_t r = b0 + (threadIdx.x & ~31); r < b1; r += HIST_ROWS * HIST_THREADS) {
        K k[HIST_ROWS];
#pragma unroll
        for (int i = 0; i < HIST_ROWS; i++) {
            const int64_t at = r + i * HIST_THREADS + lane_id();
            k[i] = at < b1 ? keys[at] : K(0);
        }
#pragma unroll
        for (int i = 0; i < HIST_ROWS; i++) {
            const bool ok = r + i * HIST_THREADS + lane_id() < b1;
            const unsigned in = __ballot_sync(0xffffffffu, ok);
            if (!in) break;
            for (int p = 0; p < passes; p++) {
                const uint32_t d = (uint32_t)(k[i] >> (p * RADIX_BITS)) & (RADIX - 1);
                const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
                if (__all_sync(0xffffffffu, !ok || d == d0)) {
                    if (lane_id() == 0) atomicAdd(&h[p * RADIX + d0], (uint32_t)__popc(in));
                } else if (ok) {
                    atomicAdd(&h[p * RADIX + d], 1u);
                }
            }
        }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < passes * RADIX; d += HIST_THREADS)
        if (h[d]) atomicAdd(&hist[d], h[d]);
}

// One pass over one tile: the tile's keys are placed in shared memory in digit
// order, then written out in that order, so the items of one digit go to
// consecutive global slots (coalesced stores).  A digit's place is the count
// of smaller digits in all keys plus that of its own digit in earlier tiles,
// which thread d looks back for (W: one word per tile and digit, two flag
// bits over the count; LIMIT: tries for a word, -1 as if none ever came -- a
// constant, which as an argument took 7% of a pass).
template <typename K>
struct SortShared {
    K key[SORT_TILE];
    uint32_t val[SORT_TILE];
    uint16_t wcnt[SORT_THREADS / 32][RADIX];
    uint32_t goff[RADIX];    // first global slot of each digit for this tile
    uint32_t lstart[RADIX];  // first tile slot of each digit
    unsigned tile;
};

template <typename K, typename W, int LIMIT>
__global__ void __launch_bounds__(SORT_THREADS, 2) k_sort_pass(const K *kin, K *kout, const uint32_t *vin,
                                                              uint32_t *vout, int64_t n, int shift,
                                                              const uint32_t *hist, W *state, unsigned *next,
                                                              rs_dev_status *st)
{
    constexpr int WARPS = SORT_THREADS / 32, FB = 8 * (int)sizeof(W) - 2;
    constexpr W SUM = (W)1 << FB, PREFIX = (W)2 << FB, MASK = SUM - 1;
    extern __shared__ __align__(16) unsigned char sort_smem[];
    SortShared<K> &S = *reinterpret_cast<SortShared<K> *>(sort_smem);
    if (threadIdx.x == 0) S.tile = atomicAdd(next, 1u);
    __syncthreads();
    const int64_t tile = S.tile, tbase = tile * SORT_TILE;
    const int lane = lane_id(), w = warp_id();
    const int64_t wbase = tbase + (int64_t)w * 32 * SORT_ITEMS;
    K key[SORT_ITEMS];
    uint32_t val[SORT_ITEMS], rank[SORT_ITEMS];
#pragma unroll
    for (int j = 0; j < SORT_ITEMS; j++) {
        const int64_t i = wbase + j * 32 + lane;
        key[j] = i < n ? kin[i] : K(0);
        val[j] = i < n ? vin[i] : 0u;
    }
    sort_rank(key, wbase, n, shift, S.wcnt[w], rank);
    __syncthreads();
    {
        const int d = threadIdx.x;
        volatile W *mine = state + tile * RADIX + d;
        uint32_t tot = 0, all;
        if (d < RADIX) {
            tot = sort_warp_starts<WARPS>(S.wcnt, d);
            *mine = (tile == 0 ? PREFIX : SUM) | (W)tot;
        }
        const uint32_t at = rs_block_scan<SORT_THREADS>(tot, all);
        const uint32_t base = rs_block_scan<SORT_THREADS>(d < RADIX ? hist[d] : 0u, all);
        if (d < RADIX) {
            S.lstart[d] = at;
            // eight predecessors a step, their loads in flight together
            W before = 0;
            bool open = LIMIT >= 0 || tile == 0;
            if (!open) dev_torn(st, 91, tile);
            for (int64_t t = tile - 1; t >= 0 && open; t -= 8) {
                W x[8];
#pragma unroll
                for (int u = 0; u < 8; u++) x[u] = t >= u ? *(const volatile W *)(state + (t - u) * RADIX + d) : PREFIX;
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    if (!open) continue;
                    for (int it = 0; x[u] == 0 && it < LIMIT; it++)
                        x[u] = *(const volatile W *)(state + (t - u) * RADIX + d);
                    if (x[u] == 0) dev_torn(st, 91, tile);
                    before += x[u] & MASK;
                    open = x[u] != 0 && !(x[u] & PREFIX);
                }
            }
            if (tile > 0) *mine = PREFIX | (before + (W)tot);
            S.goff[d] = base + (uint32_t)before;
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < SORT_ITEMS; j++) {
        if (wbase + j * 32 + lane < n) {
            const uint32_t d = (uint32_t)(key[j] >> shift) & (RADIX - 1);
            const uint32_t lp = S.lstart[d] + S.wcnt[w][d] + rank[j];
            S.key[lp] = key[j];
            S.val[lp] = val[j];
        }
    }
    __syncthreads();
    const int tn = (int)min((int64_t)SORT_TILE, n - tbase);
    for (int i = threadIdx.x; i < tn; i += SORT_THREADS) {
        const K k = S.key[i];
        const uint32_t d = (uint32_t)(k >> shift) & (RADIX - 1);
        const uint32_t pos = S.goff[d] + ((uint32_t)i - S.lstart[d]);
        if (pos < n) {  // (after a look-back that ran out of time places are wrong: see dev_torn)
            kout[pos] = k;
            vout[pos] = S.val[i];
        }
    }
}

// all passes of a small sort in one block; the result goes to (kout, vout)
template <typename K>
__global__ void __launch_bounds__(SMALL_SORT_THREADS) k_sort_small(const K *kin, K *kout, const uint32_t *vin,
                                                                  uint32_t *vout, int n, int nbits)
{
    constexpr int WARPS = SMALL_SORT_THREADS / 32;
    extern __shared__ __align__(16) unsigned char sort_smem[];
    K *skey = reinterpret_cast<K *>(sort_smem);
    uint32_t *sval = reinterpret_cast<uint32_t *>(skey + SORT_SMALL);
    uint16_t(*wcnt)[RADIX] = reinterpret_cast<uint16_t(*)[RADIX]>(sval + SORT_SMALL);
    uint32_t *lstart = reinterpret_cast<uint32_t *>(wcnt + WARPS);
    const int lane = lane_id(), w = warp_id();
    // the warps share the keys' rows evenly
    const int rows = (n + 31) / 32, per = (rows + WARPS - 1) / WARPS, wbase = 32 * per * w;
    const int wend = min(n, wbase + 32 * per);
    K key[SORT_ITEMS];
    uint32_t val[SORT_ITEMS], rank[SORT_ITEMS];
#pragma unroll
    for (int j = 0; j < SORT_ITEMS; j++) {
        const int i = wbase + j * 32 + lane;
        key[j] = i < wend ? kin[i] : K(0);
        val[j] = i < wend ? vin[i] : 0u;
    }
    for (int shift = 0; shift < nbits; shift += RADIX_BITS) {
        sort_rank(key, wbase, wend, shift, wcnt[w], rank);
        __syncthreads();
        uint32_t tot = 0, all;
        if (threadIdx.x < RADIX) tot = sort_warp_starts<WARPS>(wcnt, threadIdx.x);
        const uint32_t at = rs_block_scan<SMALL_SORT_THREADS>(tot, all);
        if (threadIdx.x < RADIX) lstart[threadIdx.x] = at;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < SORT_ITEMS; j++) {
            if (wbase + j * 32 + lane < wend) {
                const uint32_t d = (uint32_t)(key[j] >> shift) & (RADIX - 1);
                const uint32_t lp = lstart[d] + wcnt[w][d] + rank[j];
                skey[lp] = key[j];
                sval[lp] = val[j];
            }
        }
        __syncthreads();
        const bool last = shift + RADIX_BITS >= nbits;
#pragma unroll
        for (int j = 0; j < SORT_ITEMS; j++) {
            const int i = wbase + j * 32 + lane;
            if (i < wend) {
                key[j] = skey[i];
                val[j] = sval[i];
                if (last) {
                    kout[i] = key[j];
                    vout[i] = val[j];
                }
            }
        }
    }
}

template <typename K, typename W>
rs_status sort_passes(rs_ctx *ctx, K *k0, K *k1, uint32_t *v0, uint32_t *v1, int64_t n, int passes, bool *alt,
                      const char *tag)
{
    const std::string hist_name = std::string(tag) + "_hist", pass_name = std::string(tag) + "_scatter";
    const int64_t tiles = ceil_div(n, SORT_TILE);
    // digit counts and tile counters (a word per 256 counts, 64 apart), then
    // every pass's tile states
    const int64_t head = (int64_t)passes * (RADIX + 64);
    RS_WS(ctx, char, ws, WS_SORT_HIST, 4 * head + (int64_t)sizeof(W) * passes * tiles * RADIX);
    uint32_t *hist = (uint32_t *)ws, *next = hist + passes * RADIX;
    W *state = (W *)(ws + 4 * head);
    RS_CUDA(ctx, cudaMemsetAsync(ws, 0, (size_t)(4 * head + (int64_t)sizeof(W) * passes * tiles * RADIX), ctx->stream));
    const int64_t rows = (int64_t)HIST_ROWS * HIST_THREADS;
    const int64_t per = rows * std::max<int64_t>(1, n / (rows * ctx->num_sms * 8));
    RS_LAUNCH(ctx, hist_name.c_str(), k_sort_hist<K>, ceil_div(n, per), HIST_THREADS, 4 * passes * RADIX,
              (const K *)k0, n, passes, hist, per);
    auto pass = wait_limit(tag) < 0 ? k_sort_pass<K, W, -1> : k_sort_pass<K, W, RS_SPIN_LIMIT>;
    RS_CUDA(ctx, cudaFuncSetAttribute(pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortShared<K>)));
    K *ki = k0, *ko = k1;
    uint32_t *vi = v0, *vo = v1;
    for (int p = 0; p < passes; p++) {
        RS_LAUNCH(ctx, pass_name.c_str(), pass, tiles, SORT_THREADS, (int)sizeof(SortShared<K>), (const K *)ki, ko,
                  (const uint32_t *)vi, vo, n, p * RADIX_BITS, (const uint32_t *)hist + p * RADIX,
                  state + p * tiles * RADIX, next + 64 * p, ctx->d_status);
        std::swap(ki, ko);
        std::swap(vi, vo);
        *alt = !*alt;
    }
    return RS_OK;
}

template <typename K>
rs_status radix_sort(rs_ctx *ctx, K *k0, K *k1, uint32_t *v0, uint32_t *v1, int64_t n, int nbits, bool *alt,
                     const char *tag)
{
    *alt = false;
    if (n <= 1 || nbits <= 0) return RS_OK;
    if (n >= ((int64_t)1 << 32)) return rs_fail(ctx, RS_ERR_TOO_LARGE, "radix sort of 2^32 or more keys");
    if (n <= SORT_SMALL) {
        const size_t smem = SORT_SMALL * (sizeof(K) + 4) + SMALL_SORT_THREADS / 32 * RADIX * 2 + RADIX * 4;
        RS_CUDA(ctx, cudaFuncSetAttribute(k_sort_small<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const std::string name = std::string(tag) + "_small";
        RS_LAUNCH(ctx, name.c_str(), k_sort_small<K>, 1, SMALL_SORT_THREADS, smem, (const K *)k0, k1,
                  (const uint32_t *)v0, v1, (int)n, nbits);
        *alt = true;
        return RS_OK;
    }
    const int passes = (nbits + RADIX_BITS - 1) / RADIX_BITS;
    // 32-bit states hold counts below 2^30 (the injected fault sort64 takes the
    // 64-bit ones at any size, for the tests)
    if (n < ((int64_t)1 << 30) && !rs_fault("sort64")) return sort_passes<K, uint32_t>(ctx, k0, k1, v0, v1, n, passes, alt, tag);
    return sort_passes<K, unsigned long long>(ctx, k0, k1, v0, v1, n, passes, alt, tag);
}

}  // namespace

bool rs_sort_alt(int64_t n, int nbits)
{
    if (n <= 1 || nbits <= 0) return false;
    return n <= SORT_SMALL || ((nbits + RADIX_BITS - 1) / RADIX_BITS & 1);
}

rs_status rs_lookback_init(rs_ctx *ctx, int64_t tiles, RsLookback *lb, const char *tag)
{
    unsigned long long *w = (unsigned long long *)rs_ws(ctx, WS_SCAN_TMP, sizeof(unsigned long long) * (tiles + 1));
    if (!w) return ctx->fixed_ws ? RS_ERR_INTERNAL : RS_ERR_OOM;
    RS_CUDA(ctx, cudaMemsetAsync(w, 0, sizeof(unsigned long long) * (tiles + 1), ctx->stream));
    lb->next = (unsigned *)w;
    lb->state = w + 1;
    lb->limit = wait_limit(tag);
    return RS_OK;
}

rs_status rs_scan_u32(rs_ctx *ctx, uint32_t *data, int64_t n, uint32_t *total, const char *tag)
{
    return scan_top<uint32_t>(ctx, data, n, total, tag);
}

rs_status rs_scan_i64(rs_ctx *ctx, int64_t *data, int64_t n, int64_t *total, const char *tag)
{
    return scan_top<long long>(ctx, (long long *)data, n, (long long *)total, tag);
}

rs_status rs_radix_sort_u64(rs_ctx *ctx, uint64_t *k0, uint64_t *k1, uint32_t *v0, uint32_t *v1, int64_t n,
                            int nbits, bool *alt, const char *tag)
{
    return radix_sort<unsigned long long>(ctx, (unsigned long long *)k0, (unsigned long long *)k1, v0, v1, n,
                                          nbits, alt, tag);
}

rs_status rs_radix_sort_u32(rs_ctx *ctx, uint32_t *k0, uint32_t *k1, uint32_t *v0, uint32_t *v1, int64_t n,
                            int nbits, bool *alt, const char *tag)
{
    return radix_sort<uint32_t>(ctx, k0, k1, v0, v1, n, nbits, alt, tag);
}
