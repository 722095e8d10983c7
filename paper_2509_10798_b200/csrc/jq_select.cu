// Max-pool + exact top-k selection per KV head.  Two kernels share the arithmetic: select_cluster, one thread-block cluster
// of 2 to 16 CTAs per head (choose_plan), and, for calls over 128 heads or more, select_stream further down, one CTA per
// head.  The cluster kernel:
//
//   1. pool: pooled[j] = max of the centred window (edges clipped), turned into an order-preserving 32-bit integer key
//      (float order == unsigned order).  Each CTA owns a contiguous share of the positions and keeps its keys in shared
//      memory (in the workspace for very long prefixes).
//   2. the threshold: 2048 equal bins over the range of the head's keys - not their leading bits, which are the same for
//      most keys of a flat head and would need further rounds over all of them.  The histograms are summed through
//      distributed shared memory, every CTA owning a share of the bins, and every CTA finds the bin of the nkeep-th
//      largest key for itself.  Every CTA lists its keys of that bin, brings the lists of all together and finishes on
//      them - a few dozen by comparison, more by bins of its own: the key tau of the nkeep-th largest element and how many
//      elements equal to tau are kept.  (While the bin holds more than kCandMax keys it is split into 2048 bins by the
//      whole cluster again.)  Max-pooling copies every peak into up to `pool` neighbours, so ties at tau are
//      the normal case: all keys > tau are kept, then the lowest-index keys == tau.
//   3. ordered compaction: kept positions are written in ascending order (CTA rank, warp, iteration and lane order all
//      follow the position order); the list also gives every warp its number of kept keys, so nothing is counted again.
//   4. (fused layer path only) the cluster copies the kept K and V rows of its head, and the window rows behind them.
// Everything is integer arithmetic on bit patterns, hence deterministic and exact.  The kernel is a chain of short phases
// between cluster barriers (four; about 700 cycles each), so what bounds it is latency.  Measured (8 heads, us, against
// leading-bit radix rounds of 11 bits, a counting pass, clusters of 8 and one row in flight per 16 lanes in the copy):
// selection alone 12000 keys 10.6 -> 8.8, 30011 12.1 -> 11.0, 131072 21.3 -> 18.2; with the rows of a layer 131072 keys, budget
// 4096, 73.6 k -> 42.9 k cycles; the windowed layer of 11999 keys (two strided copies before) 46.3 -> 36.9 us.
// Several hundred keys in the threshold's bin (scores whose 24th roots are even; those kernels -> one list in the leading
// CTA, ranked by comparison up to 512 keys -> now): 8 x 30011 12.7 -> 15.5 -> 12.0, 8 x 60000 15.6 -> 24.4 -> 15.4, 127 x
// 60000 70 -> 116 -> 75; 8 x 500 with five different scores 9.7 -> 16.2 -> 8.4.
#include "jq_internal.cuh"
#include "jq_pool.cuh"
#include "jq_debug.cuh"
#include <cooperative_groups.h>
#include <mutex>

namespace cg = cooperative_groups;

namespace jq {
namespace {

constexpr int kClMax = 16;         // most CTAs per cluster (= per KV head)
constexpr int kSelThreads = 512, kSelWarps = kSelThreads / 32;   // two CTAs to an SM (a cluster of 16 then fits for 8 heads at a time)
constexpr int kBins = 2048;
constexpr int kOwnBins = 3 * kBins / 2;   // select_cluster: a CTA's share of the bins in each of three rounds, with two CTAs per cluster
constexpr int kRawTile = 8192;     // most scores staged per pooling step
constexpr int kHalo = 32;          // >= pool radius
constexpr int kKeysSmemMax = 24576; // keys a CTA can keep in shared memory
constexpr size_t kSelTwoPerSm = 110 * 1024;   // shared memory per CTA up to which two CTAs fit on an SM
constexpr double kSelChain = 7.5, kSelChain16 = 10.0, kSelPerKey = 0.0007;   // choose_plan's estimate, us
constexpr int kCandMax = 1024;     // keys of one bin that are finished on a list of them
constexpr int kRankMax = 64;       // of which so many are sent to every CTA and ranked by comparison; more are fetched, and split into bins again
static_assert(kClMax * kRankMax <= kCandMax, "a place for every CTA's list");
// Lists of keys and of their positions, in the place of the staged scores: this CTA's keys of the bin, and those of all CTAs
// (or the short lists that they sent).
constexpr int kOwnKey = 0, kOwnPos = kCandMax, kAllKey = 2 * kCandMax, kAllPos = 3 * kCandMax, kListWords = 4 * kCandMax;
__host__ __device__ constexpr int raw_words(int raw_tile) { return raw_tile + 2 * kHalo > kListWords ? raw_tile + 2 * kHalo : kListWords; }
static_assert(kBins == 4 * kSelThreads, "a thread takes four bins");

// Extents of what the kernel indexes (read by the bounds-checked build only).
struct SelExtents {
    long long scores;     // floats in the scores array (and keys in the global key array)
    long long out_rows;   // rows of the stacked outputs (kept indices, compacted K and V)
    long long src_heads;  // heads in one source buffer of K / V
};

// The window rows that follow every head's kept rows: K, V [Hkv][w] rows (w = 0: none).
struct WindowRows { const uint4 *K, *V; int w; };

struct SelCtl {
    int digit, krem, count;              // find_digit: the bin of the krem-th key, the rank within it, its population
    uint32_t tau;
    int need_eq;
    int cand_count;                      // this CTA's keys of the bin
    int base_gt, base_eq;                // kept-or-tied keys of the CTAs before this one
    uint32_t mn[kClMax], mx[kClMax];     // range of every CTA's keys
    int gt_of[kClMax], eq_of[kClMax], cand_of[kClMax];   // every CTA's keys above the bin (above tau, equal to tau); its keys of the bin
    int warp_gt[kSelWarps], warp_eq[kSelWarps];
    uint32_t wmn[kSelWarps], wmx[kSelWarps];
    int scan[kSelWarps];
};

// Block-wide exclusive scan of one int per thread, any number of whole warps.
__device__ __forceinline__ int cta_excl_scan(int v, int *warp_sums)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
    }
    if (lane == 31) warp_sums[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        const int ws = lane < nw ? warp_sums[lane] : 0;
        int winc = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(0xffffffffu, winc, o);
            if (lane >= o) winc += n;
        }
        if (lane < nw) warp_sums[lane] = winc - ws;
    }
    __syncthreads();
    const int excl = warp_sums[wid] + inc - v;
    __syncthreads();
    return excl;
}

// All threads of a CTA of 512 or 1024: the bin of h[kBins] that holds the krem-th key counted from the top.
template <typename Ctl>
__device__ __forceinline__ void find_digit_cta(const uint32_t *h, int krem, Ctl &ctl)
{
    const int per = kBins / (int)blockDim.x;                  // 4 or 2 bins per thread, descending
    const int hi = kBins - 1 - per * (int)threadIdx.x;
    int tot = 0;
    for (int i = 0; i < per; ++i) tot += (int)h[hi - i];
    int above = cta_excl_scan(tot, ctl.scan);
    for (int i = 0; i < per; ++i) {
        const int c = (int)h[hi - i];
        if (above < krem && krem <= above + c) { ctl.digit = hi - i; ctl.krem = krem - above; ctl.count = c; }
        above += c;
    }
    __syncthreads();
}

// The bin that holds the need-th key counted from the top, from a thread's four bins (those at kBins - 4 - 4 tid) -> ctl: the
// bin, the rank within it, its population.
__device__ __forceinline__ void find_bin(const uint4 v, int need, SelCtl &ctl)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, at = kBins - 4 - 4 * (int)threadIdx.x;
    const int c[4] = {(int)v.w, (int)v.z, (int)v.y, (int)v.x};
    int inc = c[0] + c[1] + c[2] + c[3];
    const int mine = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
    }
    if (lane == 31) ctl.scan[wid] = inc;
    __syncthreads();
    int above = __reduce_add_sync(0xffffffffu, lane < wid ? ctl.scan[lane] : 0) + inc - mine;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (above < need && need <= above + c[i]) { ctl.digit = at + 3 - i; ctl.krem = need - above; ctl.count = c[i]; }
        above += c[i];
    }
    __syncthreads();
}

// Rows [r0, r1) of a head's kept rows (256 bytes each: 16 lanes x 16 bytes), four rows of K and V in flight per 16 lanes.
// kv_in: the head's index within the buffer the rows come from; orow: the head's first row in the outputs.
__device__ __forceinline__ void copy_rows(const int32_t *out, int r0, int r1, int kv_in, long long orow, int L, const uint4 *__restrict__ Kin,
                                          const uint4 *__restrict__ Vin, uint4 *__restrict__ Kout, uint4 *__restrict__ Vout, int src_rows,
                                          const SelExtents &ext JQ_DBG_PARAM)
{
    (void)ext;
    const int lane16 = threadIdx.x & 15, grp = threadIdx.x >> 4, ngrp = blockDim.x >> 4;
    for (int t0 = r0 + 4 * grp; t0 < r1; t0 += 4 * ngrp) {
        int j[4];
        uint4 a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) j[r] = t0 + r < r1 ? min(max(__ldcg(out + t0 + r), 0), L - 1) : 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const size_t src = ((size_t)kv_in * src_rows + j[r]) * 16 + lane16;
            const bool in = t0 + r < r1 && JQ_IN((long long)kv_in * src_rows + j[r], ext.src_heads * src_rows, kDbgSelect, 1);
            a[r] = in ? Kin[src] : make_uint4(0u, 0u, 0u, 0u);
            b[r] = in ? Vin[src] : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const size_t dst = (size_t)(orow + t0 + r) * 16 + lane16;
            if (t0 + r < r1 && JQ_IN(orow + t0 + r, ext.out_rows, kDbgSelect, 2)) { Kout[dst] = a[r]; Vout[dst] = b[r]; }
        }
    }
}

// Window rows [i0, w), every `step`-th group's share, behind the kept rows of head kv (row `row0` of the outputs on).
__device__ __forceinline__ void copy_window(const WindowRows &win, int kv, long long row0, int first, int step, uint4 *__restrict__ Kout,
                                            uint4 *__restrict__ Vout, const SelExtents &ext JQ_DBG_PARAM)
{
    (void)ext;
    const int lane16 = threadIdx.x & 15;
    for (int i = first; i < win.w; i += step) {
        const size_t src = ((size_t)kv * win.w + i) * 16 + lane16, dst = (size_t)(row0 + i) * 16 + lane16;
        if (JQ_IN(row0 + i, ext.out_rows, kDbgSelect, 32)) { Kout[dst] = win.K[src]; Vout[dst] = win.V[src]; }
    }
}

// grid (Hkv * CL), cluster CL, block 512.  With htab (ragged calls) every head has a length, a budget, offsets
// into the scores, the keys and the outputs, and a source buffer of its own; L, nkeep, chunk, keys_in_smem are
// then those of the longest head and only size the shared memory.
__global__ void __launch_bounds__(kSelThreads, 2)
select_cluster(const float *__restrict__ scores, int L, int nkeep, int radius, int32_t *__restrict__ idx,
               float *__restrict__ pooled, uint32_t *__restrict__ gkeys, int chunk, int keys_in_smem, int raw_tile,
               const uint4 *__restrict__ Kin, const uint4 *__restrict__ Vin, uint4 *__restrict__ Kout,
               uint4 *__restrict__ Vout, const HeadRec *__restrict__ htab, const uint4 *const *__restrict__ Ktab,
               const uint4 *const *__restrict__ Vtab, int src_rows, int out_rows, const WindowRows win, const SelExtents ext JQ_DBG_PARAM)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), CL = (int)cluster.num_blocks();
    const int kv = (int)blockIdx.x / CL;
    int kv_in = kv;                                  // the head's index within the buffer its rows come from
    long long soff = (long long)kv * L, orow = (long long)kv * nkeep;   // offsets of the head's scores and of its kept indices
    long long krow = (long long)kv * out_rows;                          // first row of the head in the compacted outputs
    extern __shared__ __align__(16) uint8_t sm[];
    uint32_t *ghist = (uint32_t *)sm;                       // [3][kBins / CL]: the cluster's counts of the bins this CTA owns, one set per round
    uint32_t *hist = ghist + kOwnBins;                      // [kBins]
    float *raw = (float *)(hist + kBins);                   // [raw_tile + 2*kHalo]; when all is pooled,
    uint32_t *const lists = (uint32_t *)raw;                // [kListWords]
    uint32_t *keys_s = (uint32_t *)(raw + raw_words(raw_tile));
    __shared__ SelCtl ctl;

    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int raw_cap = raw_tile + 2 * kHalo, keys_cap = keys_in_smem ? chunk : 0;   // shared-memory extents (those of the launch)
    (void)raw_cap; (void)keys_cap;
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // waited for before the first store to another CTA
    for (int i = tid; i < kOwnBins + kBins; i += kSelThreads) ghist[i] = 0;
    if (tid == 0) ctl.cand_count = 0;
    cudaGridDependencySynchronize();   // everything above ran while the previous kernel of the stream was finishing
    cudaTriggerProgrammaticLaunchCompletion();   // the stream's next kernel may be set up meanwhile; it waits for this one's results
    if (htab) {
        const HeadRec r = htab[kv];
        L = r.L; nkeep = r.nkeep; kv_in = r.kv_in; soff = r.soff; orow = r.ooff; krow = r.ooff; src_rows = L;
        chunk = ((L + CL - 1) / CL + 31) / 32 * 32;   // (keys_in_smem stays the launch's: the longest head decides whether the region exists)
        if (Ktab) { Kin = Ktab[r.unit]; Vin = Vtab[r.unit]; }
    }
    const int j0 = min(rank * chunk, L), j1 = min(j0 + chunk, L), n = j1 - j0;
    const float *s = scores + soff;
    uint32_t *mykeys = keys_in_smem ? keys_s : gkeys + soff + j0;
    int32_t *out = idx + orow;
    if (pooled) pooled += soff;

    // ---- 1. max-pool -> keys, and their range
    // With the keys in shared memory and a window of at most 9, a thread pools four neighbouring positions from three
    // 16-byte reads.
    const bool fast_pool = keys_in_smem && radius <= 4;
    const int left = fast_pool ? 4 : radius;                // staged values before the first position
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    for (int t0 = 0; t0 < n; t0 += raw_tile) {
        const int tile = min(raw_tile, n - t0), staged = fast_pool ? ((tile + 3) & ~3) + 8 : tile + 2 * radius;
        __syncthreads();
        // eight loads in flight per thread: the scores come from L2, one round trip each
        for (int i0 = tid; i0 < staged; i0 += 8 * kSelThreads) {
            float vals[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int i = i0 + q * kSelThreads, j = j0 + t0 - left + i;
                vals[q] = (i < staged && j >= 0 && j < L && JQ_IN(soff + j, ext.scores, kDbgSelect, 3)) ? __ldcg(s + j) : -INFINITY;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (i0 + q * kSelThreads < staged && JQ_IN(i0 + q * kSelThreads, raw_cap, kDbgSelect, 4)) raw[i0 + q * kSelThreads] = vals[q];
        }
        __syncthreads();
        if (fast_pool) {
            const int nquads = (tile + 3) / 4;
            const float4 *raw4 = (const float4 *)raw;
            for (int g4 = tid; g4 < nquads; g4 += kSelThreads) {
                const int nval = min(4, tile - 4 * g4);              // positions of this quad inside the tile
                if (!JQ_IN(4 * (g4 + 2) + 3, raw_cap, kDbgSelect, 6) || !JQ_IN(t0 + 4 * g4 + nval - 1, keys_cap, kDbgSelect, 7)) continue;
                uint32_t key[4];
                float best[4];
                pooled_quad(raw4[g4], raw4[g4 + 1], raw4[g4 + 2], radius, key, best);
                if (nval == 4) *(uint4 *)(mykeys + t0 + 4 * g4) = make_uint4(key[0], key[1], key[2], key[3]);
                else for (int i = 0; i < nval; ++i) mykeys[t0 + 4 * g4 + i] = key[i];
#pragma unroll
                for (int i = 0; i < 4; ++i) if (i < nval) { kmin = min(kmin, key[i]); kmax = max(kmax, key[i]); }
                if (pooled && JQ_IN(soff + j0 + t0 + 4 * g4 + nval - 1, ext.scores, kDbgSelect, 8))
                    for (int i = 0; i < nval; ++i) pooled[j0 + t0 + 4 * g4 + i] = best[i];
            }
            continue;
        }
#pragma unroll 4
        for (int e = tid; e < tile; e += kSelThreads) {
            if (!JQ_IN(e + 2 * radius, raw_cap, kDbgSelect, 10)) continue;
            float best = raw[e];
            for (int u = 1; u <= 2 * radius; ++u) best = fmaxf(best, raw[e + u]);
            const uint32_t k = order_key(best);
            kmin = min(kmin, k); kmax = max(kmax, k);
            if (JQ_IN(keys_in_smem ? t0 + e : soff + j0 + t0 + e, keys_in_smem ? keys_cap : ext.scores, kDbgSelect, 11)) mykeys[t0 + e] = k;
            if (pooled && JQ_IN(soff + j0 + t0 + e, ext.scores, kDbgSelect, 12)) pooled[j0 + t0 + e] = best;
        }
    }
    // Every CTA of the cluster runs from here on: its shared memory may be written.  (The arrival is as old as the kernel:
    // with the pooling in between nobody is waited for.)
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    const int ngrp = kSelThreads / 16;
    const int r0 = (int)((long long)rank * nkeep / CL), r1 = (int)((long long)(rank + 1) * nkeep / CL);   // the rows this CTA copies
    if (nkeep >= L) {   // everything is kept (uniform over the cluster)
        for (int e = tid; e < n; e += kSelThreads) if (JQ_IN(orow + j0 + e, ext.out_rows, kDbgSelect, 13)) out[j0 + e] = j0 + e;
        if (Kin) {
            cluster.sync();
            copy_rows(out, r0, r1, kv_in, krow, L, Kin, Vin, Kout, Vout, src_rows, ext JQ_DBG_ARG_DEV);
            if (win.w) copy_window(win, kv, krow + nkeep, rank * ngrp + (tid >> 4), CL * ngrp, Kout, Vout, ext JQ_DBG_ARG_DEV);
        }
        return;
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) { ctl.wmn[wid] = kmin; ctl.wmx[wid] = kmax; }
    __syncthreads();
    if (wid == 0) {
        kmin = __reduce_min_sync(0xffffffffu, ctl.wmn[lane % kSelWarps]);
        kmax = __reduce_max_sync(0xffffffffu, ctl.wmx[lane % kSelWarps]);
        if (lane < CL) {
            SelCtl *rc = cluster.map_shared_rank(&ctl, lane);
            rc->mn[rank] = kmin; rc->mx[rank] = kmax;
        }
    }
    cluster.sync();

    // ---- 2. the threshold
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int q = 0; q < CL; ++q) { lo = min(lo, ctl.mn[q]); hi = max(hi, ctl.mx[q]); }
    uint32_t lim = hi - lo;                      // the keys in [lo, lo + lim] are the ones the threshold is among,
    int need = nkeep;                            // the need-th largest of them
    bool listed = false;
    const int own = kBins / CL;
    const int per = (n + kSelThreads - 1) / kSelThreads | 1;   // odd: neighbouring threads hit different banks
    for (int round = 0;; ++round) {
        const int sh = lim >> 11 ? 21 - __clz(lim) : 0;            // lim >> sh < 2048
        // A thread takes a run of consecutive keys and adds equal neighbouring bins as one count: the max-pool leaves
        // plateaus, so a few additions per thread replace one per key.
        {
            const int e0 = min(tid * per, n), e1 = min(e0 + per, n);
            uint32_t cur = 0u, cnt = 0u;
            for (int e = e0; e < e1; ++e) {
                if (!JQ_IN(keys_in_smem ? e : soff + j0 + e, keys_in_smem ? keys_cap : ext.scores, kDbgSelect, 14)) continue;
                const uint32_t k = mykeys[e] - lo;
                if (k > lim) continue;
                if (k >> sh != cur) { if (cnt && JQ_IN(cur, kBins, kDbgSelect, 9)) atomicAdd(&hist[cur], cnt); cur = k >> sh; cnt = 0; }
                ++cnt;
            }
            if (cnt && JQ_IN(cur, kBins, kDbgSelect, 9)) atomicAdd(&hist[cur], cnt);
        }
        __syncthreads();
        // CTA q owns the bins [q * own, (q + 1) * own): every CTA adds its counts there (starting at its own, so that they do
        // not all meet at one), then everybody reads the sums back and finds the bin for itself.
        // (At most three rounds: 32 bits of range, 11 bits each.)
        uint32_t *const sums = ghist + round * own;
        {
            const int at = (4 * tid + rank * own) & (kBins - 1);     // this thread's four bins
            const uint4 v = *(const uint4 *)(hist + at);
            *(uint4 *)(hist + at) = make_uint4(0u, 0u, 0u, 0u);     // for the next round
            // (two bins per 64-bit addition: a bin's sum stays below 2^32, so nothing carries from one to the other)
            unsigned long long *const g = (unsigned long long *)(cluster.map_shared_rank(sums, at / own) + at % own);
            if (v.x | v.y) atomicAdd(g, (unsigned long long)v.y << 32 | v.x);
            if (v.z | v.w) atomicAdd(g + 1, (unsigned long long)v.w << 32 | v.z);
        }
        cluster.sync();
        {
            const int at = kBins - 4 - 4 * tid;                      // from the top
            find_bin(*(const uint4 *)(cluster.map_shared_rank(sums, at / own) + at % own), need, ctl);
        }
        lo += (uint32_t)ctl.digit << sh;
        need = ctl.krem;
        lim = (1u << sh) - 1u;
        listed = sh != 0 && ctl.count <= kCandMax;                   // (a bin of one key value needs no list)
        if (listed || sh == 0) break;
    }
    // Warp w owns the contiguous elements [w0, w1).  Keys above the bin (listed) or above / equal to the threshold are
    // counted per warp; the bin's own keys are listed.
    const int nc = listed ? ctl.count : 0;
    const int seg = ((n + kSelWarps - 1) / kSelWarps + 31) / 32 * 32;
    const int w0 = min(wid * seg, n), w1 = min(w0 + seg, n);
    const uint32_t top = lo + lim;
    {
        int cgt = 0, ceq = 0;
        for (int base = w0; base < w1; base += 32) {
            const int e = base + lane;
            const bool in = e < w1 && JQ_IN(keys_in_smem ? e : soff + j0 + e, keys_in_smem ? keys_cap : ext.scores, kDbgSelect, 19);
            const uint32_t k = in ? mykeys[e] : 0u;
            cgt += in && k > top;
            const bool hit = in && k >= lo && k <= top;
            ceq += hit;
            if (!listed) continue;
            const uint32_t votes = __ballot_sync(0xffffffffu, hit);
            if (votes) {
                int at = 0;
                if (lane == 0) at = atomicAdd(&ctl.cand_count, __popc(votes));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(votes & ((1u << lane) - 1u));
                if (hit && JQ_IN(at, kCandMax, kDbgSelect, 15)) { lists[kOwnKey + at] = k; lists[kOwnPos + at] = (uint32_t)(j0 + e); }
            }
        }
        cgt = __reduce_add_sync(0xffffffffu, cgt);
        ceq = __reduce_add_sync(0xffffffffu, ceq);
        if (lane == 0) { ctl.warp_gt[wid] = cgt; ctl.warp_eq[wid] = listed ? 0 : ceq; }
        __syncthreads();
        if (listed && nc <= kRankMax && wid < CL) {                  // warp q sends this CTA's list to CTA q
            uint32_t *to = cluster.map_shared_rank(lists, wid) + rank * kRankMax;
            for (int i = lane; i < ctl.cand_count; i += 32)
                if (JQ_IN(i, kRankMax, kDbgSelect, 34)) { to[kAllKey + i] = lists[kOwnKey + i]; to[kAllPos + i] = lists[kOwnPos + i]; }
        }
        if (wid == 0) {
            const int g = __reduce_add_sync(0xffffffffu, lane < kSelWarps ? ctl.warp_gt[lane] : 0), q = __reduce_add_sync(0xffffffffu, lane < kSelWarps ? ctl.warp_eq[lane] : 0);
            if (lane < CL) {
                SelCtl *rc = cluster.map_shared_rank(&ctl, lane);
                rc->gt_of[rank] = g; rc->eq_of[rank] = q; rc->cand_of[rank] = ctl.cand_count;
            }
        }
        if (tid == 0) { ctl.base_gt = ctl.base_eq = 0; }
        cluster.sync();
    }
    uint32_t tau = lo;
    int need_eq = need;             // how many of the keys == tau are kept (lowest positions first)
    if (listed) {
        // Every CTA brings the lists together for itself, 16 / CL warps each.  (One list in the leading CTA, appended to by all,
        // cost a round trip between the CTAs for every group of 32 keys that had one.)
        const uint32_t *const list = lists + (nc <= kRankMax ? kOwnKey : kAllKey);
        {
            const int q = wid & (CL - 1), have = lane < CL ? ctl.cand_of[lane] : 0;
            const int before = __reduce_add_sync(0xffffffffu, lane < q ? have : 0), mine = __shfl_sync(0xffffffffu, have, q);
            const int i0 = wid / CL * 32 + lane, step = kSelWarps / CL * 32;
            if (nc <= kRankMax) {
                for (int i = i0; i < mine; i += step)
                    if (JQ_IN(before + i, kCandMax, kDbgSelect, 16)) {
                        lists[kOwnKey + before + i] = lists[kAllKey + q * kRankMax + i];
                        lists[kOwnPos + before + i] = lists[kAllPos + q * kRankMax + i];
                    }
            } else {
                const uint32_t *from = cluster.map_shared_rank(lists, q);
#pragma unroll 4
                for (int i = i0; i < mine; i += step)
                    if (JQ_IN(before + i, kCandMax, kDbgSelect, 35)) {
                        lists[kAllKey + before + i] = from[kOwnKey + i];
                        lists[kAllPos + before + i] = from[kOwnPos + i];
                    }
            }
        }
        __syncthreads();
        if (nc <= kRankMax) {
            if (tid < nc) {
                const uint32_t k = list[tid];
                int gt = 0, eq = 0;
#pragma unroll 4
                for (int i = 0; i < nc; ++i) { const uint32_t x = list[i]; gt += x > k; eq += x == k; }
                if (gt < need && need <= gt + eq) { ctl.tau = k; ctl.need_eq = need - gt; }   // (equal keys write the same)
            }
            __syncthreads();
            tau = ctl.tau;
            need_eq = ctl.need_eq;
        } else {
            // at most two rounds of bins over the list (the bin spans 21 bits at most), in this CTA alone
            for (;;) {
                const int sh = lim >> 11 ? 21 - __clz(lim) : 0;
                for (int i = tid; i < nc; i += kSelThreads) {
                    const uint32_t k = list[i] - lo;
                    if (k <= lim && JQ_IN(k >> sh, kBins, kDbgSelect, 33)) atomicAdd(&hist[k >> sh], 1u);
                }
                __syncthreads();
                uint4 *const mine = (uint4 *)(hist + kBins - 4 - 4 * tid);
                const uint4 v = *mine;
                *mine = make_uint4(0u, 0u, 0u, 0u);
                find_bin(v, need, ctl);
                lo += (uint32_t)ctl.digit << sh;
                need = ctl.krem;
                if (sh == 0) break;
                lim = (1u << sh) - 1u;
            }
            tau = lo;
            need_eq = need;
        }
        // the kept and tied keys among them before this CTA's share, and of this CTA's warps
        for (int i = tid; i - lane < nc; i += kSelThreads) {
            const uint32_t k = i < nc ? list[i] : 0u;
            const int at = i < nc ? (int)list[kCandMax + i] : L;
            const uint32_t bg = __ballot_sync(0xffffffffu, at < j0 && k > tau), be = __ballot_sync(0xffffffffu, at < j0 && k == tau);
            if (lane == 0 && bg) atomicAdd(&ctl.base_gt, __popc(bg));
            if (lane == 0 && be) atomicAdd(&ctl.base_eq, __popc(be));
            if (k >= tau && at >= j0 && at < j1) {
                const int w = (at - j0) / seg;
                if (JQ_IN(w, kSelWarps, kDbgSelect, 20)) atomicAdd(k > tau ? &ctl.warp_gt[w] : &ctl.warp_eq[w], 1);
            }
        }
        __syncthreads();
    }
    int gt_before = ctl.base_gt, eq_before = ctl.base_eq;
    for (int q = 0; q < rank; ++q) { gt_before += ctl.gt_of[q]; eq_before += ctl.eq_of[q]; }
    gt_before += __reduce_add_sync(0xffffffffu, lane < wid ? ctl.warp_gt[lane] : 0);
    eq_before += __reduce_add_sync(0xffffffffu, lane < wid ? ctl.warp_eq[lane] : 0);

    // ---- 3. ordered compaction
    const uint32_t lt_mask = (1u << lane) - 1u;
    if (ctl.warp_gt[wid] | ctl.warp_eq[wid])
        for (int base = w0; base < w1; base += 32) {
            const int e = base + lane;
            const bool in = e < w1 && JQ_IN(keys_in_smem ? e : soff + j0 + e, keys_in_smem ? keys_cap : ext.scores, kDbgSelect, 21);
            const uint32_t k = in ? mykeys[e] : 0u;
            const uint32_t bg = __ballot_sync(0xffffffffu, in && k > tau);
            const uint32_t be = __ballot_sync(0xffffffffu, in && k == tau);
            if (!(bg | be)) continue;
            const int g_here = gt_before + __popc(bg & lt_mask), e_here = eq_before + __popc(be & lt_mask);
            if (in) {
                if (k > tau) { if (JQ_IN(g_here + min(e_here, need_eq), nkeep, kDbgSelect, 17)) out[g_here + min(e_here, need_eq)] = j0 + e; }
                else if (k == tau && e_here < need_eq) { if (JQ_IN(g_here + e_here, nkeep, kDbgSelect, 18)) out[g_here + e_here] = j0 + e; }
            }
            gt_before += __popc(bg);
            eq_before += __popc(be);
        }
    // ---- 4. the rows, once every index of the head has been written.  (Without rows the cluster still leaves together: a
    // CTA's list may be being read.)
    cluster.sync();                 // (release and acquire at cluster scope: the readers are in the cluster)
    if (!Kin) return;
    copy_rows(out, r0, r1, kv_in, krow, L, Kin, Vin, Kout, Vout, src_rows, ext JQ_DBG_ARG_DEV);
    if (win.w) copy_window(win, kv, krow + nkeep, rank * ngrp + (tid >> 4), CL * ngrp, Kout, Vout, ext JQ_DBG_ARG_DEV);
}

// ------------------------------------------------------------------ many heads: one CTA per head, no cluster
//
// A call over many heads (the layers of a cache, a ragged batch) has more heads than clusters fit on the GPU, and the
// cluster kernel's time per head is mostly the latency of its barrier-separated phases.  Here a head is one CTA that
// keeps a histogram, a candidate list and a small staging buffer per warp in shared memory, so that several heads are
// resident per SM, and that walks the head's scores three times, pooling on the fly.  Every warp owns a contiguous
// share of the head and takes it 512 positions at a time: four 16-byte asynchronous copies per lane into one of the
// warp's two staging buffers, with one quad of halo on either side, from where a lane pools four neighbouring
// positions while the copies of the next 512 positions are in flight.
//   pass 1  pooled keys -> histogram of the top 11 bits (and the pooled values, when the caller wants them);
//   pass 2  the keys that share the winning digit -> candidate list (key and position), and per warp the number of
//           keys with a larger digit (passes 2 and 3 pool only the quads whose 12 staged scores reach the threshold); rounds 2 and 3 run on the list, and the list then also gives every warp its
//           number of kept keys.  (When the list would not fit, rounds 2 and 3 and the counts are passes of their own.)
//   pass 3  ordered compaction of the kept positions, then the copy of the kept rows.
// Same integer arithmetic as the cluster kernel: the same threshold key and the same ties, hence the same indices.
constexpr int kStrCand = 2048;      // candidates finished in shared memory
constexpr int kStrMaxWarps = 32;
constexpr int kStepQuads = 128;     // quads a warp takes per step
constexpr int kStageQuads = kStepQuads + 2;
constexpr int kStreamMinHeads = 128;   // calls with at least this many heads take this kernel
constexpr int kSparseQuads = 4 * 34;   // (sparse) a step is four tiles of 32 quads, each with a quad of halo on either side

struct StrCtl {
    int scan[kStrMaxWarps + 1];
    int digit, krem, count;         // find_digit_cta: the bin of the krem-th key, the rank within it, its population
    int cand_count;
    int warp_gt[kStrMaxWarps], warp_eq[kStrMaxWarps];
};

// Quad q (positions 4q .. 4q+3) of a head of L scores at s; positions outside [0, L) read as -inf.
// vec: s is 16-byte aligned.
__device__ __forceinline__ float4 load_quad(const float *__restrict__ s, int L, int q, bool vec, long long soff,
                                            const SelExtents &ext JQ_DBG_PARAM)
{
    (void)soff; (void)ext;
    const float ninf = -INFINITY;
    if (q < 0 || 4 * q >= L) return make_float4(ninf, ninf, ninf, ninf);
    if (vec && 4 * q + 4 <= L && JQ_IN(soff + 4 * q + 3, ext.scores, kDbgSelect, 22)) return *(const float4 *)(s + 4 * q);
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = (4 * q + i < L && JQ_IN(soff + 4 * q + i, ext.scores, kDbgSelect, 23)) ? s[4 * q + i] : ninf;
    return make_float4(v[0], v[1], v[2], v[3]);
}

// The warp requests quads [base - 1, base + 129) of the head into one of its two buffers: 16-byte asynchronous copies
// for the quads that lie inside the head (and are aligned), plain stores of -inf-padded values for the others.
__device__ __forceinline__ void stage_issue(float4 *dst, const float *__restrict__ s, int L, int base, bool vec, long long soff,
                                            const SelExtents &ext JQ_DBG_PARAM)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < 5; ++u) {
        if (u == 4 && lane >= 2) break;
        const int q = u < 4 ? base + 32 * u + lane : (lane == 0 ? base - 1 : base + kStepQuads);
        float4 *d = dst + (u < 4 ? 1 + 32 * u + lane : (lane == 0 ? 0 : kStageQuads - 1));
        if (vec && q >= 0 && 4 * q + 4 <= L && JQ_IN(soff + 4 * q + 3, ext.scores, kDbgSelect, 22))
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(d)), "l"(s + 4 * q) : "memory");
        else
            *d = load_quad(s, L, q, vec, soff, ext JQ_DBG_ARG_DEV);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// One quad of a tile into the warp's buffer, if its block is scored; else zeros, as what is not scored counts.
__device__ __forceinline__ void stage_quad(float4 *d, const float *__restrict__ s, int L, int q, bool scored, bool vec, long long soff,
                                           const SelExtents &ext JQ_DBG_PARAM)
{
    if (!scored)
        *d = make_float4(0.f, 0.f, 0.f, 0.f);
    else if (vec && 4 * q + 4 <= L && JQ_IN(soff + 4 * q + 3, ext.scores, kDbgSelect, 22))
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(d)), "l"(s + 4 * q) : "memory");
    else
        *d = load_quad(s, L, q, vec, soff, ext JQ_DBG_ARG_DEV);
}

// The staged quads of the step at `base` of the warp's walk over [qa, qb), 128 quads per step: waits for the step's
// copies and has the next step's under way (two buffers per warp), so that a step's reads from memory overlap the
// pooling of the step before.  Every lane of the warp calls it once per step, in order.
__device__ __forceinline__ const float4 *stage_step(float4 *bufs, const float *__restrict__ s, int L, int base, int qa, int qb, bool vec,
                                                    long long soff, const SelExtents &ext JQ_DBG_PARAM)
{
    const int step = (base - qa) / kStepQuads;
    float4 *cur = bufs + (step & 1) * kStageQuads, *nxt = bufs + ((step + 1) & 1) * kStageQuads;
    if (step == 0) {
        __syncwarp();                                        // the reads of an earlier pass are done
        stage_issue(cur, s, L, base, vec, soff, ext JQ_DBG_ARG_DEV);
    }
    __syncwarp();                                            // the previous step's reads of the other buffer are done
    if (base + kStepQuads < qb) {
        stage_issue(nxt, s, L, base + kStepQuads, vec, soff, ext JQ_DBG_ARG_DEV);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    return cur;
}

// Order key of the largest of the 12 staged scores around quad `at`: an upper bound of the quad's four pooled keys
// (every window lies inside those 12), so a quad whose bound is below a threshold holds nothing at or above it and
// the passes that only look for such keys skip its pooling.
__device__ __forceinline__ uint32_t quad_bound_key(const float4 *buf, int at)
{
    const float4 a = buf[at], b = buf[at + 1], c = buf[at + 2];
    const float m = max3f(max3f(a.x, a.y, a.z), max3f(a.w, b.x, b.y), max3f(max3f(b.z, b.w, c.x), max3f(c.y, c.z, c.w), -INFINITY));
    return order_key(m);
}

// Adds the digits of a thread's (up to) four neighbouring keys to the histogram: runs of equal digits as one count (the
// max-pool leaves plateaus); digit 0xffffffff marks a key that does not take part.
__device__ __forceinline__ void hist_add_runs(uint32_t *hist, const uint32_t (&digit)[4], int nval JQ_DBG_PARAM)
{
    uint32_t cur = 0xffffffffu, cnt = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i < nval) {
            if (digit[i] != cur) {
                if (cnt && cur != 0xffffffffu && JQ_IN(cur, kBins, kDbgSelect, 24)) atomicAdd(&hist[cur], cnt);
                cur = digit[i]; cnt = 0;
            }
            ++cnt;
        }
    }
    if (cnt && cur != 0xffffffffu && JQ_IN(cur, kBins, kDbgSelect, 24)) atomicAdd(&hist[cur], cnt);
}

// grid (Hkv), block kThreads = 512 (two CTAs to an SM) or 1024 (one); dynamic shared memory: two staging buffers of
// kStageQuads float4 per warp.  Arguments as for select_cluster.
__host__ __device__ constexpr int stream_ctas_per_sm(int threads) { return threads == 512 ? 2 : 1; }
template <int kThreads, bool kSparse>
__global__ void __launch_bounds__(kThreads, stream_ctas_per_sm(kThreads))
select_stream(const float *__restrict__ scores, int L, int nkeep, int radius, int32_t *__restrict__ idx,
              float *__restrict__ pooled, const uint4 *__restrict__ Kin, const uint4 *__restrict__ Vin,
              uint4 *__restrict__ Kout, uint4 *__restrict__ Vout, const HeadRec *__restrict__ htab,
              const uint4 *const *__restrict__ Ktab, const uint4 *const *__restrict__ Vtab, int src_rows, int out_rows,
              const WindowRows win, const ScoredTiles scored,
              const SelExtents ext JQ_DBG_PARAM)
{
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ uint32_t hist[kBins];
    __shared__ uint32_t cand_key[kStrCand];
    __shared__ int cand_pos[kStrCand];
    __shared__ StrCtl ctl;
    constexpr int T = kThreads, nw = T / 32;
    const int kv = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int kBufQuads = kSparse ? kSparseQuads : kStageQuads;
    float4 *buf = (float4 *)sm + wid * 2 * kBufQuads;     // the warp's two staging buffers
    uint32_t *const tiles = (uint32_t *)((float4 *)sm + nw * 2 * kBufQuads);   // (sparse) every warp's tiles that take part
    int kv_in = kv;
    long long soff = (long long)kv * L, orow = (long long)kv * nkeep, krow = (long long)kv * out_rows;
    cudaGridDependencySynchronize();   // everything above ran while the previous kernel of the stream was finishing
    if (htab) {
        const HeadRec r = htab[kv];
        L = r.L; nkeep = r.nkeep; kv_in = r.kv_in; soff = r.soff; orow = r.ooff; krow = r.ooff; src_rows = L;
        if (Ktab) { Kin = Ktab[r.unit]; Vin = Vtab[r.unit]; }
    }
    if (nkeep > L) nkeep = L;
    const float *s = scores + soff;
    int32_t *out = idx + orow;
    if (pooled) pooled += soff;
    const bool vec = (((size_t)s) & 15) == 0;
    const int nq = (L + 3) / 4;
    // warp w owns the contiguous quads [qa, qb); every warp makes the same number of steps
    const int segq = kSparse ? 32 * (((L + 127) / 128 + nw - 1) / nw) : (nq + nw - 1) / nw;
    const int qa = min(wid * segq, nq), qb = min(qa + segq, nq);
    int n_tiles = 0;                                           // (sparse) the warp's tiles that take part
    if (kSparse) {
        // a tile's entry: its number, its scored blocks, whether the block before it and the one behind it are scored
        const long long tile0 = scored.tbase ? scored.tbase[kv] : (long long)kv * scored.tph;
        const uint8_t *const from = scored.bits + tile0;
        auto bits_of = [&](int t) { return JQ_IN(tile0 + t, scored.tiles, kDbgSelect, 37) ? (uint32_t)__ldcg(from + t) : 0u; };
        const int nt = (L + 127) / 128, ta = min(wid * (segq >> 5), nt), tb = min(ta + (segq >> 5), nt);
        for (int t0 = ta; t0 < tb; t0 += 32) {
            const int t = t0 + lane;
            const uint32_t b = t < tb ? bits_of(t) : 0u;
            uint32_t before = __shfl_up_sync(0xffffffffu, b, 1) >> 7, behind = __shfl_down_sync(0xffffffffu, b, 1) & 1u;
            if (lane == 0) before = t > 0 ? bits_of(t - 1) >> 7 : 0u;
            if ((lane == 31 || t + 1 >= tb) && t < tb) behind = t + 1 < nt ? bits_of(t + 1) & 1u : 0u;
            const bool on = t < tb && (b | before | behind) != 0u;
            const uint32_t m = __ballot_sync(0xffffffffu, on);
            const int at = ta + n_tiles + __popc(m & ((1u << lane) - 1u));
            if (on && JQ_IN(at, scored.max_tiles, kDbgSelect, 36)) tiles[at] = (uint32_t)t | b << 16 | before << 24 | behind << 25;
            n_tiles += __popc(m);
        }
        __syncwarp();
    }
    // One walk over the warp's share in order of position: f(q, nval, st) for 32 quads at a time, of which lane l has quad q with
    // nval positions that take part, staged as st[l + 1] between its neighbours.
    auto walk = [&](auto f) {
        if constexpr (kSparse) {
            const uint32_t *const mine = tiles + min(wid * (segq >> 5), (L + 127) / 128);
            __syncwarp();                                      // the reads of an earlier walk are done
            auto request = [&](int i, float4 *to) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (i + u >= n_tiles) break;
                    const uint32_t e = mine[i + u], t = e & 0xffffu;
                    float4 *const d = to + 34 * u + 1;
                    stage_quad(d + lane, s, L, (int)(32 * t) + lane, e >> (16 + (lane >> 2)) & 1u, vec, soff, ext JQ_DBG_ARG_DEV);
                    if (lane < 2) stage_quad(d + (lane ? 32 : -1), s, L, (int)(32 * t) + (lane ? 32 : -1), e >> (24 + lane) & 1u, vec, soff, ext JQ_DBG_ARG_DEV);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            request(0, buf);
#pragma unroll 1
            for (int i = 0; i < n_tiles; i += 4) {
                const float4 *const cur = buf + (i >> 2 & 1) * kBufQuads;
                request(i + 4, buf + (~i >> 2 & 1) * kBufQuads);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
                __syncwarp();
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (i + u >= n_tiles) break;
                    const uint32_t e = mine[i + u], b = e >> 16 & 0xffu, act = b | b << 1 | b >> 1 | (e >> 24 & 1u) | (e >> 25 & 1u) << 7;
                    const int q = (int)(32 * (e & 0xffffu)) + lane;
                    f(q, act >> (lane >> 2) & 1u ? max(0, min(4, L - 4 * q)) : 0, cur + 34 * u);
                }
                __syncwarp();
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        } else {
            for (int base = qa; base < qb; base += kStepQuads) {
                const float4 *bf = stage_step(buf, s, L, base, qa, qb, vec, soff, ext JQ_DBG_ARG_DEV);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int q = base + 32 * u + lane;
                    f(q, q < qb ? min(4, L - 4 * q) : 0, bf + 32 * u);
                }
            }
        }
    };

    // ---- pass 1: histogram of the top 11 bits of the pooled keys
    for (int i = tid; i < kBins; i += T) hist[i] = 0;
    if (tid == 0) ctl.cand_count = 0;
    __syncthreads();
    walk([&](int q, int nval, const float4 *bf) {
        uint32_t key[4];
        float best[4];
        pooled_quad(bf[lane], bf[lane + 1], bf[lane + 2], radius, key, best);
        if (pooled && nval && JQ_IN(soff + 4 * q + nval - 1, ext.scores, kDbgSelect, 25))
            for (int i = 0; i < nval; ++i) pooled[4 * q + i] = best[i];
        // one addition per warp when all its positions share the digit (the usual case: 128 neighbouring
        // positions of similar size), else runs of equal digits per thread
        const uint32_t d0 = key[0] >> 21;
        bool same = true;
        for (int i = 1; i < 4; ++i) if (i < nval && (key[i] >> 21) != d0) same = false;
        const uint32_t lead = __shfl_sync(0xffffffffu, d0, 0);
        if (__all_sync(0xffffffffu, nval == 0 || (same && d0 == lead))) {
            const int tot = __reduce_add_sync(0xffffffffu, nval);
            if (lane == 0 && tot && JQ_IN(lead, kBins, kDbgSelect, 24)) atomicAdd(&hist[lead], (uint32_t)tot);
        } else {
            const uint32_t dg[4] = {key[0] >> 21, key[1] >> 21, key[2] >> 21, key[3] >> 21};
            hist_add_runs(hist, dg, nval JQ_DBG_ARG_DEV);
        }
    });
    __syncthreads();
    if (nkeep >= L) {                                          // everything is kept
        for (int e = tid; e < L; e += T) if (JQ_IN(orow + e, ext.out_rows, kDbgSelect, 26)) out[e] = e;
    } else {
        // ---- the threshold key tau and how many keys equal to it are kept
        find_digit_cta(hist, nkeep, ctl);
        uint32_t pre = (uint32_t)ctl.digit;
        int krem = ctl.krem;
        const bool listed = ctl.count <= kStrCand;
        if (lane == 0) { ctl.warp_gt[wid] = 0; ctl.warp_eq[wid] = 0; }
        __syncthreads();
        if (listed) {
            // pass 2: the keys with the winning first digit, with their positions; the warp's keys above that digit
            int hi_cnt = 0;
            walk([&](int q, int nval, const float4 *bf) {
                if (nval == 0 || (quad_bound_key(bf, lane) >> 21) < pre) return;
                uint32_t key[4];
                float best[4];
                pooled_quad(bf[lane], bf[lane + 1], bf[lane + 2], radius, key, best);
                int nhit = 0;
                for (int i = 0; i < 4; ++i) if (i < nval) { nhit += (key[i] >> 21) == pre; hi_cnt += (key[i] >> 21) > pre; }
                if (nhit) {
                    int at = atomicAdd(&ctl.cand_count, nhit);
                    for (int i = 0; i < 4; ++i)
                        if (i < nval && (key[i] >> 21) == pre) {
                            if (JQ_IN(at, kStrCand, kDbgSelect, 27)) { cand_key[at] = key[i]; cand_pos[at] = 4 * q + i; }
                            ++at;
                        }
                }
            });
            hi_cnt = __reduce_add_sync(0xffffffffu, hi_cnt);
            if (lane == 0) ctl.warp_gt[wid] = hi_cnt;
            __syncthreads();
        }
        const int nc = listed ? ctl.cand_count : 0;
        for (int r2 = 1; r2 < 3; ++r2) {
            const int sh = (r2 == 1) ? 10 : 0, wd = (r2 == 2) ? 10 : 11;
            const uint32_t mask = (1u << wd) - 1u;
            for (int i = tid; i < kBins; i += T) hist[i] = 0;
            __syncthreads();
            if (listed) {
                for (int e = tid; e < nc; e += T) {
                    const uint32_t k = cand_key[e];
                    if ((k >> (sh + wd)) == pre && JQ_IN((k >> sh) & mask, kBins, kDbgSelect, 24)) atomicAdd(&hist[(k >> sh) & mask], 1u);
                }
            } else {
                walk([&](int q, int nval, const float4 *bf) {
                    if (nval == 0 || (quad_bound_key(bf, lane) >> (sh + wd)) < pre) return;
                    uint32_t key[4], dg[4];
                    float best[4];
                    pooled_quad(bf[lane], bf[lane + 1], bf[lane + 2], radius, key, best);
                    for (int i = 0; i < 4; ++i) dg[i] = (key[i] >> (sh + wd)) == pre ? ((key[i] >> sh) & mask) : 0xffffffffu;
                    hist_add_runs(hist, dg, nval JQ_DBG_ARG_DEV);
                });
            }
            __syncthreads();
            find_digit_cta(hist, krem, ctl);
            pre = (pre << wd) | (uint32_t)ctl.digit;
            krem = ctl.krem;
            __syncthreads();
        }
        const uint32_t tau = pre;
        const int need_eq = krem;       // how many of the keys == tau are kept (lowest positions first)

        // ---- kept keys per warp: from the list, or by a pass of its own
        if (listed) {
            for (int e = tid; e < nc; e += T) {
                const uint32_t k = cand_key[e];
                const int w = min((cand_pos[e] >> 2) / segq, nw - 1);
                if (k > tau) atomicAdd(&ctl.warp_gt[w], 1);
                else if (k == tau) atomicAdd(&ctl.warp_eq[w], 1);
            }
        } else {
            int cgt = 0, ceq = 0;
            walk([&](int q, int nval, const float4 *bf) {
                if (nval == 0 || quad_bound_key(bf, lane) < tau) return;
                uint32_t key[4];
                float best[4];
                pooled_quad(bf[lane], bf[lane + 1], bf[lane + 2], radius, key, best);
                for (int i = 0; i < 4; ++i) if (i < nval) { cgt += key[i] > tau; ceq += key[i] == tau; }
            });
            cgt = __reduce_add_sync(0xffffffffu, cgt);
            ceq = __reduce_add_sync(0xffffffffu, ceq);
            if (lane == 0) { ctl.warp_gt[wid] = cgt; ctl.warp_eq[wid] = ceq; }
        }
        __syncthreads();
        int gt_before = 0, eq_before = 0;
        for (int w = 0; w < wid; ++w) { gt_before += ctl.warp_gt[w]; eq_before += ctl.warp_eq[w]; }

        // ---- pass 3: ordered compaction (position order = warp, step, quad, position within the quad)
        walk([&](int q, int nval, const float4 *bf) {
            const bool may = nval != 0 && quad_bound_key(bf, lane) >= tau;
            if (!__any_sync(0xffffffffu, may)) return;         // nothing of these 128 quads is at or above tau
            uint32_t key[4] = {0u, 0u, 0u, 0u};
            float best[4];
            if (may) pooled_quad(bf[lane], bf[lane + 1], bf[lane + 2], radius, key, best);
            int g = 0, e = 0;
            for (int i = 0; i < 4; ++i) if (may && i < nval) { g += key[i] > tau; e += key[i] == tau; }
            const int mine = g | (e << 16);
            int inc = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += n;
            }
            const int total = __shfl_sync(0xffffffffu, inc, 31);
            int g_here = gt_before + ((inc - mine) & 0xffff), e_here = eq_before + ((inc - mine) >> 16);
            for (int i = 0; i < 4; ++i) {
                if (!may || i >= nval) continue;
                if (key[i] > tau) {
                    if (JQ_IN(g_here + min(e_here, need_eq), nkeep, kDbgSelect, 28)) out[g_here + min(e_here, need_eq)] = 4 * q + i;
                    ++g_here;
                } else if (key[i] == tau) {
                    if (e_here < need_eq && JQ_IN(g_here + e_here, nkeep, kDbgSelect, 29)) out[g_here + e_here] = 4 * q + i;
                    ++e_here;
                }
            }
            gt_before += total & 0xffff;
            eq_before += total >> 16;
        });
    }
    if (!Kin) return;

    // ---- the kept rows
    __syncthreads();
    copy_rows(out, 0, nkeep, kv_in, krow, L, Kin, Vin, Kout, Vout, src_rows, ext JQ_DBG_ARG_DEV);
    if (win.w) copy_window(win, kv, krow + nkeep, tid >> 4, T >> 4, Kout, Vout, ext JQ_DBG_ARG_DEV);
}

// Shared memory of a CTA whose cluster has `cl` CTAs, the share of the head it holds, and whether its keys stay on chip.
struct SelPlan { int cl, chunk, in_smem, raw_tile; size_t smem; };

SelPlan plan_for(int L, int cl)
{
    SelPlan p;
    p.cl = cl;
    p.chunk = ((L + cl - 1) / cl + 31) / 32 * 32;
    p.in_smem = p.chunk <= kKeysSmemMax;
    p.raw_tile = p.chunk < kRawTile ? p.chunk : kRawTile;
    p.smem = (size_t)(kOwnBins + kBins + raw_words(p.raw_tile)) * 4 + (p.in_smem ? (size_t)p.chunk * 4 : 0);
    return p;
}

cudaLaunchConfig_t sel_config(const SelPlan &p, int heads, cudaLaunchAttribute (&attr)[2], cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(heads * p.cl));
    cfg.blockDim = dim3(kSelThreads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)p.cl; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    // Launched with programmatic stream serialisation: the CTAs may be set up while the kernel before it in the stream (the
    // scoring kernel) drains; the kernel waits for that kernel's memory before reading anything.
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

// Clusters of 2, 4, 8, 16 CTAs resident at a time, with two CTAs per SM (up to 100 KB of shared memory each) and with one.
struct SelDevice { int resident[4][2] = {}; bool ready = false; };
bool sel_device(SelDevice *out)
{
    static SelDevice devs[64];
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lock(mu);
    SelDevice &d = devs[dev];
    if (!d.ready) {
        const int max_smem = (kOwnBins + kBins + raw_words(kRawTile) + kKeysSmemMax) * 4;
        if (cudaFuncSetAttribute(select_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem) != cudaSuccess) return false;
        if (cudaFuncSetAttribute(select_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
        for (int i = 0; i < 4; ++i)
            for (int x = 0; x < 2; ++x) {
                SelPlan p = plan_for(1, 2 << i);
                p.smem = x == 0 ? kSelTwoPerSm : (size_t)max_smem;
                cudaLaunchAttribute attr[2];
                const cudaLaunchConfig_t cfg = sel_config(p, 1, attr, nullptr);
                if (cudaOccupancyMaxActiveClusters(&d.resident[i][x], select_cluster, &cfg) != cudaSuccess) { cudaGetLastError(); d.resident[i][x] = 0; }
            }
        if (d.resident[0][0] < 1 || d.resident[0][1] < 1) return false;
        d.ready = true;
    }
    *out = d;
    return true;
}

// Cluster size for Hkv heads of L keys: the least estimated time, rounds of resident clusters times the time of one.  That is
// a chain of phases between cluster barriers, longer in a cluster of 16, plus work in proportion to a CTA's share.  Measured
// for 8 heads with 2, 4, 8, 16 CTAs: 12.3, 9.8, 8.8, 10.3 us for 12000 keys, -, -, 19.8, 16.8 for 131072.
SelPlan choose_plan(int Hkv, int L, const SelDevice &dev)
{
    SelPlan best = plan_for(L, 8);
    double best_cost = 1e300;
    for (int i = 3; i >= 0; --i) {
        const SelPlan p = plan_for(L, 2 << i);
        const int resident = dev.resident[i][p.smem <= kSelTwoPerSm ? 0 : 1];
        if (resident < 1 || (!p.in_smem && best_cost < 1e300)) continue;
        const double cost = (double)((Hkv + resident - 1) / resident) * ((p.cl == 16 ? kSelChain16 : kSelChain) + kSelPerKey * p.chunk);
        if (cost < best_cost) { best = p; best_cost = cost; }
    }
    return best;
}

jq_status launch_select_cluster(const float *scores, const jq_shape &s, int nkeep, int Lmax, int32_t *idx, float *pooled,
                                const Workspace &w, cudaStream_t st, const void *K, const void *V, void *Kout, void *Vout,
                                const UnitTables *tables, int src_rows, int out_rows, const WindowRows &win, const SelExtents &ext)
{
    SelDevice dev;
    if (!sel_device(&dev)) return JQ_ERR_CUDA;
    const SelPlan p = choose_plan(s.Hkv, Lmax, dev);
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = sel_config(p, s.Hkv, attr, st);
    if (cudaLaunchKernelEx(&cfg, select_cluster, scores, s.L, nkeep, (s.pool - 1) / 2, idx, pooled, w.keys, p.chunk,
                           p.in_smem, p.raw_tile, (const uint4 *)K, (const uint4 *)V, (uint4 *)Kout, (uint4 *)Vout,
                           tables ? tables->heads : nullptr, (const uint4 *const *)(tables && Kout ? tables->K : nullptr),
                           (const uint4 *const *)(tables && Kout ? tables->V : nullptr), src_rows, out_rows, win, ext JQ_DBG_ARG) != cudaSuccess) {
        cudaGetLastError();
        return JQ_ERR_CUDA;
    }
    count_launch(1);
    return check_launch();
}

// The many-head kernel: 512 threads per head (measured best from 8K to 64K keys per head, 256 to 1024 heads), 1024
// when the scores of the heads that 512 would hold in flight (a head is read three times) are far more than the L2.
jq_status launch_select_stream(const float *scores, const jq_shape &s, int nkeep, int Lmax, int32_t *idx, float *pooled,
                               cudaStream_t st, const void *K, const void *V, void *Kout, void *Vout, int sms, int dev,
                               const UnitTables *tables, int src_rows, int out_rows, const WindowRows &win, const ScoredTiles *sparse, const SelExtents &ext)
{
    const long long resident = (long long)sms * stream_ctas_per_sm(512), inflight = s.Hkv < resident ? s.Hkv : resident;
    const int threads = sparse || inflight * Lmax * 4 <= (96ll << 20) ? 512 : 1024;
    const auto kernel = sparse ? select_stream<512, true> : threads == 512 ? select_stream<512, false> : select_stream<1024, false>;
    const size_t dyn = sparse ? (size_t)16 * 2 * kSparseQuads * sizeof(float4) + (size_t)kMaxSparseTiles * 4
                              : (size_t)(threads / 32) * 2 * kStageQuads * sizeof(float4);
    static bool attr_done[64][3] = {};
    const int which = sparse ? 2 : threads == 512 ? 0 : 1;
    if (dev < 0 || dev >= 64) return JQ_ERR_CUDA;
    if (!attr_done[dev][which]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn) != cudaSuccess) return JQ_ERR_CUDA;
        attr_done[dev][which] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)s.Hkv);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as for the cluster kernel
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, scores, s.L, nkeep, (s.pool - 1) / 2, idx, pooled, (const uint4 *)K,
                           (const uint4 *)V, (uint4 *)Kout, (uint4 *)Vout, tables ? tables->heads : nullptr,
                           (const uint4 *const *)(tables && Kout ? tables->K : nullptr),
                           (const uint4 *const *)(tables && Kout ? tables->V : nullptr), src_rows, out_rows, win, sparse ? *sparse : ScoredTiles(), ext JQ_DBG_ARG) != cudaSuccess) {
        cudaGetLastError();
        return JQ_ERR_CUDA;
    }
    count_launch(1);
    return check_launch();
}

}  // namespace

bool select_reads_scored_tiles(const jq_shape &s, int max_L) { return s.Hkv >= kStreamMinHeads && (s.pool - 1) / 2 <= 4 && max_L <= 128 * kMaxSparseTiles; }

jq_status launch_select(const float *scores, const jq_shape &s, int32_t *idx, float *pooled,
                        const Workspace &w, cudaStream_t st, const void *K, const void *V, void *Kout, void *Vout,
                        const UnitTables *tables, int src_head_rows, int out_head_rows, const void *Kwin, const void *Vwin, const ScoredTiles *sparse)
{
    const int src_rows = src_head_rows > s.L ? src_head_rows : s.L;
    // with tables: the plan and the shared memory follow the longest head; every head reads its own record
    const int Lmax = tables ? tables->max_L : s.L;
    const int nkeep = s.budget < Lmax ? s.budget : Lmax;
    const int out_rows = out_head_rows > nkeep ? out_head_rows : nkeep;
    const WindowRows win = {(const uint4 *)Kwin, (const uint4 *)Vwin, Vwin ? s.w : 0};
    SelExtents ext;
    ext.scores = tables ? tables->total_keys : (long long)s.Hkv * s.L;
    ext.out_rows = tables ? tables->total_rows : (long long)s.Hkv * out_rows;
    ext.src_heads = tables ? tables->hpu : s.Hkv;
    // many heads and a window the quad pooling covers: one CTA per head
    if (s.Hkv >= kStreamMinHeads && (s.pool - 1) / 2 <= 4) {
        const int sms = device_sms();
        int dev = 0;
        if (sms < 1 || cudaGetDevice(&dev) != cudaSuccess) return JQ_ERR_CUDA;
        return launch_select_stream(scores, s, nkeep, Lmax, idx, pooled, st, K, V, Kout, Vout, sms, dev, tables, src_rows, out_rows, win, sparse, ext);
    }
    return launch_select_cluster(scores, s, nkeep, Lmax, idx, pooled, w, st, K, V, Kout, Vout, tables, src_rows, out_rows, win, ext);
}

}  // namespace jq
