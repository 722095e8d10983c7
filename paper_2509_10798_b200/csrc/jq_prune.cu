// The eviction of a small budget from many keys: ONE streaming pass over K, and a second look at the few keys that can be kept.
//
//   row_stats         pass 1 over all heads of the call: a CTA takes a contiguous run of key tiles, computes S = Q K^T on the
//                     tensor cores and keeps, per query row, (reference m, l = sum of exponentials), as score_fused does.  Beside
//                     them it leaves the largest logit of every row in every block of 16 keys, as a half (2 bytes per row and
//                     block against the 4096 of the block's keys).
//   block_bounds      merges the statistics into the normalisers M_r and sums, for every block of 16 keys,
//                         score[j] <= UB[block of j] = sum_r exp2(c max_r - M_r):     one exponential for 16.
//   score_candidates  a cluster of 1 to 16 CTAs per KV head.  Round 1 scores the blocks with the largest bounds (S^T = K Q^T on the
//                     tensor cores, the blocks gathered 16 rows at a time by TMA into tiles of 128 keys) and counts, in a
//                     histogram, the pooled scores that they alone guarantee: the nkeep-th largest of these, rounded down, is a
//                     value that the threshold of the selection cannot lie below.  Round 2 scores the blocks whose bounds reach it
//                     and that round 1 left out.  A block whose bound does not reach it holds no kept key and no neighbour that
//                     makes one kept: what is not scored counts as zero.
//   the selection     (jq_select.cu) pools, selects and copies the rows as it does behind score_fused.  Its result is the same: every
//                     position that is kept has the score that it has there.
//
// Nothing is assumed about the data for the results; the time depends on it.  Where the bounds do not separate (every query's logits within a
// few tenths of each other), every block is scored, by the clusters of the heads alone, and a call takes longer than by the two-pass
// kernels, the more so the fewer heads share the GPU (us, two-pass -> this way; in brackets keys of which some stand out):
//   32 layers of 8 heads x 32768, 128 rows    985 -> 1055 (945 -> 540)       12 layers of 8 x 131072, 256 rows   2300 -> 2790 (2265 -> 1390)
//   64 x 16384, 128 rows                       127 -> 147 (124 -> 94)        8 x 131072, 256 rows                 201 -> 277 (191 -> 139)
//   8 x 131072, 128 rows                       131 -> 199 (127 -> 106)       2 x 300015, 256 rows                 125 -> 310 (123 -> 112)
// Scoring such heads from end to end with all CTAs that are free (tiles claimed through a list in memory, clusters without a head beside
// the others) was tried: 277 -> 241 us for 8 x 131072, and 1.5 % slower where the bounds do separate.
// prune_taken has the rule by which a call comes here, with what was measured.
//
// The bound holds for the scores as they are computed, not only on paper: the rounding of the half is added (block_bounds), the sum
// is raised by 1 / 512, and it is rounded up to 16 bits.  The logits that are bounded (Q K^T) and those that are scored (K Q^T) are sums of the
// same products, added along d in the same steps; that the tensor cores give the same for both is what the margins rely on where
// large products cancel (within a logit's own size they are far wider than 32-bit rounding), and test_logits_that_cancel holds it to that.
//
// What bounds it (32 layers of 8 heads, us, measured back to back on one GPU): 32768 keys, 128 rows, 512 kept: row_stats 370 (2.1 GB
// of K and 0.13 of maxima: 6.1 TB/s of the 6.5 that a copy reaches), block_bounds 50, score_candidates 50, selection 45, the last three chains of
// dependent steps per head that leave every unit half idle (ex2 54 and 33 %, issue 58 and 24 %, of the first two under ncu); the two-pass
// kernels 980.  131072 keys, 256 rows, 1024 kept: 2900 (the ex2 unit at 65 %, and the power limit: sustained calls take 7 % longer),
// 215, 140, 80; before 6000.
#include "jq_sm100.cuh"
#include "jq_tmem_ld.cuh"
#include "jq_debug.cuh"
#include <cstddef>
#include <cstring>
#include <cuda_fp16.h>
#include <mutex>

namespace jq {
namespace {

constexpr int kPTile = 128;                      // keys per tile
constexpr uint32_t kPHalf = kPTile * 128;        // one 64-column half of a tile
constexpr uint32_t kPStage = 2 * kPHalf;
constexpr int kPBlock = 16;                      // keys per block
constexpr uint32_t kPBlockHalf = kPBlock * 128;  // one 64-column half of a block

// ------------------------------------------------------------------ row statistics

constexpr int kSGroups = 4, kSEpi = 4 * kSGroups;   // epilogue groups, and their warps
constexpr int kSMaxStages = 5;
constexpr uint32_t kSSlots = 4, kSSlotCols = 128, kSTmemCols = 512;
constexpr int kSThreads = (kSEpi + 2) * 32;
static_assert(kSGroups == (int)kSSlots, "a slot per epilogue group");
// A role that waits while others work sleeps between polls (ns).
constexpr uint32_t kSSleepLong = 256, kSSleepShort = 32;

struct SCtl {
    uint64_t full[kSMaxStages], empty[kSMaxStages];
    uint64_t q_full[2], q_empty[2];
    uint64_t t_full[kSSlots], t_empty[kSSlots];
    uint32_t tmem_base;
    int abort_flag;
};
constexpr uint32_t kSCtlBytes = 1024;
static_assert(sizeof(SCtl) <= kSCtlBytes, "control block");

struct SParams {
    int L, tph;                // one shape: keys and tiles per head (the window tile included)
    int R, Rpad, w;
    int wtile;                 // every head has one more tile, the last, holding the w window keys
    int stages, hpu;           // hpu: heads per unit (ragged calls)
    long long T;               // tiles of all heads
    float c;
    int heads;
    float2 *part;              // [(CTA + head) * groups + group][R]: the statistics of one CTA's share of a head
    uint32_t *bmax;            // [tile][4][Rpad]: maxima of two blocks of 16 keys each, as halves, times c
    int *status;
    const HeadRec *htab;       // heads of different lengths or budgets (null otherwise): their records,
    const long long *tbase;    // and first tiles
    const CUtensorMap *maps, *qmaps;   // units in buffers of their own: [units] tensor maps of K, of Qwin
#ifdef JQ_DEBUG
    DebugRecord *dbg_rec;
    long long n_part, n_bmax;
#endif
};

// The head that tile `tile` of T belongs to: the last one whose first tile is not past it.  Heads of one length, or nearly, are found
// at once; the search through the others is a chain of reads from memory.
__device__ __forceinline__ int head_of_tile(const long long *tbase, int heads, long long T, long long tile)
{
    int lo = 0, hi = heads - 1;
    const int guess = min((int)(tile * heads / T), hi);
    const long long here = tbase[guess], next = guess < hi ? tbase[guess + 1] : T;
    if (here <= tile && tile < next) return guess;
    if (here <= tile) lo = guess + 1; else hi = guess - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tbase[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Where a CTA's run of tiles starts, and how a role walks it.
struct Walk {
    int h, t, tph, L;
    __device__ __forceinline__ void load(const SParams &P)
    {
        if (!P.htab) return;
        L = P.htab[h].L;
        tph = (L + kPTile - 1) / kPTile;
    }
    __device__ __forceinline__ void start(const SParams &P, long long tile)
    {
        tph = P.tph; L = P.L;
        if (!P.htab) {
            h = (int)(tile / P.tph);
            t = (int)(tile - (long long)h * P.tph);
            return;
        }
        h = head_of_tile(P.tbase, P.heads, P.T, tile);
        t = (int)(tile - P.tbase[h]);
        load(P);
    }
    __device__ __forceinline__ void advance(const SParams &P, int n)   // (never past the last tile of the call)
    {
        t += n;
        while (t >= tph) { t -= tph; ++h; load(P); }
    }
};

// Two block maxima, times c, as halves: the first block in the low half.
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi)
{
    uint32_t d;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// x + y, with x a half.
__device__ __forceinline__ float add_half(uint32_t x, float y)
{
    float d;
    asm("{\n\t.reg .b16 h;\n\tcvt.u16.u32 h, %1;\n\tadd.rn.f32.f16 %0, h, %2;\n\t}" : "=f"(d) : "r"(x), "f"(y));
    return d;
}

// As p1_half, with the largest of the 16 values handed back.
__device__ __forceinline__ float p1_half_max(uint32_t (&v)[16], int c0, int valid, float c, float lazy, float2 cc, RowState &st)
{
    if (valid < c0 + 16) {
#pragma unroll
        for (int t = 0; t < 16; ++t) if (c0 + t >= valid) v[t] = 0xff800000u;
    }
    const float cm = max_of16(v);
    if (cm > st.m + lazy) {
        const float f = ex2(c * (st.m - cm));
        st.l01 = make_float2(st.l01.x * f, st.l01.y * f);
        st.l23 = make_float2(st.l23.x * f, st.l23.y * f);
        st.m = cm;
    }
    const float nb = -st.m * c;
    exp_acc16(st.l01, st.l23, v, cc, make_float2(nb, nb));
    return cm;
}

// grid: one CTA per SM; CTA b takes tiles [b T / G, (b + 1) T / G) of the call.  Warps 0 .. 15 are the epilogue groups
// (a thread owns a query row), then
// the TMA producer and the MMA issuer.  (Four groups over four slots, also for up to 128 rows: 6 % over three groups that look
// ahead, 32 layers of 32768 keys 601 -> 565 us.)
template <bool kWide>
__global__ void __launch_bounds__(kSThreads, 1)
row_stats(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapQ,
          const __grid_constant__ CUtensorMap mapW, const __grid_constant__ SParams P)
{
    constexpr int kEpi = kSEpi, kGroups = kSGroups, nblk = kWide ? 2 : 1, bs = nblk - 1;   // blocks of 128 query rows
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    if (smem_u32(smem_raw) & 1023u) {
        if (threadIdx.x == 0) atomicMax(P.status + kWStatus, (int)JQ_ERR_CUDA);
        return;
    }
    constexpr uint32_t q_bytes = 128 * nblk * kD * 2;
    uint8_t *const qbuf = smem_raw, *const kbuf = smem_raw + 2 * (size_t)q_bytes;
    SCtl *const ctl = (SCtl *)(kbuf + (size_t)P.stages * kPStage);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = P.R, Rpad = P.Rpad, stages = P.stages;
    int *const status = P.status;
#ifdef JQ_DEBUG
    DebugRecord *const dbg = P.dbg_rec;
#endif
    const long long G = gridDim.x, first = blockIdx.x * P.T / G;
    const int ntiles = (int)((blockIdx.x + 1) * P.T / G - first);
    if (threadIdx.x == 0) {
        for (int s = 0; s < kSMaxStages; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&ctl->q_full[s], 1); mbar_init(&ctl->q_empty[s], 1); }
        for (uint32_t s = 0; s < kSSlots; ++s) { mbar_init(&ctl->t_full[s], 1); mbar_init(&ctl->t_empty[s], 4); }
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kEpi + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(kSTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t *)&ctl->tmem_base;
    cudaGridDependencySynchronize();             // no global memory has been touched so far
    cudaTriggerProgrammaticLaunchCompletion();   // the next kernel may be set up where there is room; it waits for this one's results

    if (warp == kEpi) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0) {
            uint32_t st = 0, ph = 0, qn = 0;
            int prev_h = -1, prev_unit = -1, c2 = 0;
            const CUtensorMap *mk = &mapK, *mq = &mapQ;
            Walk at;
            at.start(P, first);
#pragma unroll 1
            for (int n = 0; n < ntiles; ++n) {
                if (at.h != prev_h) {
                    prev_h = c2 = at.h;
                    if (P.maps) {
                        const int unit = at.h / P.hpu;
                        c2 = at.h - unit * P.hpu;
                        if (unit != prev_unit) {
                            mk = P.maps + unit; mq = P.qmaps + unit;
                            tensormap_acquire(mk); tensormap_acquire(mq);
                            prev_unit = unit;
                        }
                    }
                    const uint32_t qb = qn & 1;
                    if (!mbar_wait(&ctl->q_empty[qb], ((qn >> 1) & 1) ^ 1, &ctl->abort_flag, status, kSSleepLong)) break;
                    mbar_expect_tx(&ctl->q_full[qb], q_bytes);
                    tma_load_3d(qbuf + (size_t)qb * q_bytes, mq, &ctl->q_full[qb], 0, 0, c2);
                    tma_load_3d(qbuf + (size_t)qb * q_bytes + q_bytes / 2, mq, &ctl->q_full[qb], 64, 0, c2);
                    ++qn;
                }
                if (!mbar_wait(&ctl->empty[st], ph ^ 1, &ctl->abort_flag, status, kSSleepLong)) break;
                mbar_expect_tx(&ctl->full[st], kPStage);
                const bool wt = P.wtile && at.t == at.tph - 1;   // the window keys of the head (rows past w read as zero)
                const CUtensorMap *map = wt ? &mapW : mk;
                const int j0 = wt ? 0 : at.t * kPTile;
                if (JQ_IN(st, stages, kDbgPrune, 1)) {
                    tma_load_3d(kbuf + (size_t)st * kPStage, map, &ctl->full[st], 0, j0, c2);
                    tma_load_3d(kbuf + (size_t)st * kPStage + kPHalf, map, &ctl->full[st], 64, j0, c2);
                }
                if (++st == (uint32_t)stages) { st = 0; ph ^= 1; }
                if (n + 1 < ntiles) at.advance(P, 1);
            }
        }
        __syncwarp();
    } else if (warp == kEpi + 1) {
        // ---------------------------------------------------------------- MMA issuer (all 32 lanes walk the loop)
        const uint32_t idesc = instr_desc(128, kPTile);
        uint32_t st = 0, ph = 0, qn = 0, u = 0;
        int prev_h = -1;
        bool ok = true;
        Walk at;
        at.start(P, first);
#pragma unroll 1
        for (int n = 0; n < ntiles && ok; ++n) {
            if (at.h != prev_h) {
                if (qn > 0) tc_commit(&ctl->q_empty[(qn - 1) & 1]);   // the previous head's queries are free once its products retire
                if (!mbar_wait(&ctl->q_full[qn & 1], (qn >> 1) & 1, &ctl->abort_flag, status, kSSleepShort)) { ok = false; break; }
                prev_h = at.h; ++qn;
            }
            if (!mbar_wait(&ctl->full[st], ph, &ctl->abort_flag, status, kSSleepShort)) { ok = false; break; }
            const uint32_t k_lo = desc_lo(smem_u32(kbuf) + st * kPStage), q_lo = desc_lo(smem_u32(qbuf) + ((qn - 1) & 1) * q_bytes);
#pragma unroll 1
            for (int blk = 0; blk < nblk; ++blk, ++u) {
                const uint32_t slot = u % kSSlots;
                if (!mbar_wait(&ctl->t_empty[slot], ((u / kSSlots) & 1) ^ 1, &ctl->abort_flag, status, kSSleepShort)) { ok = false; break; }
                tc_fence_after();
                if (!JQ_IN(st, stages, kDbgPrune, 2)) { ok = false; break; }
                tc_mma_block(tmem + slot * kSSlotCols, q_lo + (uint32_t)blk * (kPHalf >> 4), k_lo, q_bytes / 2, kPHalf, idesc);
                tc_commit(&ctl->t_full[slot]);
            }
            if (ok) tc_commit(&ctl->empty[st]);
            if (++st == (uint32_t)stages) { st = 0; ph ^= 1; }
            if (n + 1 < ntiles) at.advance(P, 1);
        }
    } else {
        // ---------------------------------------------------------------- epilogue groups: accumulator block u is group u % kGroups'
        const int grp = warp >> 2, quarter = warp & 3, row0 = quarter * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
        const int nunits = ntiles << bs;
        const float c = P.c, lazy = 64.f / c;
        const float2 cc = make_float2(c, c);
        const int blk = grp & bs, row = blk * 128 + row0;       // with two blocks of query rows a group always has the same one
        const int win = min(P.w, row % P.w + 1);                // window keys up to the row's own position
        uint32_t va[16], vb[16];
        bool ok = true;
        auto release = [&](uint32_t slot) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->t_empty[slot], 1);
        };
        auto begin = [&](uint32_t u) -> bool {
            const uint32_t slot = u % kSSlots;
            if (!mbar_wait(&ctl->t_full[slot], (u / kSSlots) & 1, &ctl->abort_flag, status, kSSleepShort)) return false;
            tc_fence_after();
            JQ_TMEM_LD16(lane_addr + slot * kSSlotCols, va);
            return true;
        };
        RowState rs = {-INFINITY, make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        Walk at;
        if (ntiles > 0) at.start(P, first);
        int pub = ntiles > 0 ? at.h : 0, tile = 0;            // next head whose statistics this warp has to publish; tile of the run
        // Every group publishes for every head of the CTA's run, nothing seen as (-inf, 0).
        auto publish_upto = [&](int head_end) {
#pragma unroll 1
            for (; pub < head_end; ++pub) {
                const long long slot = ((long long)blockIdx.x + pub) * kGroups + grp;
                float2 *dst = P.part + slot * R;
                const bool in = JQ_IN(slot * R + R - 1, P.n_part, kDbgPrune, 3);
                if (row < R && in) dst[row] = make_float2(rs.m, (rs.l01.x + rs.l01.y) + (rs.l23.x + rs.l23.y));
                rs.m = -INFINITY;
                rs.l01 = rs.l23 = make_float2(0.f, 0.f);
            }
        };
#pragma unroll 1
        for (int k = grp; k < nunits; k += kGroups) {
            const int n = k >> bs;
            at.advance(P, n - tile);
            tile = n;
            if (at.h != pub) publish_upto(at.h);
            const uint32_t u = (uint32_t)k, slot = u % kSSlots, taddr = lane_addr + slot * kSSlotCols;
            if (!begin(u)) { ok = false; break; }
            // keys of the tile that count for this thread's row: the prefix keys or, in the window tile, the causal part of it
            const bool wt = P.wtile && at.t == at.tph - 1;
            const int valid = wt ? win : min(kPTile, at.L - at.t * kPTile);
            uint32_t *const bm = P.bmax + (first + n) * 4 * Rpad + row;
            const bool store = row < Rpad && JQ_IN((first + n + 1) * 4 * Rpad - 1, P.n_bmax, kDbgPrune, 4);   // warp-uniform
#pragma unroll 1
            for (int c0 = 0; c0 < kPTile; c0 += 32) {
                JQ_TMEM_WAIT16(va);
                JQ_TMEM_LD16(taddr + c0 + 16, vb);
                const float ma = p1_half_max(va, c0, valid, c, lazy, cc, rs);
                JQ_TMEM_WAIT16(vb);
                if (c0 + 32 < kPTile) JQ_TMEM_LD16(taddr + c0 + 32, va);
                else release(slot);
                const float mb = p1_half_max(vb, c0 + 16, valid, c, lazy, cc, rs);
                if (store) bm[(c0 >> 5) * Rpad] = pack_half2(ma * c, mb * c);
            }
        }
        if (ok && ntiles > 0) {
            at.advance(P, ntiles - 1 - tile);
            publish_upto(at.h + 1);
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");   // (a read requested ahead on a path that gave up)
    }
    tc_fence_before();
    __syncthreads();
    if (*(volatile int *)&ctl->abort_flag) __nanosleep(200000);   // let copies still in flight land before the CTA goes
    if (warp == kEpi + 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSTmemCols) : "memory");
    }
}

// ------------------------------------------------------------------ what the kernels behind row_stats share

constexpr int kCMaxCluster = 16;
constexpr int kCBins = 1024;                     // bins of 1/16 octave: 64 octaves from 2^-54 up to 2^10
constexpr int kCBase = (127 - 54) << 4;
constexpr int kCMaxStages = 4;
constexpr int kCMaxBlocks = 32767;               // block numbers are kept in 16 bits

struct CParams {
    int L, tph, nkeep;         // one shape (tph: tiles per head in row_stats' numbering, the window tile included)
    int heads, R, Rbox, Rpad, radius;
    int sms, hpu;              // row_stats' grid; heads per unit (ragged calls)
    int stages, share;         // score_candidates: K ring; most tiles of a head that a CTA looks after
    int first_pct;             // blocks of round 1 per 100 pairs kept
    long long T;
    float c;
    const float2 *part;
    const uint32_t *bmax;
    float *Ms;                 // [heads][kMaxR]: minus the row normalisers
    uint16_t *ub;              // [tile][8]: bounds of the blocks, upper 16 bits of a float
    uint8_t *scored;           // [tile]: the blocks that have been scored, as bits (null: the scores of the others are written as zeros)
    float *scores;
    int *status;
    const HeadRec *htab;
    const long long *tbase;
    const CUtensorMap *qmaps, *block_maps;   // [units]
    long long n_scores;        // floats in the scores array
#ifdef JQ_DEBUG
    DebugRecord *dbg_rec;
    long long n_part, n_bmax;
#endif
};

// A head as these kernels see it: its length and budget, its tiles (in row_stats' numbering: all, and the first one's number)
// and its scores.
struct HeadAt {
    int L, nkeep, tph1;
    long long soff, tbase;
};
__device__ __forceinline__ HeadAt head_at(const CParams &P, int h)
{
    HeadAt a;
    if (P.htab) {
        const HeadRec *r = P.htab + h;
        a.L = r->L; a.nkeep = r->nkeep; a.soff = r->soff; a.tbase = P.tbase[h];
        a.tph1 = (a.L + kPTile - 1) / kPTile;
    } else {
        a.L = P.L; a.nkeep = P.nkeep; a.soff = (long long)h * P.L; a.tbase = (long long)h * P.tph; a.tph1 = P.tph;
    }
    return a;
}

// The bin of a value >= 0 (given as the upper 16 bits of a float, rounded either way): its lower edge is not above the value.
__device__ __forceinline__ int bin_of(uint32_t top16) { return min(max((int)(top16 >> 3) - kCBase, 0), kCBins - 1); }
// The lower edge of a bin, as the upper 16 bits of a float; of the lowest bin 0.
__device__ __forceinline__ uint32_t edge_of(int bin) { return bin > 0 ? (uint32_t)(bin + kCBase) << 3 : 0u; }

template <int kThreads>
__device__ __forceinline__ void named_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory"); }

// Threads 0 .. kThreads - 1 of a CTA: exclusive scan of one int per thread, and the sum.  sums: an int per warp.
template <int kThreads>
__device__ __forceinline__ int scan_threads(int v, int &total, int *sums)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += x; }
    if (lane == 31) sums[warp] = inc;
    named_sync<kThreads>();
    const int s = lane < kThreads / 32 ? sums[lane] : 0;
    total = __reduce_add_sync(0xffffffffu, s);
    const int before = __reduce_add_sync(0xffffffffu, lane < warp ? s : 0);
    named_sync<kThreads>();
    return before + inc - v;
}

// The same threads: the bin that holds the target-th entry from the top (without so many entries: bin 0).  get(i) gives the
// counts of bins i, i + 1.
template <int kThreads, int kN, typename Get>
__device__ __forceinline__ int find_bin(Get get, int target, int *res, int *sums)
{
    constexpr int per = kN / kThreads;                        // consecutive bins of a thread, from the top
    const int at = kN - per * ((int)threadIdx.x + 1);
    int n[per], sum = 0, total;
#pragma unroll
    for (int i = 0; i < per; i += 2) { const uint2 v = get(at + i); n[i] = (int)v.x; n[i + 1] = (int)v.y; }
#pragma unroll
    for (int i = 0; i < per; ++i) sum += n[i];
    if (threadIdx.x == 0) *res = 0;
    int above = scan_threads<kThreads>(sum, total, sums);
#pragma unroll
    for (int i = per - 1; i >= 0; --i) {
        if (above < target && target <= above + n[i]) *res = at + i;
        above += n[i];
    }
    named_sync<kThreads>();
    return *res;
}

// ------------------------------------------------------------------ bounds

constexpr int kBThreads = 256, kBStages = 3;     // stages: tiles of a warp, two on their way while one is worked on
__host__ __device__ constexpr int bounds_per_sm(bool wide) { return wide ? 2 : 3; }
__host__ __device__ constexpr int bounds_smem(bool wide) { return kBThreads / 32 * kBStages * (wide ? 4096 : 2048); }

// grid: two or three CTAs per SM, CTA b takes tiles [b T / G, (b + 1) T / G).  Per head: the normalisers from row_stats' partial statistics,
// then a bound per block of 16 keys.  Neither the read of the maxima bounds it (3.2 TB/s with up to 128 rows, 2.1 with more) nor the
// exponentials (the ex2 unit 54 and 38 % busy): a CTA does the merge of a head, a chain of loads, before it streams the head's
// tiles; how the time divides has not been measured.  (The cap of 80 registers for three CTAs costs block_bounds<false> 52 bytes of spills.)
// The bound stays above what it bounds: a maximum x
// within 24 of its row's normaliser M has been rounded by at most (|M| + 24) / 2048, of which a little more is added (room for the rounding
// of x - M); smaller ones are below 2^-24, which every row adds; the sum is raised by 1 / 512,
// far above what exponentials and sums are off by; a normaliser near the end of a half's range makes every bound of the head
// infinite.  (With wider margins, 64, 1 / 64, the ragged batch of 128 units took 1862 us instead of 1847.)
template <bool kWide>
__global__ void __launch_bounds__(kBThreads, bounds_per_sm(kWide))
block_bounds(const __grid_constant__ CParams P)
{
    __shared__ float Ms[kMaxR];
    __shared__ float2 other[kMaxR];
    __shared__ int huge;
    extern __shared__ __align__(16) uint8_t bounds_raw[];
    constexpr int kJ = kWide ? 8 : 4;                         // most pieces of 32 rows
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, pair = lane >> 3, g = lane & 7;
    const int R = P.R, Rpad = P.Rpad, nj = Rpad >> 5;
    // The warp's stages.  Lanes 8 q .. 8 q + 7 have the blocks 2 q and 2 q + 1 of a tile: lane 8 q + g, of every piece of 32 rows, the
    // rows 4 g .. 4 g + 3, 16 bytes that it copies and reads itself.
    uint4 *const ring = (uint4 *)bounds_raw + warp * kBStages * kJ * 32 + lane;
#ifdef JQ_DEBUG
    DebugRecord *const dbg = P.dbg_rec;
#endif
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();   // the stream's next kernel may be set up meanwhile; it waits for this one's results
    const long long G = gridDim.x;
    long long f = blockIdx.x * P.T / G;
    const long long end = (blockIdx.x + 1) * P.T / G;
    int h = P.htab ? head_of_tile(P.tbase, P.heads, P.T, f) : (int)(f / P.tph);
#pragma unroll 1
    for (; f < end; ++h) {
        const HeadAt a = head_at(P, h);
        const int t0 = (int)(f - a.tbase), tph = (a.L + kPTile - 1) / kPTile, nb = (a.L + kPBlock - 1) / kPBlock;
        const int t1 = (int)min((long long)tph, end - a.tbase);       // (the window tile has no bounds)
        f = a.tbase + a.tph1;
        if (tid == 0) huge = 0;
        const uint32_t *const mine = P.bmax + a.tbase * 4 * Rpad + pair * Rpad + 4 * g;
        auto request = [&](int t, int stage) {
            const uint32_t *const from = mine + (long long)t * 4 * Rpad;
            const uint32_t to = smem_u32(ring + stage * kJ * 32);
            if (t < t1 && JQ_IN((a.tbase + t + 1) * 4 * Rpad - 1, P.n_bmax, kDbgPrune, 6)) {
#pragma unroll
                for (int j = 0; j < kJ; ++j)
                    if (j < nj) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + j * 512), "l"(from + 32 * j) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        request(t0 + warp, 0);
        request(t0 + warp + kBThreads / 32, 1);
        {   // the CTAs of row_stats that had tiles of this head, each with a pair per row and group:
            // kDeep loads in flight (a head that all CTAs share has up to 38 or 76 pairs per row)
            constexpr int kDeep = 16;
            const long long c_lo = ((a.tbase + 1) * P.sms - 1) / P.T, c_hi = ((a.tbase + a.tph1) * P.sms - 1) / P.T;   // owners of the first and last tile
            constexpr int kSub = kWide ? 1 : 2;                       // threads per row
            const int row = tid & (kWide ? 255 : 127), sub = kWide ? 0 : tid >> 7;
            // (with two blocks of query rows every other group has the row)
            constexpr int kStep = kWide ? 2 : 1;
            const int nsl = (int)(c_hi - c_lo + 1) * (kSGroups / kStep);
            const long long s0 = (c_lo + h) * kSGroups + (kWide ? row >> 7 : 0);
            const float2 *src = P.part + s0 * R + row;
            float m = -INFINITY, l = 0.f;
            if (row < R) {
#pragma unroll 1
                for (int i0 = sub; i0 < nsl; i0 += kDeep * kSub) {
                    float2 p[kDeep];
                    float mn = m;
#pragma unroll
                    for (int k = 0; k < kDeep; ++k) {
                        const int i = i0 + kSub * k;
                        p[k] = i < nsl && JQ_IN((s0 + i * kStep) * R + row, P.n_part, kDbgPrune, 5) ? __ldcg(src + (size_t)(i * kStep) * R) : make_float2(-INFINITY, 0.f);
                        if (p[k].y > 0.f) mn = fmaxf(mn, p[k].x);
                    }
                    if (mn > -INFINITY) {
                        l *= ex2(P.c * (m - mn));
#pragma unroll
                        for (int k = 0; k < kDeep; ++k) if (p[k].y > 0.f) l = fmaf(p[k].y, ex2(P.c * (p[k].x - mn)), l);
                        m = mn;
                    }
                }
            }
            if (sub == 1) other[row] = make_float2(m, l);
            __syncthreads();
            if (sub == 0) {
                float M = INFINITY;                                   // silences a column that is not a query row
                if (row < R) {
                    if (kSub == 2) {
                        const float2 o = other[row];
                        const float mn = fmaxf(m, o.x);
                        l = (l > 0.f ? l * ex2(P.c * (m - mn)) : 0.f) + (o.y > 0.f ? o.y * ex2(P.c * (o.x - mn)) : 0.f);
                        m = mn;
                    }
                    M = fmaf(P.c, m, log2f(l));
                    if (!(fabsf(M) < 60000.f)) huge = 1;
                }
                Ms[row] = -M;
                if (!kWide) Ms[128 + row] = -INFINITY;
                if (t0 == 0 && JQ_IN(h, P.heads, kDbgPrune, 15)) { P.Ms[(size_t)h * kMaxR + row] = -M; if (!kWide) P.Ms[(size_t)h * kMaxR + 128 + row] = -INFINITY; }
            }
            __syncthreads();
        }
        float nm[4 * kJ];
#pragma unroll
        for (int j = 0; j < kJ; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float x = Ms[32 * j + 4 * g + i];
                nm[4 * j + i] = x > -INFINITY ? x + (fabsf(x) + 24.f) * (1.f / 2040.f) : x;   // (a row that is none stays at -inf)
            }
        const float least = huge ? INFINITY : (float)R * 6e-8f;
        int stage = 0;
#pragma unroll 1
        for (int t = t0 + warp; t < t1; t += kBThreads / 32) {
            request(t + 2 * (kBThreads / 32), stage == 0 ? 2 : stage - 1);
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            float2 sum = make_float2(0.f, 0.f), sum2 = sum;
#pragma unroll
            for (int j = 0; j < kJ; ++j) {
                if (j >= nj) break;
                const uint4 v = ring[(stage * kJ + j) * 32];
                const uint32_t e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 x = make_float2(ex2(add_half(e[i] & 0xffffu, nm[4 * j + i])), ex2(add_half(e[i] >> 16, nm[4 * j + i])));
                    if (i & 1) sum2 = __fadd2_rn(sum2, x); else sum = __fadd2_rn(sum, x);
                }
            }
            sum = __fadd2_rn(sum, sum2);
            // two sums over eight lanes: after an exchange of halves a lane holds one block's part
            const bool odd = lane & 4;
            float r = (odd ? sum.y : sum.x) + __shfl_xor_sync(0xffffffffu, odd ? sum.x : sum.y, 4);
            r += __shfl_xor_sync(0xffffffffu, r, 2);
            r += __shfl_xor_sync(0xffffffffu, r, 1);
            const int blk = 2 * pair + (odd ? 1 : 0);
            if ((lane & 3) == 0 && JQ_IN(a.tbase + t, P.T, kDbgPrune, 16))
                P.ub[(a.tbase + t) * 8 + blk] = 8 * t + blk < nb ? (uint16_t)((__float_as_uint((r + least) * (1.f + 1.f / 512.f)) + 0xffffu) >> 16) : (uint16_t)0;
            stage = stage == kBStages - 1 ? 0 : stage + 1;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");          // (the next head starts with the first stage again)
        __syncthreads();
    }
}

// ------------------------------------------------------------------ scores of the candidates

__host__ __device__ constexpr int cand_groups(bool wide) { return wide ? 4 : 2; }
__host__ __device__ constexpr int cand_threads(bool wide) { return cand_groups(wide) * 128 + 64; }

struct CCtl {
    uint64_t full[kCMaxStages], empty[kCMaxStages], q_full, t_full[2], t_empty[2];
    uint32_t tmem_base;
    int abort_flag;
    int n;                                       // blocks on this CTA's list
    int found;                                   // (find_bin)
    int sums[16];
    int cnt[kCMaxCluster];                       // candidates of every CTA's share of the head
    alignas(16) float xs[2][2][kPTile];          // (R > 128) the second column half's sums on their way to the first half's threads
    alignas(16) float Ms[kMaxR];                 // minus the row normalisers
};
constexpr uint32_t kCCtlBytes = 4096;
static_assert(sizeof(CCtl) <= kCCtlBytes && offsetof(CCtl, Ms) % 16 == 0, "control block");

__device__ __forceinline__ uint32_t remote(const void *p, uint32_t rank)   // the same place in CTA `rank` of the cluster
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ uint2 remote_ld2(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void remote_st(uint32_t a, int v) { asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void remote_st16(uint32_t a, uint16_t v) { asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"(v) : "memory"); }

template <bool kWide>
__global__ void __launch_bounds__(cand_threads(kWide), kWide ? 1 : 2)
score_candidates(const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CParams P)
{
    constexpr int kGroups = cand_groups(kWide), kEpi = 4 * kGroups, kTE = 32 * kEpi;
    constexpr uint32_t kSlotCols = kWide ? 256 : 128, kCols = 2 * kSlotCols;   // two accumulators in tensor memory
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t q_bytes = (uint32_t)P.Rbox * kD * 2;
    uint8_t *const qbuf = smem_raw, *const kbuf = smem_raw + q_bytes;
    CCtl *const ctl = (CCtl *)(kbuf + (size_t)P.stages * kPStage);
    uint32_t *const hist = (uint32_t *)((uint8_t *)ctl + kCCtlBytes);            // [kCBins]
    uint16_t *const ub = (uint16_t *)(hist + kCBins);                            // [8 share]: bounds of this CTA's share
    uint16_t *const list = ub + 8 * P.share;                                     // [8 share]: blocks that this CTA scores
    uint32_t *const words = (uint32_t *)(list + 8 * P.share);                    // [share / 4 + 1]: blocks as bits,
    int *const wbase = (int *)(words + P.share / 4 + 1);                         // and how many come before each word
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t rank, C;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const int head = (int)(blockIdx.x / C);
    int *const status = P.status;
    const int Rpad = P.Rpad;
#ifdef JQ_DEBUG
    DebugRecord *const dbg = P.dbg_rec;
#endif
    if (smem_u32(smem_raw) & 1023u) {   // uniform over the grid
        if (tid == 0) atomicMax(status + kWStatus, (int)JQ_ERR_CUDA);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < kCMaxStages; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        mbar_init(&ctl->q_full, 1);
        for (int s = 0; s < 2; ++s) { mbar_init(&ctl->t_full[s], 1); mbar_init(&ctl->t_empty[s], kWide ? 8 : 4); }
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kEpi + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(kCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < kCBins; i += blockDim.x) hist[i] = 0u;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t *)&ctl->tmem_base;
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // waited for before another CTA's memory is touched
    cudaGridDependencySynchronize();             // nothing in global memory has been touched so far
    cudaTriggerProgrammaticLaunchCompletion();   // the stream's next kernel may be set up meanwhile; it waits for this one's results

    const HeadAt at = head_at(P, head);
    const int L = at.L, nkeep = at.nkeep;
    int kv_in = head;
    const CUtensorMap *mb = &mapB, *mq = &mapQ;
    if (P.qmaps) {
        const int unit = head / P.hpu;
        kv_in = head - unit * P.hpu;
        mq = P.qmaps + unit; mb = P.block_maps + unit;
    }
    const int tph = (L + kPTile - 1) / kPTile, nb = (L + kPBlock - 1) / kPBlock;
    const int ts = (int)((long long)rank * tph / C), te = (int)((long long)(rank + 1) * tph / C);   // tiles of the head that this CTA looks after
    const int b0 = 8 * ts, nbs = min(8 * te, nb) - b0, nw = (nbs + 31) >> 5;                    // their blocks, as words of 32
    auto cluster_sync = [&]() {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    };
    auto sync_all = [&]() { if (C == 1) __syncthreads(); else cluster_sync(); };   // all warps of the head's CTAs
    // counts of two bins, over all CTAs of the head
    auto counts = [&](int i) -> uint2 {
        if (C == 1) return *(const uint2 *)(hist + i);
        uint2 s = make_uint2(0u, 0u);
#pragma unroll 4
        for (uint32_t d = 0; d < C; ++d) { const uint2 v = remote_ld2(remote(hist + i, d)); s.x += v.x; s.y += v.y; }
        return s;
    };

    uint32_t st = 0, ph = 0, u = 0;                           // K ring and its phase; tiles so far
    uint32_t lo16 = 0u, hi16 = 0u;                            // the blocks of a round: bounds in [lo16, hi16)
    if (warp == kEpi) {
        if (lane == 0) {
            if (P.qmaps) { tensormap_acquire(mq); tensormap_acquire(mb); }
            mbar_expect_tx(&ctl->q_full, q_bytes);
            tma_load_3d(qbuf, mq, &ctl->q_full, 0, 0, kv_in);
            tma_load_3d(qbuf + q_bytes / 2, mq, &ctl->q_full, 64, 0, kv_in);
        }
        __syncwarp();
        if (P.qmaps) tensormap_acquire(mb);                    // (all lanes load)
    } else if (warp < kEpi) {
        for (int i = tid; i < kMaxR; i += kTE) if (JQ_IN(head, P.heads, kDbgPrune, 17)) ctl->Ms[i] = __ldcg(P.Ms + (size_t)head * kMaxR + i);
        const uint16_t *const src = P.ub + (size_t)(at.tbase + ts) * 8;
        for (int t = tid; t < te - ts; t += kTE) {
            if (!JQ_IN(t, P.share, kDbgPrune, 7) || !JQ_IN(at.tbase + ts + t, P.T, kDbgPrune, 18)) continue;
            const uint4 v = __ldcg((const uint4 *)src + t);
            ((uint4 *)ub)[t] = v;
            const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) if (8 * t + e < nbs) atomicAdd(&hist[bin_of(x[e >> 1] >> (16 * (e & 1)) & 0xffffu)], 1u);
        }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    sync_all();

    const int wanted = max(1, min(nb, (int)((long long)nkeep * P.first_pct / 100) + 1));
#pragma unroll 1
    for (int round = 0; round < 2; ++round) {
        // ---- the blocks of this round: [lo16, hi16) of the bounds
        if (warp < kEpi) {
            const uint32_t edge = edge_of(find_bin<kTE, kCBins>(counts, round == 0 ? wanted : nkeep, &ctl->found, ctl->sums));
            if (round == 0) { lo16 = edge; hi16 = 0x10000u; }
            else { hi16 = lo16; lo16 = min(edge, lo16); }
            // this CTA's share of them, and their places in the head's list
            for (int w = warp; w < nw; w += kEpi) {
                const int i = 32 * w + lane;
                const uint32_t x = i < nbs && JQ_IN(i, 8 * P.share, kDbgPrune, 19) ? ub[i] : 0x10000u, m = __ballot_sync(0xffffffffu, x >= lo16 && x < hi16);
                if (lane == 0 && JQ_IN(w, P.share / 4 + 1, kDbgPrune, 20)) words[w] = m;
            }
            named_sync<kTE>();
            int total;
            const int base = scan_threads<kTE>(tid < nw ? __popc(words[tid]) : 0, total, ctl->sums);
            if (tid < nw && JQ_IN(tid, P.share / 4 + 1, kDbgPrune, 21)) wbase[tid] = base;
            named_sync<kTE>();
            int before = 0, per_cta = 0x40000000;
            if (C > 1) {
                if (warp == 0 && lane < (int)C) remote_st(remote(&ctl->cnt[rank], lane), total);
                cluster_sync();
                const int have = lane < (int)C ? ctl->cnt[lane] : 0;
                const int all = __reduce_add_sync(0xffffffffu, have);
                before = __reduce_add_sync(0xffffffffu, lane < (int)rank ? have : 0);
                per_cta = max(8, ((all + (int)C - 1) / (int)C + 7) & ~7);        // whole tiles
                if (tid == 0) ctl->n = min(max(all - (int)rank * per_cta, 0), per_cta);
            } else if (tid == 0) ctl->n = total;
            for (int w = warp; w < nw; w += kEpi) {
                const uint32_t m = words[w];
                if ((m >> lane & 1u) == 0u) continue;
                const int i = before + wbase[w] + __popc(m & ((1u << lane) - 1u)), to = C > 1 ? i / per_cta : 0, x = i - to * per_cta;
                if (!JQ_IN(x, 8 * P.share, kDbgPrune, 8) || !JQ_IN(to, C, kDbgPrune, 9)) continue;
                if (C > 1) remote_st16(remote(list + x, (uint32_t)to), (uint16_t)(b0 + 32 * w + lane));
                else list[x] = (uint16_t)(32 * w + lane);
            }
            for (int i = tid; i < kCBins; i += kTE) hist[i] = 0u;   // (everybody has read it)
        } else if (C > 1) cluster_sync();
        sync_all();
        const int n = ctl->n, nt = (n + 7) >> 3;
        if (warp == kEpi) {
            // ------------------------------------------------------------ TMA producer: up to eight blocks to a tile, two lanes each
#pragma unroll 1
            for (int i = 0; i < nt; ++i) {
                const int have = min(8, n - 8 * i);
                if (!__all_sync(0xffffffffu, mbar_wait(&ctl->empty[st], ph ^ 1, &ctl->abort_flag, status, 64))) break;
                if (lane == 0) mbar_expect_tx(&ctl->full[st], (uint32_t)have * 2u * kPBlockHalf);
                __syncwarp();
                if ((lane >> 1) < have) {
                    const int x = lane >> 1, half = lane & 1, blk = list[8 * i + x];
                    if (JQ_IN(blk, nb, kDbgPrune, 11) && JQ_IN(st, P.stages, kDbgPrune, 12))
                        tma_load_3d(kbuf + (size_t)st * kPStage + half * kPHalf + x * kPBlockHalf, mb, &ctl->full[st], 64 * half, blk * kPBlock, kv_in);
                }
                __syncwarp();
                if (++st == (uint32_t)P.stages) { st = 0; ph ^= 1; }
            }
        } else if (warp == kEpi + 1) {
            // ------------------------------------------------------------ MMA issuer
            const uint32_t ia = instr_desc(kPTile, min(128, Rpad)), ib = instr_desc(kPTile, max(32, Rpad - 128));
            const uint32_t q_lo = desc_lo(smem_u32(qbuf));
            bool ok = mbar_wait(&ctl->q_full, 0, &ctl->abort_flag, status, 32);   // (also without tiles: the copy must have landed when the CTA leaves)
#pragma unroll 1
            for (int i = 0; i < nt && ok; ++i, ++u) {
                const uint32_t slot = u & 1;
                if (!mbar_wait(&ctl->full[st], ph, &ctl->abort_flag, status, 32) ||
                    !mbar_wait(&ctl->t_empty[slot], ((u >> 1) & 1) ^ 1, &ctl->abort_flag, status, 32)) { ok = false; break; }
                tc_fence_after();
                const uint32_t k_lo = desc_lo(smem_u32(kbuf) + st * kPStage), d = tmem + slot * kSlotCols;
                tc_mma_block(d, k_lo, q_lo, kPHalf, q_bytes / 2, ia);
                if (kWide) tc_mma_block(d + 128, k_lo, q_lo + (kPHalf >> 4), kPHalf, q_bytes / 2, ib);
                tc_commit(&ctl->t_full[slot]);
                tc_commit(&ctl->empty[st]);
                if (++st == (uint32_t)P.stages) { st = 0; ph ^= 1; }
            }
        } else {
            // ------------------------------------------------------------ epilogue: a thread owns a key and adds exp2(c s - M_r) over the rows
            const int grp = warp >> 2, quarter = warp & 3, row0 = quarter * 32 + lane;
            const uint32_t mine = kWide ? (uint32_t)grp >> 1 : (uint32_t)grp;     // which of the two accumulators: every other tile
            const int half = kWide ? grp & 1 : 0;                                 // (R > 128) the first or the second 128 columns
            const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + mine * kSlotCols + (uint32_t)half * 128;
            const int np = (half ? Rpad - 128 : min(128, Rpad)) >> 5;
            const float2 cc = make_float2(P.c, P.c);
            const float4 *const bias = (const float4 *)(ctl->Ms + 128 * half);
            uint32_t va[16], vb[16];
#pragma unroll 1
            for (int i = (int)((mine - u) & 1u); i < nt; i += 2) {
                const uint32_t uu = u + (uint32_t)i;
                // (after a wait that ran out the loop goes on without reading: the groups meet at a barrier below)
                const bool ok = __all_sync(0xffffffffu, mbar_wait(&ctl->t_full[mine], (uu >> 1) & 1, &ctl->abort_flag, status, 32));
                tc_fence_after();
                if (ok) JQ_TMEM_LD16(lane_addr, va);
                float2 a01 = make_float2(0.f, 0.f), a23 = a01;
#pragma unroll 1
                for (int p = 0; p < (ok ? np : 0); ++p) {
                    JQ_TMEM_WAIT16(va);
                    JQ_TMEM_LD16(lane_addr + 32 * p + 16, vb);
                    exp_acc16(a01, a23, va, cc, bias + 8 * p);
                    JQ_TMEM_WAIT16(vb);
                    if (p + 1 < np) JQ_TMEM_LD16(lane_addr + 32 * p + 32, va);
                    else {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&ctl->t_empty[mine], 1);
                    }
                    exp_acc16(a01, a23, vb, cc, bias + 8 * p + 4);
                }
                float sum = (a01.x + a01.y) + (a23.x + a23.y);
                if (kWide) {                                  // the two halves of a key's sum meet in the first half's thread
                    float *const xs = ctl->xs[mine][(uu >> 1) & 1];
                    if (half) xs[row0] = sum;
                    asm volatile("bar.sync %0, 256;" ::"r"(2 + mine) : "memory");
                    if (half) continue;
                    sum += xs[row0];
                }
                const int x = 8 * i + (row0 >> 4), blk = x < n ? list[x] : nb, key = blk * kPBlock + (row0 & 15);
                const bool have = x < n && key < L;
                if (have && JQ_IN(at.soff + key, P.n_scores, kDbgPrune, 13)) P.scores[at.soff + key] = sum;
                if (round == 0) {
                    // what this block alone guarantees of the pooled scores of its positions
                    float m = have ? sum : 0.f;
                    int w = 0;
#pragma unroll 1
                    while (w < min(P.radius, 15)) {
                        const int s = min(2 * w + 1, min(P.radius, 15) - w);
                        m = fmaxf(m, fmaxf(__shfl_up_sync(0xffffffffu, m, s, 16), __shfl_down_sync(0xffffffffu, m, s, 16)));
                        w += s;
                    }
                    if (have) atomicAdd(&hist[bin_of(__float_as_uint(m) >> 16)], 1u);
                }
            }
        }
        if (warp < kEpi) u += (uint32_t)nt;
        sync_all();
    }
    if (warp >= kEpi) {
        // all products have been read: the two warps are through
        if (warp == kEpi + 1) {
            if (*(volatile int *)&ctl->abort_flag) __nanosleep(200000);   // let copies still in flight land before the CTA goes
            __syncwarp();
            tc_fence_after();
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
        }
        return;
    }

    // what nothing needs counts as zero: told to the selection as bits, or written where it reads every score
    if (P.scored) {
        for (int t = tid; t < te - ts; t += kTE) {
            uint32_t m = 0u;
#pragma unroll
            for (int e = 0; e < 8; ++e) m |= (uint32_t)(8 * t + e < nbs && ub[8 * t + e] >= lo16) << e;
            if (JQ_IN(at.tbase + ts + t, P.T, kDbgPrune, 22)) P.scored[at.tbase + ts + t] = (uint8_t)m;
        }
        return;
    }
    float *const s = P.scores + at.soff + (long long)b0 * kPBlock;
    const int m = min(nbs * kPBlock, L - b0 * kPBlock);
    for (int i = tid; i < m; i += kTE)
        if (ub[i >> 4] < lo16 && JQ_IN(at.soff + (long long)b0 * kPBlock + i, P.n_scores, kDbgPrune, 14)) s[i] = 0.f;
}

// ------------------------------------------------------------------ host side

constexpr size_t stats_smem(int Rbox, int stages) { return 2 * (size_t)Rbox * kD * 2 + (size_t)stages * kPStage + kSCtlBytes; }
size_t cand_smem(int Rbox, int stages, int share) { return (size_t)Rbox * kD * 2 + (size_t)stages * kPStage + kCCtlBytes + kCBins * 4 + (size_t)share * 32 + (size_t)(share / 4 + 1) * 8; }
constexpr size_t kCMaxSmem = 227 * 1024, kCTwoPerSm = 113 * 1024;

struct PruneDevice {
    int sms = 0;
    int resident[2][kCMaxCluster + 1] = {};   // [R > 128][C]: clusters of C CTAs that fit at a time with an SM for each CTA (what the
                                              // runtime answers for a kernel that allocates tensor memory, also where two fit)
    bool ready = false;
};

bool prune_device(PruneDevice *out)
{
    static PruneDevice devs[64];
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lock(mu);
    PruneDevice &d = devs[dev];
    if (!d.ready) {
        d.sms = device_sms();
        if (d.sms < 1) return false;
        for (auto k : {row_stats<false>, row_stats<true>})
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCMaxSmem) != cudaSuccess) return false;
        for (int wide = 0; wide < 2; ++wide) {
            if (cudaFuncSetAttribute(wide ? block_bounds<true> : block_bounds<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bounds_smem(wide)) != cudaSuccess) return false;
            const auto k = wide ? score_candidates<true> : score_candidates<false>;
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCMaxSmem) != cudaSuccess ||
                cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
            for (int C = 1; C <= kCMaxCluster; ++C) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3((unsigned)C);
                cfg.blockDim = dim3((unsigned)cand_threads(wide));
                cfg.dynamicSmemBytes = wide ? kCMaxSmem : kCTwoPerSm;
                cudaLaunchAttribute attr[1];
                attr[0].id = cudaLaunchAttributeClusterDimension;
                attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
                cfg.attrs = attr;
                cfg.numAttrs = 1;
                if (cudaOccupancyMaxActiveClusters(&d.resident[wide][C], k, &cfg) != cudaSuccess) { cudaGetLastError(); d.resident[wide][C] = 0; }
            }
        }
        d.ready = true;
    }
    *out = d;
    return true;
}

// The scratch: maxima, partial statistics, normalisers, bounds, scored blocks.
struct PruneScratch { size_t part, Ms, ub, scored, bytes; };
PruneScratch prune_layout(long long tiles, int heads, int R)
{
    const int Rpad = (R + 31) & ~31;
    PruneScratch s;
    s.part = align_up((size_t)tiles * 4 * Rpad * 4, 256);
    s.Ms = s.part + align_up((size_t)(heads + 256) * kSGroups * R * sizeof(float2), 256);
    s.ub = s.Ms + align_up((size_t)heads * kMaxR * 4, 256);
    s.scored = s.ub + align_up((size_t)tiles * 16, 256);
    s.bytes = s.scored + align_up((size_t)tiles, 256);
    return s;
}

template <typename... A>
bool launch(void (*kernel)(A...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st, int cluster, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) { cudaGetLastError(); return false; }
    count_launch(1);
    return true;
}

}  // namespace

size_t prune_bytes(long long tiles, int heads, int R) { return prune_layout(tiles, heads, R).bytes; }

// Positions that are kept per block of 16 that holds one, roughly: a peak of the scores lifts the whole window around it.
static double kept_per_block(int pool) { return pool >= 7 ? 7.0 : pool >= 3 ? 3.5 : 1.3; }

// Whether a call takes this way.  tiles, keys, kept: of all heads, the lengths and what the heads keep.  What it saves is the second
// pass over the tiles; what it costs is two more launches (with what they have to do before their first byte), and the scores of
// the candidates, in proportion to the share that is kept.  Both sides were measured over 579 calls (us, two-pass kernel -> this
// way; keys without structure, and in brackets keys that share directions by segments, which the bounds separate badly), with a
// window of 7 and 128 query rows:
//   8 heads x 32768, 65536, 131072 keys, 1 % kept       47 -> 58, 76 -> 75, 128 -> 108
//   64 x 8192, 16384, 32768, 1 %                         76 -> 71 (92), 137 -> 100 (130), 240 -> 157 (220)
//   64 x 32768, 3 % and 8 %                              252 -> 188 (240), 272 -> 260 (297)
//   256 x 4096, 3 %                                      136 -> 114 (148)
//   64 x 32768, 1.5 %, windows of 1, 3, 13               252 -> 262, 251 -> 179, 256 -> 164
// With 8 query rows 64 x 32768 keys take 211 -> 141 (1 %), with 256 rows 371 -> 240.  Shorter heads than about 10000 keys gain little
// and lose most where the bounds separate badly; fewer than 8 rows have not been measured and stay where they were.
static double saved_per_tile(int R) { return R > 128 ? 9.0e-3 : R > 64 ? 6.2e-3 : 5.5e-3; }   // us
// us that have to be saved.  With fewer than four heads the kernels behind row_stats have a cluster or three on the whole GPU and take two to
// three times as long (1 x 500000, 256 rows 165 -> 166; 2 x 500000, 64, 128, 256 rows 156 -> 161, 166 -> 169, 233 -> 202; 2 x 300015,
// 256 rows 123 -> 112; 3 x 249386, 64 rows, keys in segments 91 -> 125).
static double prune_least(int heads, int R) { return heads >= 4 ? 30.0 : R > 128 ? 40.0 : 60.0; }

bool prune_possible(int heads, int R, long long keys, int max_L)
{
    const long long tiles = keys / kPTile + heads;
    return R >= 8 && tiles < (1ll << 30) && max_L <= kPBlock * kCMaxBlocks && keys >= 10000ll * heads && (double)tiles * saved_per_tile(R) >= prune_least(heads, R);
}

bool prune_taken(const jq_shape &s, int heads, long long tiles, long long keys, long long kept, int max_L)
{
    const int R = s.group * s.w;
    if (!prune_possible(heads, R, keys, max_L)) return false;
    const double share = (double)kept / (double)keys * 7.0 / kept_per_block(s.pool);
    return (double)tiles * (saved_per_tile(R) - 0.08 * share) >= prune_least(heads, R);
}

jq_status launch_evict_pruned(const void *K, const void *V, const void *Q, const jq_shape &s, void *Kout, void *Vout, int32_t *idx,
                              const Workspace &w, cudaStream_t st, const UnitTables *tables, int src_head_rows, int out_head_rows,
                              const void *Kwin, const void *Vwin)
{
    PruneDevice dev;
    if (!prune_device(&dev)) return JQ_ERR_CUDA;
    const int R = s.group * s.w, Rbox = R <= 128 ? 128 : 256, Rpad = (R + 31) & ~31, wide = R > 128;
    const int wtile = Kwin ? 1 : 0, tph = (s.L + kPTile - 1) / kPTile + wtile;
    const long long T = tables ? tables->total_tiles : (long long)s.Hkv * tph;
    SParams S = {};
    S.L = s.L; S.tph = tph; S.R = R; S.Rpad = Rpad; S.w = s.w; S.wtile = wtile;
    S.stages = wide ? 3 : 5;
    S.T = T; S.heads = s.Hkv; S.hpu = tables ? tables->hpu : s.Hkv;
    S.c = 1.4426950408889634f / sqrtf((float)s.d);
    S.bmax = (uint32_t *)w.prune;
    const PruneScratch lay = prune_layout(T, s.Hkv, R);
    char *const scratch = (char *)w.prune;
    S.part = (float2 *)(scratch + lay.part);
    S.status = w.status;
    const int grid = (int)(T < dev.sms ? T : dev.sms);
    CParams P = {};
    CUtensorMap mapK, mapQ, mapW, mapB;
    if (tables) {
        memset(&mapK, 0, sizeof mapK);
        mapQ = mapW = mapB = mapK;
        if (tables->tbase) { S.htab = tables->heads; S.tbase = tables->tbase; }   // (lengths from tables are a chain of reads before anything starts)
        S.maps = (const CUtensorMap *)tables->maps;
        S.qmaps = (const CUtensorMap *)tables->qmaps;
    } else {
        if (!make_tensor_map(&mapK, K, s.L, s.Hkv, kPTile, src_head_rows) || !make_tensor_map(&mapQ, Q, R, s.Hkv, Rbox) ||
            !make_tensor_map(&mapB, K, s.L, s.Hkv, kPBlock, src_head_rows))
            return JQ_ERR_CUDA;
        if (Kwin) { if (!make_tensor_map(&mapW, Kwin, s.w, s.Hkv, kPTile)) return JQ_ERR_CUDA; } else mapW = mapK;
    }
    const int max_tph = ((tables ? tables->max_L : s.L) + kPTile - 1) / kPTile;
    // CTAs per head: as many as leave the heads resident at a time
    int C = 1;
    for (int x = 1; x <= kCMaxCluster && x <= max_tph; ++x)
        if (dev.resident[wide][x] >= s.Hkv) C = x;
    P.stages = wide ? 3 : 2;
    while (C < kCMaxCluster && C < max_tph && cand_smem(Rbox, P.stages, (max_tph + C - 1) / C) > (wide ? kCMaxSmem : kCTwoPerSm)) ++C;
    P.share = (max_tph + C - 1) / C;
    size_t smem = cand_smem(Rbox, P.stages, P.share);
    // Where an SM each is to be had, no two CTAs share one: set up while block_bounds drains, they would sit in pairs on the SMs that are
    // free first, with others left empty (64 heads x 16384 keys, 128 CTAs: 16 SMs had two and 36 none, and the calls took 96 us instead of 94, 184
    // instead of 147 where the scores are nearly equal and all keys are candidates).
    if (s.Hkv * C <= dev.sms && smem <= kCTwoPerSm) smem = kCTwoPerSm + 1024;
    if (smem > kCMaxSmem) return JQ_ERR_CUDA;   // (prune_taken's limit on the length keeps every call below)
    P.L = s.L; P.tph = tph; P.nkeep = s.budget < s.L ? s.budget : s.L;
    P.heads = s.Hkv; P.R = R; P.Rbox = Rbox; P.Rpad = Rpad; P.radius = (s.pool - 1) / 2;
    P.sms = grid; P.hpu = S.hpu;
    // Round 1 should take as many blocks as hold the kept positions.  A peak lifts, within its block, pool - r (r + 1) / 16 positions on
    // average: with fewer blocks than the budget has of those the threshold's bound falls among the positions that are not lifted,
    // and round 2 takes nearly everything (a fifth too few: 32 layers of 32768 keys 600 -> 945 us); more cost next to nothing,
    // they are mostly blocks that round 2 would ask for (half as many again: 596).
    const int r = P.radius < 15 ? P.radius : 15;
    P.first_pct = (int)(130.0 / (2 * r + 1 - r * (r + 1) / 16.0));
    P.T = T; P.c = S.c; P.part = S.part; P.bmax = S.bmax; P.scores = w.scores; P.status = w.status;
    P.Ms = (float *)(scratch + lay.Ms); P.ub = (uint16_t *)(scratch + lay.ub);
    const bool sparse = select_reads_scored_tiles(s, tables ? tables->max_L : s.L);
    ScoredTiles scored;
    scored.bits = P.scored = sparse ? (uint8_t *)(scratch + lay.scored) : nullptr;
    scored.tbase = S.tbase; scored.tph = tph; scored.max_tiles = max_tph; scored.tiles = T;
    P.htab = S.htab; P.tbase = S.tbase; P.qmaps = S.qmaps; P.block_maps = tables ? (const CUtensorMap *)tables->block_maps : nullptr;
    P.n_scores = tables ? tables->total_keys : (long long)s.Hkv * s.L;
#ifdef JQ_DEBUG
    S.dbg_rec = P.dbg_rec = debug_record();
    if (!S.dbg_rec) return JQ_ERR_CUDA;
    S.n_bmax = P.n_bmax = T * 4 * Rpad;
    S.n_part = P.n_part = (long long)(s.Hkv + 256) * kSGroups * R;
#endif
    const int bounds_ctas = bounds_per_sm(wide) * dev.sms;
    if (!launch(wide ? row_stats<true> : row_stats<false>, (unsigned)grid, (unsigned)kSThreads, stats_smem(Rbox, S.stages), st, 0, mapK, mapQ, mapW, S) ||
        !launch(wide ? block_bounds<true> : block_bounds<false>, (unsigned)(T < bounds_ctas ? T : bounds_ctas), (unsigned)kBThreads, (size_t)bounds_smem(wide), st, 0, P) ||
        !launch(wide ? score_candidates<true> : score_candidates<false>, (unsigned)(s.Hkv * C), (unsigned)cand_threads(wide), smem, st, C, mapB, mapQ, P))
        return JQ_ERR_CUDA;
    return launch_select(w.scores, s, idx, nullptr, w, st, K, V, Kout, Vout, tables, src_head_rows, out_head_rows, Vwin ? Kwin : nullptr, Vwin,
                         sparse ? &scored : nullptr);
}

}  // namespace jq
