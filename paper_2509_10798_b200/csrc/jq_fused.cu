// The whole pass for one layer of a short prefix in ONE launch: a thread-block cluster per KV head scores the head's keys,
// selects the kept positions and copies their rows.  (Longer prefixes, and calls over many heads, take the grid-wide
// scoring kernel and the selection kernel; fused_plan has the rule.)
//
// What bounds it: latency.  A head of a few thousand keys is a few microseconds of work for its cluster, and the two
// kernels of the general path spend most of their time on launches, on grid-wide counters in global memory (the merge of
// the row statistics takes two of them) and on the radix select's chain of cluster barriers.  Here nothing but K, Q, V and
// the outputs touches global memory: row statistics and scores are pushed between the CTAs' shared memories (distributed
// shared memory, each exchange one mbarrier per CTA that counts the arrivals), and after the one all-gather of the scores
// every CTA selects on its own copy of the head, redundantly, so that the selection needs no exchange at all.
//
//   warps 0..15   sixteen epilogue warps, four groups of 128 threads, that take the accumulator blocks in turn or, when the
//                 CTA has only one or two, a quarter or a half of their columns each;
//   warp 16       TMA producer: the query rows once, the CTA's key tiles into a ring of stages - resident for both passes
//                 if they all fit, else read a second time (from the L2);
//   warp 17       issues the tcgen05.mma of both passes, S = Q K^T and then S^T = K Q^T, four accumulator slots ahead.
// Pass 1: a thread owns a query row and keeps (reference, sum of exponentials) over its columns; the four groups' pairs
// are combined in shared memory and pushed to every CTA of the cluster, which all derive the same normalisers.
// Pass 2: a thread owns a key; the four groups' partial sums are added in group order and the score is pushed to every CTA.
// Selection: 2048 bins over the range of the pooled keys, the few keys of the
// threshold's bin ranked by comparison, one block-wide scan for the ordered compaction; CTA r then copies the r-th share of
// the kept rows.  (Loops are kept rolled wherever they can be: the code runs once per launch, and what a phase costs is
// mostly the fetching of its instructions.)
//
// The keys may come in two parts, [0, LA) and [LA, LA + LB), in buffers of their own (a cache and the pairs decoded since:
// the pass over the concatenation without making it), and the outputs may be the head of the first buffer: rows only move
// towards lower positions, so the cluster moves them a chunk at a time, reading a chunk completely before writing it.
//
// Measured (B200, back-to-back calls through the Python entry points, two launches -> this one): 2 heads x 2048 keys, 64 query
// rows 24.8 -> 9.8 us; 8 x 4096, 128 rows 30.8 -> 17.8 us; 8 x 8192 34.8 -> 27.0 us; re-eviction of 8 x (1024 + 256) keys, in
// place, 45.6 -> 15.9 us (six strided copies and two launches before).
#include "jq_sm100.cuh"
#include "jq_tmem_ld.cuh"
#include "jq_pool.cuh"
#include "jq_debug.cuh"
#include <cstddef>
#include <cstring>
#include <mutex>

namespace jq {
namespace {

constexpr int kFTile = 128;                         // keys per tile
constexpr int kFWarps = 16;                         // epilogue warps
constexpr int kFT = 32 * kFWarps;                   // threads that take part in the selection
constexpr int kFThreads = kFT + 64;                 // plus the producer and the MMA warp
[[maybe_unused]] constexpr int kFMaxCluster = 16; // (sizes the statistics' extent)
constexpr int kFMaxStages = 6;
constexpr int kFCand = 512;                         // keys of one bin that are ranked by comparison
constexpr int kFMaxL = 12288;                       // what shared memory has room for, and about where the general path overtakes
constexpr int kFRowPad = 8;                         // float2s between the CTAs' statistics: their rows fall into different banks
static_assert(kFMaxL <= 4 * 7 * kFT, "the compaction's masks hold seven quads of a thread, four bits each");
constexpr int kFHalo = 32;                          // >= pool radius, in floats
constexpr uint32_t kFHalf = kFTile * 128;           // one 64-column half of a tile
constexpr uint32_t kFStage = 2 * kFHalf;
constexpr uint32_t kFTmemCols = 512, kFSlots = 4, kFSlotCols = 128;
constexpr uint32_t kFSleep = 32;                    // ns between polls of an epilogue warp: sixteen spinning warps slow the MMA warp down
constexpr int kFBins = 2048;
constexpr size_t kFMaxSmem = 227 * 1024;
constexpr size_t kFMinSmem = 116 * 1024;            // one CTA per SM: two could not both hold all of the tensor memory

struct FCtl {
    uint64_t full[kFMaxStages], empty[kFMaxStages];
    uint64_t q_full, t_full[kFSlots], t_empty[kFSlots];
    uint64_t x_full, s_full;                        // row statistics / scores of all CTAs of the cluster have arrived here
    uint32_t tmem_base;
    int abort_flag;
    int digit, krem, count;                         // find_bin's answer; then the threshold's rank among its equals
    uint32_t tau;
    int ncand;
    int scan[2][kFWarps];
    uint32_t wmin[kFWarps], wmax[kFWarps];
    alignas(16) float Ms[kMaxR];                    // minus the row normalisers
};
constexpr uint32_t kFCtlBytes = 2048;
static_assert(sizeof(FCtl) <= kFCtlBytes && offsetof(FCtl, Ms) % 16 == 0, "control block");

struct FParams {
    int L, LA, LB, tA, tT;      // keys: all, of the first and of the second part; tiles of the first part, of both
    int R, Rbox, Rpad, w;
    int split;                  // 1, 2 or 4: column parts of an accumulator block, each taken by a group of its own
    int nt, stages, resident;   // most tiles a CTA scores in pass 1; stages of the ring; whether they hold all of them
    int wtile;                  // the w window keys are one more tile of pass 1 (of rank 0)
    int nkeep, radius;
    int bulk;                   // every CTA's keys start at a multiple of four: its scores go to the others as one copy each
    int run;                    // kept rows a CTA copies at a time
    uint32_t o_ctl, o_rstat, o_part, o_scores;   // offsets into the dynamic shared memory
    float c;
    int *status;
    const uint4 *KA, *VA, *KB, *VB;     // rows of 16 x 16 bytes
    long long a_rows;           // rows between consecutive heads of the first part
    uint4 *Kout, *Vout;
    long long out_rows;         // rows between consecutive heads of the outputs
    int32_t *idx;               // [Hkv][nkeep]
    const uint4 *KW, *VW;       // window rows that follow the kept ones (or null)
    int inplace;                // the outputs are the first part's own rows
#ifdef JQ_DEBUG
    DebugRecord *dbg_rec;
#endif
};

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t peer_addr(const void *p, uint32_t rank)   // the same place in CTA `rank` of the cluster
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
// Stores into another CTA's shared memory that are counted, in bytes, by a barrier of that CTA: its waiters see them, and
// the sender neither fences nor waits (a store, a release and an arrival took the sender the round trip).
__device__ __forceinline__ void push2(uint32_t to, uint32_t bar, float x, float y)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%2, %3}, [%1];" ::"r"(to), "r"(bar), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void push4(uint32_t to, uint32_t bar, float x, float y, float z, float w)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%2, %3, %4, %5}, [%1];"
                 ::"r"(to), "r"(bar), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ void push1(uint32_t to, uint32_t bar, float x)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %2, [%1];" ::"r"(to), "r"(bar), "f"(x) : "memory");
}
// A copy from this CTA's shared memory into another's, counted by a barrier there (all of it 16-byte aligned).
__device__ __forceinline__ void push_bulk(uint32_t to, const void *from, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(to), "r"(smem_u32(from)), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_cluster(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait for the cluster's arrivals (same limit and same consequence as mbar_wait).
__device__ __noinline__ bool wait_cluster(uint64_t *bar, int *abort_flag, int *status)
{
    const long long t0 = clock64();
    for (;;) {
        for (int i = 0; i < 256; ++i) if (mbar_try_cluster(bar, 0)) return true;
        if (*(volatile int *)abort_flag) return false;
        if (clock64() - t0 > kWaitCycles) {
            *(volatile int *)abort_flag = 1;
            atomicMax(status + kWStatus, (int)JQ_ERR_TIMEOUT);
            return false;
        }
    }
}
__device__ __forceinline__ void group_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kFT) : "memory"); }   // the epilogue warps

// Exclusive scan of one int per epilogue thread; one barrier (the caller alternates between two rows of `sums`).
__device__ __forceinline__ int scan512(int v, int *sums)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
    }
    if (lane == 31) sums[wid] = inc;
    group_sync();
    const int before = __reduce_add_sync(0xffffffffu, lane < wid ? sums[lane & (kFWarps - 1)] : 0);
    return before + inc - v;
}

// The bin of h[kFBins] that holds the krem-th key counted from the top -> ctl: the bin, the rank within it, its population.
__device__ __forceinline__ void find_bin(const uint32_t *h, int krem, FCtl *ctl)
{
    const int hi = kFBins - 4 - 4 * (int)threadIdx.x;         // a thread's four bins, from the top
    const uint4 b = *(const uint4 *)(h + hi);
    const int c[4] = {(int)b.w, (int)b.z, (int)b.y, (int)b.x};
    int above = scan512(c[0] + c[1] + c[2] + c[3], ctl->scan[0]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (above < krem && krem <= above + c[i]) { ctl->digit = hi + 3 - i; ctl->krem = krem - above; ctl->count = c[i]; }
        above += c[i];
    }
    group_sync();
}

// Pooled values of quad q for a radius above 4 (out of line: the loop around it is fetched faster without).  The four windows
// share the positions [4q + 3 - radius, 4q + radius], taken as whole quads and what is left of them on either side; each
// window then has three more of its own.  (The halo is at least as wide as the radius.)
__device__ __noinline__ float4 pool_wide(const float *scores, int q, int radius)
{
    const float4 *s4 = (const float4 *)scores;
    const int from = 4 * q + 3 - radius, to = 4 * q + radius, qa = (from + 3) >> 2, qb = (to + 1) >> 2;
    float4 c = s4[qa];
#pragma unroll 1
    for (int x = qa + 1; x < qb; ++x) {
        const float4 v = s4[x];
        c = make_float4(fmaxf(c.x, v.x), fmaxf(c.y, v.y), fmaxf(c.z, v.z), fmaxf(c.w, v.w));
    }
    float core = fmaxf(max3f(c.x, c.y, c.z), c.w);
    for (int j = from; j < 4 * qa; ++j) core = fmaxf(core, scores[j]);
    for (int j = 4 * qb; j <= to; ++j) core = fmaxf(core, scores[j]);
    const float l2 = fmaxf(scores[from - 2], scores[from - 1]), r1 = scores[to + 1], r2 = fmaxf(r1, scores[to + 2]);
    return make_float4(max3f(core, l2, scores[from - 3]), max3f(core, l2, r1), max3f(core, scores[from - 1], r2), max3f(core, r2, scores[to + 3]));
}

__global__ void __launch_bounds__(kFThreads, 1)
evict_fused(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
            const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapW, const __grid_constant__ FParams P)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *const qbuf = smem_raw;
    const uint32_t q_bytes = (uint32_t)P.Rbox * kD * 2;
    uint8_t *const kbuf = smem_raw + q_bytes;
    FCtl *const ctl = (FCtl *)(smem_raw + P.o_ctl);
    float2 *const rstat = (float2 *)(smem_raw + P.o_rstat);   // [cluster][Rbox + pad]: every CTA's statistics of every row
    float *const part = (float *)(smem_raw + P.o_part);       // pass 1: [4][Rbox] float2; pass 2: [blocks per tile * split][nt * 128]
    float *const scores = (float *)(smem_raw + P.o_scores) + kFHalo;   // [L], with a halo of -inf on either side
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank(), C = cluster_size();
    const int kv = (int)(blockIdx.x / C);
    const int t0 = (int)(rank * (uint32_t)P.tT / C), t1 = (int)((rank + 1) * (uint32_t)P.tT / C), nt = t1 - t0;
    const int nt1 = nt + (P.wtile && rank == 0 ? 1 : 0);      // tiles of pass 1
    // the keys of this CTA's tiles are consecutive: the first one, and how many (the last quad of the head whole)
    auto key_of = [&](int t) { return t < P.tA ? t * kFTile : P.LA + (t - P.tA) * kFTile; };
    const int own_first = key_of(t0), own_keys = ((t1 == P.tT ? P.L : key_of(t1)) - own_first + 3) & ~3;
    const int nblk = P.Rbox / 128, L = P.L, R = P.R, Rpad = P.Rpad;
    const int nrw = (R + 31) / 32;                            // warps that push row statistics
    const int rpitch = P.Rbox + kFRowPad;
    int *const status = P.status;
#ifdef JQ_DEBUG
    DebugRecord *const dbg = P.dbg_rec;
#endif
    if (smem_u32(smem_raw) & 1023u) {   // uniform over the grid
        if (tid == 0) atomicMax(status + kWStatus, (int)JQ_ERR_CUDA);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < kFMaxStages; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        mbar_init(&ctl->q_full, 1);
        for (uint32_t s = 0; s < kFSlots; ++s) { mbar_init(&ctl->t_full[s], 1); mbar_init(&ctl->t_empty[s], 4 * P.split); }
        mbar_init(&ctl->x_full, 1);
        mbar_init(&ctl->s_full, 1);
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // what will be pushed here: a pair for every row from every CTA; every score, in quads where a quad is aligned (the
        // last one of the head whole)
        mbar_expect_tx(&ctl->x_full, C * (uint32_t)nrw * 32u * 8u);
        const int up = (P.LB > 0 ? P.LA + ((P.LA & 3) ? P.LB : (P.LB + 3) & ~3) : (P.LA + 3) & ~3);
        mbar_expect_tx(&ctl->s_full, (uint32_t)(P.bulk ? up - own_keys : up) * 4u);
    }
    if (warp == kFWarps && lane < 4) {   // (they are kernel parameters: nothing that the previous kernel writes)
        const CUtensorMap *m = lane == 0 ? &mapA : lane == 1 ? &mapB : lane == 2 ? &mapQ : &mapW;
        asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
    }
    if (warp == kFWarps + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(kFTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // every CTA of the cluster has its barriers set up before anybody pushes (waited for where pass 1 ends)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    const uint32_t tmem = *(volatile uint32_t *)&ctl->tmem_base;
    cudaGridDependencySynchronize();             // nothing in global memory has been touched so far
    cudaTriggerProgrammaticLaunchCompletion();   // the stream's next kernel may be set up meanwhile; it waits for this one's results

    if (warp == kFWarps) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0) {
            auto load_tile = [&](int i, uint32_t st) {        // i-th tile of this CTA; nt = the window tile
                const int t = t0 + i;
                const bool wt = i == nt, b = t >= P.tA;
                const CUtensorMap *map = wt ? &mapW : b ? &mapB : &mapA;
                const int j0 = wt ? 0 : (b ? t - P.tA : t) * kFTile;
                mbar_expect_tx(&ctl->full[st], kFStage);
                if (JQ_IN(st, P.stages, kDbgFused, 1)) {
                    tma_load_3d(kbuf + (size_t)st * kFStage, map, &ctl->full[st], 0, j0, kv);
                    tma_load_3d(kbuf + (size_t)st * kFStage + kFHalf, map, &ctl->full[st], 64, j0, kv);
                }
            };
            mbar_expect_tx(&ctl->q_full, q_bytes);
            tma_load_3d(qbuf, &mapQ, &ctl->q_full, 0, 0, kv);
            tma_load_3d(qbuf + q_bytes / 2, &mapQ, &ctl->q_full, 64, 0, kv);
            if (P.resident) {
                for (int i = 0; i < nt1; ++i) load_tile(i, (uint32_t)i);
            } else {
                uint32_t st = 0, ph = 0;
                for (int i = 0; i < nt1 + nt; ++i) {
                    if (!mbar_wait(&ctl->empty[st], ph ^ 1, &ctl->abort_flag, status, 64)) break;
                    load_tile(i < nt1 ? i : i - nt1, st);
                    if (++st == (uint32_t)P.stages) { st = 0; ph ^= 1; }
                }
            }
        }
        __syncwarp();
    } else if (warp == kFWarps + 1) {
        // ---------------------------------------------------------------- MMA issuer (all 32 lanes walk the loop)
        const uint32_t idesc1 = instr_desc(128, kFTile);
        const uint32_t idesc2a = instr_desc(kFTile, min(128, Rpad)), idesc2b = instr_desc(kFTile, max(32, Rpad - 128));
        uint32_t st = 0, ph = 0, u = 0;
        bool ok = mbar_wait(&ctl->q_full, 0, &ctl->abort_flag, status, 32);
        const uint32_t q_lo = desc_lo(smem_u32(qbuf));
#pragma unroll 1
        for (int i = 0; i < nt1 + nt && ok; ++i) {
            const bool pass1 = i < nt1;
            if (P.resident) st = (uint32_t)(pass1 ? i : i - nt1);
            if (pass1 || !P.resident) { if (!mbar_wait(&ctl->full[st], ph, &ctl->abort_flag, status, 32)) { ok = false; break; } }
            const uint32_t k_lo = desc_lo(smem_u32(kbuf) + st * kFStage);
#pragma unroll 1
            for (int blk = 0; blk < nblk; ++blk, ++u) {
                const uint32_t slot = u % kFSlots;
                if (!mbar_wait(&ctl->t_empty[slot], ((u / kFSlots) & 1) ^ 1, &ctl->abort_flag, status, 32)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d = tmem + slot * kFSlotCols, qb_lo = q_lo + (uint32_t)blk * (kFHalf >> 4);
                if (!JQ_IN(st, P.stages, kDbgFused, 2)) { ok = false; break; }
                if (pass1) tc_mma_block(d, qb_lo, k_lo, q_bytes / 2, kFHalf, idesc1);
                else tc_mma_block(d, k_lo, qb_lo, kFHalf, q_bytes / 2, blk == 0 ? idesc2a : idesc2b);
                tc_commit(&ctl->t_full[slot]);
            }
            if (!P.resident) {
                if (ok) tc_commit(&ctl->empty[st]);
                if (++st == (uint32_t)P.stages) { st = 0; ph ^= 1; }
            }
        }
    } else {
        // ---------------------------------------------------------------- epilogue warps: both passes
        const int grp = warp >> 2, quarter = warp & 3, row0 = quarter * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
        const float c = P.c, lazy = 64.f / c;
        const float2 cc = make_float2(c, c);
        bool ok = true;
        auto release = [&](uint32_t slot) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->t_empty[slot], 1);
        };
        {   // the halo of -inf around the scores
            const int pad = ((L + 3) & ~3) - L + kFHalo;
            if (tid < kFHalo) scores[tid - kFHalo] = -INFINITY;
            for (int i = tid; i < pad; i += kFT) scores[L + i] = -INFINITY;
        }
        uint32_t va[16], vb[16];
        bool pre = false;                                     // the first read of the next block has been requested
        auto begin = [&](uint32_t uu, uint32_t col) {
            JQ_TMEM_LD16(lane_addr + (uu % kFSlots) * kFSlotCols + col, va);
        };
        auto ready = [&](uint32_t uu) -> bool {               // one look, warp-uniform
            if (!__all_sync(0xffffffffu, mbar_test(&ctl->t_full[uu % kFSlots], (uu / kFSlots) & 1))) return false;
            tc_fence_after();
            return true;
        };
        auto await = [&](uint32_t uu) -> bool {
            if (!mbar_wait(&ctl->t_full[uu % kFSlots], (uu / kFSlots) & 1, &ctl->abort_flag, status, kFSleep)) return false;
            tc_fence_after();
            return true;
        };
        // The groups take the blocks in turn or, when the CTA has fewer than three, parts of their columns: group grp has
        // part `cpart` of the blocks first, first + step, ...
        const int lgS = P.split == 4 ? 2 : P.split >> 1, first = grp >> lgS, step = 4 >> lgS, cpart = grp & (P.split - 1);
        // ---- pass 1.  The next 16 columns, of the same block or of the group's next one if that is complete, are read while
        // the 16 before them are exponentiated.
        const int win_i[2] = {P.wtile ? min(P.w, row0 % P.w + 1) : 0, P.wtile ? min(P.w, (row0 + 128) % P.w + 1) : 0};
        RowState st0 = {-INFINITY, make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, st1 = st0;
        const int n1 = nt1 * nblk, n2 = nt * nblk;
        const int cb = cpart * (kFTile >> lgS), ce = cb + (kFTile >> lgS);
#pragma unroll 1
        for (int u = first; u < n1; u += step) {
            const int i = u >> (nblk - 1), blk = u & (nblk - 1), t = t0 + i;
            if (!pre) {
                if (!await(u)) { ok = false; break; }
                begin(u, cb);
            }
            // keys of the tile that count for this thread's row: those of the prefix, or, in the window tile, the
            // window keys up to the row's own position (causal)
            const int valid = i == nt ? (blk ? win_i[1] : win_i[0])
                                      : t < P.tA ? min(kFTile, P.LA - t * kFTile) : min(kFTile, P.LB - (t - P.tA) * kFTile);
            const uint32_t taddr = lane_addr + ((uint32_t)u % kFSlots) * kFSlotCols;
            if (blk == 1) { const RowState x = st0; st0 = st1; st1 = x; }
#pragma unroll 1
            for (int c0 = cb; c0 < ce; c0 += 32) {
                JQ_TMEM_WAIT16(va);
                JQ_TMEM_LD16(taddr + c0 + 16, vb);
                if (valid > c0) p1_half(va, c0, valid, c, lazy, cc, st0);   // (a read without any key has no reference)
                JQ_TMEM_WAIT16(vb);
                if (c0 + 32 < ce) JQ_TMEM_LD16(taddr + c0 + 32, va);
                else {
                    release((uint32_t)u % kFSlots);
                    pre = u + step < n1 && ready(u + step);
                    if (pre) begin(u + step, cb);
                }
                if (valid > c0 + 16) p1_half(vb, c0 + 16, valid, c, lazy, cc, st0);
            }
            if (blk == 1) { const RowState x = st0; st0 = st1; st1 = x; }
        }
        float2 *const gstat = (float2 *)part;
        gstat[grp * P.Rbox + row0] = make_float2(st0.m, (st0.l01.x + st0.l01.y) + (st0.l23.x + st0.l23.y));
        if (nblk == 2) gstat[grp * P.Rbox + 128 + row0] = make_float2(st1.m, (st1.l01.x + st1.l01.y) + (st1.l23.x + st1.l23.y));
        group_sync();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        {   // the groups' pairs of a row are combined by 4 (or 2) threads, each of which pushes the result to its share of the CTAs
            const int lgR = nblk == 1 ? 7 : 8, nsub = kFT >> lgR, row = tid & (P.Rbox - 1), sub = tid >> lgR;
            if ((row >> 5) < nrw) {
                float2 p[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) p[q] = gstat[q * P.Rbox + row];
                float m = -INFINITY, l = 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q) if (p[q].y > 0.f) m = fmaxf(m, p[q].x);
#pragma unroll
                for (int q = 0; q < 4; ++q) if (p[q].y > 0.f) l = fmaf(p[q].y, ex2(c * (p[q].x - m)), l);
                if (JQ_IN(rank * rpitch + row, kFMaxCluster * (kMaxR + kFRowPad), kDbgFused, 3))
#pragma unroll 1
                    for (int d = sub; d < (int)C; d += nsub)
                        push2(peer_addr(rstat + rank * rpitch + row, d), peer_addr(&ctl->x_full, d), m, l);
            }
        }
        ok = wait_cluster(&ctl->x_full, &ctl->abort_flag, status) && ok;
        {   // the row's normaliser from the CTAs' pairs, by 4 (or 2) neighbouring lanes, in an order that all CTAs share
            const int lgN = nblk == 1 ? 2 : 1, nsub = 1 << lgN, row = tid >> lgN, sub = tid & (nsub - 1);
            float m = -INFINITY, l = 0.f;
#pragma unroll 1
            for (int d = sub; d < (int)C; d += nsub) { const float2 p = rstat[d * rpitch + row]; if (row < R && p.y > 0.f) m = fmaxf(m, p.x); }
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
            if (nsub == 4) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
#pragma unroll 1
            for (int d = sub; d < (int)C; d += nsub) { const float2 p = rstat[d * rpitch + row]; if (row < R && p.y > 0.f) l = fmaf(p.y, ex2(c * (p.x - m)), l); }
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            if (nsub == 4) l += __shfl_xor_sync(0xffffffffu, l, 2);
            if (sub == 0) ctl->Ms[row] = row < R ? -fmaf(c, m, log2f(l)) : -INFINITY;   // -inf silences a column that is not a query row
        }
        group_sync();
        // ---- pass 2, the same way: part `cpart` of a block's 32-column pieces
        pre = false;
        auto pieces = [&](int v) { return (nblk == 1 || (v & 1) == 0 ? min(128, Rpad) : Rpad - 128) >> 5; };
#pragma unroll 1
        for (int v = first; v < n2 && ok; v += step) {
            const int u = n1 + v, i = v >> (nblk - 1), blk = v & (nblk - 1), np = pieces(v);
            const int pb = cpart * np >> lgS, pe = (cpart + 1) * np >> lgS;
            if (!pre) {
                if (!await(u)) { ok = false; break; }
                begin(u, 32 * pb);
            }
            const uint32_t taddr = lane_addr + ((uint32_t)u % kFSlots) * kFSlotCols;
            const float4 *bias = (const float4 *)(ctl->Ms + 128 * blk);
            float2 a01 = make_float2(0.f, 0.f), a23 = a01;
            if (pb == pe) {                                   // no column of this block is this group's
                release((uint32_t)u % kFSlots);
                pre = false;
            }
#pragma unroll 1
            for (int p = pb; p < pe; ++p) {
                JQ_TMEM_WAIT16(va);
                JQ_TMEM_LD16(taddr + 32 * p + 16, vb);
                exp_acc16(a01, a23, va, cc, bias + 8 * p);
                JQ_TMEM_WAIT16(vb);
                if (p + 1 < pe) JQ_TMEM_LD16(taddr + 32 * p + 32, va);
                else {
                    release((uint32_t)u % kFSlots);
                    pre = v + step < n2 && ready(u + step);
                    if (pre) begin(u + step, 32 * (cpart * pieces(v + step) >> lgS));
                }
                exp_acc16(a01, a23, vb, cc, bias + 8 * p + 4);
            }
            const int at = ((blk * P.split + cpart) * P.nt + i) * kFTile + row0;
            if (JQ_IN(at, nblk * P.split * P.nt * kFTile, kDbgFused, 4)) part[at] = (a01.x + a01.y) + (a23.x + a23.y);
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        group_sync();
        // ---- the scores of this CTA's keys go to every CTA of the cluster: into this CTA's array first and from there as one copy to
        // each of the others or, where the keys' places do not allow that, four at a time, two threads to a quad's targets.
        // (One by one a CTA of ten that has ten tiles sends 3200 stores of 16 bytes: 8 heads x 11999 keys 33.6 -> 32.9 us.)
        const int share = P.bulk ? 0 : 1;
#pragma unroll 1
        for (int i = 4 * (tid >> share); i < nt * kFTile; i += 4 * (kFT >> share)) {
            const int t = t0 + i / kFTile, r = i & (kFTile - 1), ps = P.nt * kFTile;
            const bool b = t >= P.tA;
            const int j = (b ? t - P.tA : t) * kFTile + r, key = b ? P.LA + j : j, have = min(4, (b ? P.LB : P.LA) - j);
            if (have <= 0 || !JQ_IN(key + have - 1, L, kDbgFused, 5)) continue;
            float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
            for (int x = 0; x < nblk * P.split; ++x) {
                const float4 p = *(const float4 *)(part + x * ps + i);
                s[0] += p.x; s[1] += p.y; s[2] += p.z; s[3] += p.w;
            }
            const bool whole = (key & 3) == 0 && (have == 4 || (key + have == L && (b || P.LB == 0)));   // (the last quad's missing positions are -inf anyway)
#pragma unroll
            for (int e = 1; e < 4; ++e) if (e >= have) s[e] = -INFINITY;
            if (P.bulk) {
                *(float4 *)(scores + key) = make_float4(s[0], s[1], s[2], s[3]);
                continue;
            }
#pragma unroll 1
            for (int d = tid & 1; d < (int)C; d += 2) {
                const uint32_t to = peer_addr(scores + key, (uint32_t)d), bar = peer_addr(&ctl->s_full, (uint32_t)d);
                if (whole) push4(to, bar, s[0], s[1], s[2], s[3]);
                else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) if (e < have) push1(to + 4 * e, bar, s[e]);
                }
            }
        }
        if (P.bulk) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the copies read what has just been stored
            group_sync();
            if (warp == 0 && lane < (int)C && lane != (int)rank && own_keys > 0)
                push_bulk(peer_addr(scores + own_first, (uint32_t)lane), scores + own_first, (uint32_t)own_keys * 4u, peer_addr(&ctl->s_full, (uint32_t)lane));
        }
    }
    if (warp >= kFWarps) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // (the epilogue warps waited before they pushed)

    // Queries and stages are free once pass 2 is through (every product has been read); the selection takes their place.
    uint32_t *const hist = (uint32_t *)smem_raw;
    uint32_t *const cand = hist + kFBins;
    int *const list = (int *)(cand + kFCand);                 // the kept positions, ascending
    uint32_t *const keys = (uint32_t *)(list + ((P.nkeep + 3) & ~3));
    if (warp < kFWarps) {
        // ---------------------------------------------------------------- selection, on this CTA's copy of the scores
        for (int i = tid; i < kFBins / 4; i += kFT) ((uint4 *)hist)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (tid == 0) ctl->ncand = 0;
        wait_cluster(&ctl->s_full, &ctl->abort_flag, status);
    }
    // nobody pushes to this CTA any more and this CTA pushes to nobody: once all have got here, any may leave (nothing is
    // handed over, so the arrival need not be a release, which would wait for this CTA's stores)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    if (warp < kFWarps && P.nkeep >= L) {
        for (int t = tid; t < P.nkeep; t += kFT) list[t] = t;
        group_sync();
    } else if (warp < kFWarps) {
        // A thread owns NQ consecutive quads: the max-pool's plateaus then mostly fall within a thread, which adds them to the
        // histogram as one count, and thread order is position order.  NQ is odd: 16-byte reads at a stride of an odd number
        // of quads meet no bank conflicts.
        const int nq = (L + 3) / 4, NQ = ((nq + kFT - 1) / kFT) | 1, q0 = min(tid * NQ, nq), q1 = min(q0 + NQ, nq);
        const float4 *s4 = (const float4 *)scores;
        uint4 *k4 = (uint4 *)keys;
        // pooled keys of the thread's positions, and the range of all of them
        uint32_t kmin = 0xffffffffu, kmax = 0u;
        float4 a = s4[q0 - 1], b = s4[q0];
#pragma unroll 1
        for (int q = q0; q < q1; ++q) {
            uint32_t k[4];
            float best[4];
            if (!JQ_IN(4 * q + 3, (L + 3) & ~3, kDbgFused, 7)) continue;
            if (P.radius <= 4) {
                const float4 nx = s4[q + 1];
                pooled_quad(a, b, nx, P.radius, k, best);
                a = b; b = nx;
            } else {
                const float4 w = pool_wide(scores, q, P.radius);
                best[0] = w.x; best[1] = w.y; best[2] = w.z; best[3] = w.w;
#pragma unroll
                for (int e = 0; e < 4; ++e) k[e] = order_key(best[e]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (4 * q + e >= L) k[e] = 0u;                            // below every score's key
                else { kmin = min(kmin, k[e]); kmax = max(kmax, k[e]); }
            }
            k4[q] = make_uint4(k[0], k[1], k[2], k[3]);
        }
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        if (lane == 0) { ctl->wmin[warp] = kmin; ctl->wmax[warp] = kmax; }
        group_sync();
        kmin = __reduce_min_sync(0xffffffffu, ctl->wmin[lane & (kFWarps - 1)]);
        kmax = __reduce_max_sync(0xffffffffu, ctl->wmax[lane & (kFWarps - 1)]);
        // The threshold key: 2048 equal bins over the keys' own range (a score's leading bits alone would put most keys of
        // a flat head into a few bins), then the bin's few keys ranked by comparison - or binned again while they are many.
        uint32_t lo = kmin, lim = kmax - kmin, tau;
        int need_eq = P.nkeep;                                            // rank of the threshold among the keys in [lo, lo + lim]
#pragma unroll 1
        for (;;) {
            const int sh = lim >> 11 ? 21 - __clz(lim) : 0;               // lim >> sh < 2048
            uint32_t cur = 0u, cnt = 0u;
#pragma unroll 1
            for (int q = q0; q < q1; ++q) {
                const uint4 kk = k4[q];
                const uint32_t k[4] = {kk.x - lo, kk.y - lo, kk.z - lo, kk.w - lo};
#pragma unroll
                for (int e = 0; e < 4; ++e) {                             // neighbours often share the bin: runs as one count
                    const bool in = k[e] <= lim, other = in && k[e] >> sh != cur;
                    if (other && cnt && JQ_IN(cur, kFBins, kDbgFused, 6)) atomicAdd(&hist[cur], cnt);
                    cnt = other ? 1u : cnt + in;
                    cur = other ? k[e] >> sh : cur;
                }
            }
            if (cnt && JQ_IN(cur, kFBins, kDbgFused, 6)) atomicAdd(&hist[cur], cnt);
            group_sync();
            find_bin(hist, need_eq, ctl);
            lo += (uint32_t)ctl->digit << sh;
            need_eq = ctl->krem;
            const int count = ctl->count;
            if (sh == 0) { tau = lo; break; }
            lim = (1u << sh) - 1u;
            if (count <= kFCand) {
#pragma unroll 1
                for (int q = q0; q < q1; ++q) {
                    const uint4 kk = k4[q];
                    const uint32_t k[4] = {kk.x, kk.y, kk.z, kk.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (k[e] - lo <= lim) {
                            const int at = atomicAdd(&ctl->ncand, 1);
                            if (JQ_IN(at, kFCand, kDbgFused, 12)) cand[at] = k[e];
                        }
                }
                group_sync();
                if (tid < count) {
                    const uint32_t k = cand[tid];
                    int gt = 0, eq = 0;
#pragma unroll 4
                    for (int i = 0; i < count; ++i) { const uint32_t x = cand[i]; gt += x > k; eq += x == k; }
                    if (gt < need_eq && need_eq <= gt + eq) { ctl->tau = k; ctl->krem = need_eq - gt; }   // (equal keys write the same)
                }
                group_sync();
                tau = ctl->tau;
                need_eq = ctl->krem;
                break;
            }
            for (int i = tid; i < kFBins / 4; i += kFT) ((uint4 *)hist)[i] = make_uint4(0u, 0u, 0u, 0u);
            group_sync();
        }
        // ---- ordered compaction: need_eq of the keys == tau are kept, the lowest positions.  (After a wait that ran out, scores
        // and counts may be anything, copies in flight may land on them, and the warps may learn of it at different times: the
        // selection then runs to its end like any other, within its arrays whatever it reads - a thread's first place in the
        // list is brought into range, and its at most 28 entries from there reach at most into the keys, which have been
        // read - and no row is copied.)
        uint32_t gtm = 0u, eqm = 0u;                                      // bit 4 i + e: position e of the thread's i-th quad
#pragma unroll 1
        for (int q = q0, i = 0; q < q1; ++q, i += 4) {
            const uint4 kk = k4[q];
            gtm |= ((kk.x > tau) | (kk.y > tau) << 1 | (kk.z > tau) << 2 | (kk.w > tau) << 3) << i;
            eqm |= ((kk.x == tau) | (kk.y == tau) << 1 | (kk.z == tau) << 2 | (kk.w == tau) << 3) << i;
        }
        const int before = scan512(__popc(gtm) | __popc(eqm) << 16, ctl->scan[1]);   // (at most 12288 positions: 14 bits each)
        const int eb = before >> 16, room = max(need_eq - eb, 0);
        int t = min(max((before & 0xffff) + min(eb, need_eq), 0), P.nkeep), j = 4 * q0;
        while (__popc(eqm) > room) eqm ^= 0x80000000u >> __clz(eqm);
#pragma unroll 1
        for (uint32_t m = gtm | eqm; m; m >>= 1, ++j)
            if (m & 1u) { if (JQ_IN(t, P.nkeep, kDbgFused, 13)) list[t] = j; ++t; }
        group_sync();
    }

    // The kept rows are dealt out to the CTAs in runs of S rows: run x belongs to CTA x % C.
    const int S = P.run, steps = (P.nkeep + S * (int)C - 1) / (S * (int)C);
    // ---------------------------------------------------------------- the kept rows (256 bytes: 16 lanes x 16 bytes)
    const bool work = warp < kFWarps && !*(volatile int *)&ctl->abort_flag;
    const int lane16 = tid & 15, rg = tid >> 4;
    constexpr int ng = kFT / 16;
    const long long arow = (long long)kv * P.a_rows, brow = (long long)kv * P.LB, orow = (long long)kv * P.out_rows;
    if (!P.inplace) {
        if (work) {
            const int t0r = (int)rank * S, n = min(S, P.nkeep - t0r);    // one run per CTA
            for (int i = rg; i < n; i += 4 * ng) {
                uint4 a[4], b[4];
                int j[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) j[x] = i + x * ng < n ? min(max(list[t0r + i + x * ng], 0), L - 1) : 0;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const bool in = i + x * ng < n, sb = j[x] >= P.LA;
                    const size_t src = (size_t)(sb ? brow + (j[x] - P.LA) : arow + j[x]) * 16 + lane16;
                    a[x] = in ? (sb ? P.KB : P.KA)[src] : make_uint4(0u, 0u, 0u, 0u);
                    b[x] = in ? (sb ? P.VB : P.VA)[src] : make_uint4(0u, 0u, 0u, 0u);
                }
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int t = t0r + i + x * ng;
                    const size_t dst = (size_t)(orow + t) * 16 + lane16;
                    if (i + x * ng < n && JQ_IN(t, P.out_rows, kDbgFused, 8)) {
                        P.Kout[dst] = a[x]; P.Vout[dst] = b[x];
                        if (lane16 == 0) P.idx[(size_t)kv * P.nkeep + t] = j[x];
                    }
                }
            }
            if (P.KW)                      // the window rows behind them
                for (int i = (int)rank * ng + rg; i < P.w; i += (int)C * ng) {
                    const size_t src = ((size_t)kv * P.w + i) * 16 + lane16, dst = (size_t)(orow + P.nkeep + i) * 16 + lane16;
                    if (JQ_IN(P.nkeep + i, P.out_rows, kDbgFused, 9)) { P.Kout[dst] = P.KW[src]; P.Vout[dst] = P.VW[src]; }
                }
        }
    } else {
        // Kept row t comes from position list[t] >= t: a step of one run per CTA reads all its rows before the cluster
        // writes any of them, and what it writes lies below everything that later steps read.
        uint4 *const stage = (uint4 *)keys;                   // [S][2][16] (the keys have served)
#pragma unroll 1
        for (int st = 0; st < steps; ++st) {
            const int t0r = (st * (int)C + (int)rank) * S, n = min(S, P.nkeep - t0r);
            if (work)
                for (int i = rg; i < n; i += 4 * ng) {         // four rows in flight per 16 lanes
                    uint4 a[4], b[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int r = i + x * ng, j = r < n ? min(max(list[t0r + i + x * ng], 0), L - 1) : 0;
                        const bool sb = j >= P.LA, moves = r < n && (j != t0r + r || sb);   // (a row of the first part that keeps its place is there already)
                        const size_t src = (size_t)(sb ? brow + (j - P.LA) : arow + j) * 16 + lane16;
                        a[x] = moves ? (sb ? P.KB : P.KA)[src] : make_uint4(0u, 0u, 0u, 0u);
                        b[x] = moves ? (sb ? P.VB : P.VA)[src] : make_uint4(0u, 0u, 0u, 0u);
                        if (r < n && lane16 == 0) P.idx[(size_t)kv * P.nkeep + t0r + r] = j;
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int r = i + x * ng;
                        if (r < n && JQ_IN(r, S, kDbgFused, 10)) { stage[(2 * r) * 16 + lane16] = a[x]; stage[(2 * r + 1) * 16 + lane16] = b[x]; }
                    }
                }
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // (of the arrival before the selection)
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // (waited for by the next step, or at the exit)
            if (work)
                for (int i = rg; i < n; i += ng) {
                    const size_t dst = (size_t)(orow + t0r + i) * 16 + lane16;
                    if ((list[t0r + i] != t0r + i || t0r + i >= P.LA) && JQ_IN(t0r + i, P.out_rows, kDbgFused, 11)) { P.Kout[dst] = stage[(2 * i) * 16 + lane16]; P.Vout[dst] = stage[(2 * i + 1) * 16 + lane16]; }
                }
        }
    }
    // ---------------------------------------------------------------- exit
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    bool gave_up = false;
    if (warp == kFWarps + 1) gave_up = *(volatile int *)&ctl->abort_flag != 0;   // (there is nothing left to wait for)
    tc_fence_before();
    __syncthreads();
    if (warp == kFWarps + 1) {
        if (gave_up) __nanosleep(200000);        // let copies, pushes and products still in flight land before the CTA goes
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kFTmemCols) : "memory");
    }
}

// ------------------------------------------------------------------ host side

struct FusedDevice { int resident[kFMaxCluster + 1] = {}; bool ready = false; };   // [C]: clusters of C CTAs that fit at a time

bool fused_device(FusedDevice *out)
{
    static FusedDevice devs[64];
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lock(mu);
    FusedDevice &d = devs[dev];
    if (!d.ready) {
        if (cudaFuncSetAttribute(evict_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFMaxSmem) != cudaSuccess) return false;
        if (cudaFuncSetAttribute(evict_fused, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
        for (int C = 1; C <= kFMaxCluster; ++C) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)C);
            cfg.blockDim = dim3(kFThreads);
            cfg.dynamicSmemBytes = kFMaxSmem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&d.resident[C], evict_fused, &cfg) != cudaSuccess) { cudaGetLastError(); d.resident[C] = 0; }
        }
        d.ready = true;
    }
    *out = d;
    return true;
}

// Shared memory of a CTA that scores `nt` tiles of a head of L keys in a cluster of C; fills in the layout.  False if it
// does not fit (the ring needs two stages).
bool fused_layout(int L, int nkeep, int C, int nt, FParams *P, size_t *smem)
{
    const size_t q = (size_t)P->Rbox * kD * 2, rstat = (size_t)C * (P->Rbox + kFRowPad) * 8;
    const int nblk = P->Rbox / 128;
    P->split = nt * nblk == 1 ? 4 : nt * nblk == 2 ? 2 : 1;
    const size_t psum = (size_t)nblk * P->split * nt * kFTile * 4, pstat = (size_t)4 * P->Rbox * 8, part = psum > pstat ? psum : pstat;
    const size_t sc = (size_t)(((L + 3) & ~3) + 2 * kFHalo) * 4;
    const size_t fixed = q + kFCtlBytes + align_up(rstat, 128) + align_up(part, 128) + align_up(sc, 128);
    int stages = fixed < kFMaxSmem ? (int)((kFMaxSmem - fixed) / kFStage) : 0;
    if (stages > kFMaxStages) stages = kFMaxStages;
    P->resident = nt <= stages;
    if (P->resident) stages = nt;
    else if (stages < 2) return false;
    // the selection's histogram, position list, keys and (in place, after them) staged rows take the place of queries and stages
    const size_t per = (size_t)((nkeep + C - 1) / C);
    size_t alias = q + (size_t)stages * kFStage;
    const size_t need = (size_t)(kFBins + kFCand) * 4 + align_up((size_t)nkeep * 4, 16), keys = (size_t)((L + 3) & ~3) * 4;
    if (alias < need + keys || (P->inplace && alias < need + 64 * 512)) return false;
    P->run = (int)per;
    if (P->inplace && per * 512 > alias - need) {
        // more memory for the staged rows, if there is some, so that all rows move in one step (a step is two barriers of the cluster
        // and a round trip to memory: 8 x (1024 + 256) keys 16.0 -> 15.0 us, 103 rows per CTA where 100 fitted)
        const size_t more = align_up(need + per * 512 - alias, 1024);
        if (fixed - q + alias + more <= kFMaxSmem) alias += more;
        else P->run = (int)((alias - need) / 512);
    }
    P->nt = nt;
    P->stages = stages;
    size_t off = alias;
    P->o_ctl = (uint32_t)off; off += kFCtlBytes;
    P->o_rstat = (uint32_t)off; off += align_up(rstat, 128);
    P->o_part = (uint32_t)off; off += align_up(part, 128);
    P->o_scores = (uint32_t)off; off += align_up(sc, 128);
    *smem = off > kFMinSmem ? off : kFMinSmem;
    return true;
}

}  // namespace

// Whether this kernel takes the call, and with which cluster size (0: no): the cheaper of the two ways by what was measured
// (us per call, back to back).  This kernel: a chain of exchanges, the tiles of a CTA one after the other, and the selection,
// which every CTA runs over the whole head; clusters that do not fit at a time take turns (of 16 CTAs 7 fit, of 10 11).
// 8 heads x 1024, 2048, 4096, 8192, 12000 keys in clusters of 8: 10.1, 11.9, 17.9, 29.4, 38.1; of 10: -, 12.3, 17.9, 27.2,
// 34.7; of 4: 11.4, 14.8, 24.4, 40.1, 54.3; with 256 rows 4096 and 8192 keys 24.9, 40.6; 24.9, 37.3; 35.2, 62.0.  A window
// wider than 9 adds 0.5 us per 1000 keys: 8 x 4096, 8192, 12000 keys, pool 63: 20.4, 31.3, 39.7.
// The two kernels of the general path: launches and merge, the tiles of all SMs (past about ten each the next group of heads
// hides the merge), a little per head and per 1000 keys of a head for the selection, and a step at 128 heads, where the other
// selection kernel takes over.  32, 64, 128, 256 heads x 3000 keys: 37.0, 49.3, 88.4, 136.8 (this kernel 23.7, 36.6, 63.7,
// 128.1); x 8192 51.3, 80.7, 150.2, 269.1 (43.5, 72.6, 135.5, 269.3); x 12000 60.9, 102, 204 (58.3, 98.6, 188); with 256 rows
// x 8192 65.8, 110, 214, 400 (65.5, 116, 236, 489).  160 x 3000: 105 (112), 512 x 1000: 156 (111).  Over 412 calls of 1 to 512
// heads, 100 to 12000 keys, 8 to 256 rows the rule's choice takes 0.2 % longer than the better one, at most 9 %.
static int fused_plan(const jq_shape &s, const FusedSource &src, int nkeep, FParams *P, size_t *smem)
{
    FusedDevice dev;
    if (s.L > kFMaxL || !fused_device(&dev)) return 0;
    const int TT = (src.LA + kFTile - 1) / kFTile + (src.LB + kFTile - 1) / kFTile, win = src.Kwin ? 1 : 0;
    const bool wide = P->Rbox == 256;
    const double chain = wide ? 9.3 : 7.4, per_tile = wide ? 2.6 : 1.0 + 0.4 * P->Rpad / 128;
    int best = 0;
    double best_cost = 1e30;
    for (int C = 1; C <= kFMaxCluster && C <= TT; ++C) {
        if (dev.resident[C] < 1) continue;
        const int up = (TT + C - 1) / C, first = TT / C + win, nt = up > first ? up : first;   // (rank 0 has the window tile)
        FParams T = *P;
        size_t sm;
        if (!fused_layout(s.L, nkeep, C, nt, &T, &sm)) continue;
        const double per_key = (C > 8 ? 1.04e-3 : 1.24e-3) + (s.pool > 9 ? 0.5e-3 : 0.0);
        const double cost = (double)((s.Hkv + dev.resident[C] - 1) / dev.resident[C]) * (chain + per_tile * nt + per_key * s.L);
        if (cost < best_cost) { best_cost = cost; best = C; *P = T; *smem = sm; }
    }
    // (the general path appends and moves back with strided copies, two of each, about 4.5 us a piece)
    const double tiles = (double)s.Hkv * (TT + win), first = tiles < 1500.0 ? tiles : 1500.0, rest = tiles - first;
    const double other = (wide ? 23.5 + 0.02 * first + 0.014 * rest + 0.06 * s.Hkv
                               : 22.5 + (0.0115 * first + 0.0095 * rest) * (0.87 + 0.13 * P->Rpad / 128) + 0.04 * s.Hkv) +
                         (s.Hkv >= 128 ? 8.0 : 0.0) + 0.25e-3 * s.L + (src.LB > 0 ? 9.0 : 0.0) + (src.inplace ? 9.0 : 0.0);
    return best_cost <= other ? best : 0;
}

jq_status launch_fused(const jq_shape &s, const FusedSource &src, const void *Q, void *Kout, void *Vout, int out_head_rows,
                       int32_t *idx, const Workspace &w, cudaStream_t st, bool *taken)
{
    *taken = false;
    FParams P = {};
    const int R = s.group * s.w, nkeep = s.budget < s.L ? s.budget : s.L;
    P.R = R; P.Rbox = R <= 128 ? 128 : 256; P.Rpad = (R + 31) & ~31; P.w = s.w;
    P.inplace = src.inplace ? 1 : 0;
    size_t smem = 0;
    const int C = fused_plan(s, src, nkeep, &P, &smem);
    if (!C) return JQ_OK;
    P.L = s.L; P.LA = src.LA; P.LB = src.LB;
    P.tA = (src.LA + kFTile - 1) / kFTile; P.tT = P.tA + (src.LB + kFTile - 1) / kFTile;
    P.wtile = src.Kwin ? 1 : 0;
    P.nkeep = nkeep; P.radius = (s.pool - 1) / 2;
    // (a copy is set up behind a fence and a barrier: with one tile per CTA the stores are 0.2 us faster, with ten the copies 0.6)
    P.bulk = P.nt >= 6 && (src.LB == 0 || (src.LA & 3) == 0);
    P.c = 1.4426950408889634f / sqrtf((float)s.d);
    P.status = w.status;
    P.a_rows = src.a_rows > src.LA ? src.a_rows : src.LA;
    P.KA = (const uint4 *)src.KA; P.VA = (const uint4 *)src.VA; P.KB = (const uint4 *)src.KB; P.VB = (const uint4 *)src.VB;
    P.Kout = (uint4 *)Kout; P.Vout = (uint4 *)Vout; P.idx = idx;
    P.out_rows = out_head_rows > nkeep ? out_head_rows : nkeep;
    P.KW = (const uint4 *)(src.Vwin ? src.Kwin : nullptr); P.VW = (const uint4 *)src.Vwin;
    CUtensorMap mapA, mapB, mapQ, mapW;
    if (!make_tensor_map(&mapQ, Q, R, s.Hkv, P.Rbox)) return JQ_ERR_CUDA;
    mapA = mapB = mapW = mapQ;
    if (src.LA > 0 && !make_tensor_map(&mapA, src.KA, src.LA, s.Hkv, kFTile, (int)P.a_rows)) return JQ_ERR_CUDA;
    if (src.LB > 0 && !make_tensor_map(&mapB, src.KB, src.LB, s.Hkv, kFTile)) return JQ_ERR_CUDA;
    if (src.Kwin && !make_tensor_map(&mapW, src.Kwin, s.w, s.Hkv, kFTile)) return JQ_ERR_CUDA;
#ifdef JQ_DEBUG
    P.dbg_rec = debug_record();
    if (!P.dbg_rec) return JQ_ERR_CUDA;
#endif
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(s.Hkv * C));
    cfg.blockDim = dim3(kFThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, evict_fused, mapA, mapB, mapQ, mapW, P) != cudaSuccess) {
        cudaGetLastError();
        return JQ_ERR_CUDA;
    }
    *taken = true;
    count_launch(1);
    return check_launch();
}

}  // namespace jq
