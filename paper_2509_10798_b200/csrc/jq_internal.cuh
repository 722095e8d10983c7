// Internal declarations shared by the translation units of libjq (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "jq.h"

namespace jq {

constexpr int kD = 128;          // head dimension the kernels are built for
constexpr int kMaxR = 256;       // query rows per KV head (group * w)
constexpr int kSlots = 640;      // partial (reference, sum-exp) slots per KV head in the workspace (up to 4 per CTA)
constexpr int kStatusWords = 64; // first 256 bytes of the workspace

// Device status word values (sticky since jq_workspace_init): 0 ok, else a jq_status.
struct Workspace {
    int *status;        // [kStatusWords]
    float *Mrow;        // [Hkv][R]   log2-domain normaliser per query row: c*max + log2(sumexp)
    float2 *part;       // [Hkv][kSlots][R]   (raw max, sum of exp2(c*(s-max))) per contributing block
    float *scores;      // [Hkv][L]   pre-pool scores (of the two-launch path)
    uint32_t *keys;     // [Hkv][L]   order-preserving bit patterns of the pooled scores (of heads whose keys do not fit on chip)
    void *prune;        // scratch of the one-pass eviction, in the place of Mrow and part (carve_pruned; null otherwise)
    size_t bytes;       // total
};
// Bytes of that scratch for `tiles` tiles of keys in total (every head's rounded up, window tiles included).
size_t prune_bytes(long long tiles, int heads, int R);

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Carve-up of a workspace for `heads` KV heads with R query rows each and `keys` prefix positions in total
// (heads x L for one shape; the sum over the units of a ragged call).
static inline Workspace carve(void *base, size_t heads, size_t R, size_t keys)
{
    Workspace w;
    char *p = (char *)base;
    size_t off = 0;
    w.status = (int *)(p + off);
    off += align_up(kStatusWords * sizeof(int), 256);
    w.prune = nullptr;
    w.Mrow = (float *)(p + off);
    off += align_up(heads * R * sizeof(float), 256);
    w.part = (float2 *)(p + off);
    off += align_up(heads * kSlots * R * sizeof(float2), 256);
    w.scores = (float *)(p + off);
    off += align_up(keys * sizeof(float), 256);
    w.keys = (uint32_t *)(p + off);
    off += align_up(keys * sizeof(uint32_t), 256);
    w.bytes = off;
    return w;
}
static inline Workspace carve(void *base, const jq_shape &s)
{
    return carve(base, (size_t)s.Hkv, (size_t)s.group * s.w, (size_t)s.Hkv * s.L);
}
// The same for a call that takes the one-pass eviction.  Its scratch can be larger: a workspace that has room for carve() only is as
// good as any, the call then goes the other way.
static inline Workspace carve_pruned(void *base, size_t heads, size_t R, size_t keys)
{
    Workspace w = {};
    char *p = (char *)base;
    size_t off = 0;
    w.status = (int *)(p + off);
    off += align_up(kStatusWords * sizeof(int), 256);
    w.prune = p + off;
    off += prune_bytes((long long)(keys / 128 + 2 * heads), (int)heads, (int)R);
    w.scores = (float *)(p + off);
    off += align_up(keys * sizeof(float), 256);
    w.keys = (uint32_t *)(p + off);
    off += align_up(keys * sizeof(uint32_t), 256);
    w.bytes = off;
    return w;
}
// Bytes of a workspace with which a call over `heads` heads can go either way, whatever its budget.
bool prune_possible(int heads, int R, long long keys, int max_L);
// (tables, prune_tables: bytes of the tables behind it, either way)
static inline size_t workspace_need(size_t heads, size_t R, size_t keys, int max_L, size_t tables = 0, size_t prune_tables = 0)
{
    const size_t a = carve(nullptr, heads, R, keys).bytes + tables;
    const size_t b = prune_possible((int)heads, (int)R, (long long)keys, max_L) ? carve_pruned(nullptr, heads, R, keys).bytes + prune_tables : 0;
    return a > b ? a : b;
}
static inline size_t workspace_need(const jq_shape &s) { return workspace_need((size_t)s.Hkv, (size_t)s.group * s.w, (size_t)s.Hkv * s.L, s.L); }

// Units (layers, sequences) of one head geometry living in buffers of their own, with prefix lengths and
// budgets of their own (jq_evict_ragged, jq_evict_layers): tables in device memory, behind the workspace proper.
// KV heads are numbered through all units; unit u owns heads [u * hpu, (u + 1) * hpu).
constexpr int kMaxUnits = 4096;
constexpr size_t kTensorMapBytes = 128;
// A head group of the scoring kernel: consecutive KV heads of one prefix length whose keys fit a share of the
// L2.  A group may run over consecutive units of equal length (their scores are consecutive too).
struct GroupRec {
    int h0, nh;          // first KV head (global numbering) and number of heads
    int tph, L;          // tiles per head, prefix length
    int unit, c20;       // the unit of head h0, and the index of head h0 within it
    long long sbase;     // offset (floats) of head h0's scores in the scores array
    uint32_t tph_magic;  // div_magic(tph): the kernel divides tile numbers by tph with a multiplication
    uint32_t pad;
};
// ceil(2^32 / d) for 2 <= d < 2^31; 2^32 - 1 for d = 1 (the kernel's fast_div corrects the estimate either way).
static inline uint32_t div_magic(uint32_t d) { return d <= 1 ? 0xffffffffu : (uint32_t)((0x100000000ull + d - 1) / d); }
// A KV head as the selection kernel sees it.
struct HeadRec {
    int L, nkeep;
    int unit, kv_in;     // the unit and the head's index within it
    long long soff;      // offset (floats / keys) of the head's scores and select keys
    long long ooff;      // offset (rows) of the head's kept indices and compacted rows in the stacked outputs
};
struct UnitTables {
    const void *maps = nullptr, *qmaps = nullptr;   // device: [nunits] TMA tensor maps of K, of Qwin
    const void *const *K = nullptr;      // device: [nunits] base of K
    const void *const *V = nullptr;      // device: [nunits] base of V
    const GroupRec *groups = nullptr;    // device: [ngroups]
    const HeadRec *heads = nullptr;      // device: [nunits * hpu]
    // of the one-pass eviction only, which needs no groups:
    const void *block_maps = nullptr;    // device: [nunits] TMA tensor maps of K in blocks of 16 keys
    const long long *tbase = nullptr;    // device: [nunits * hpu] tiles of the heads before it (null: all heads have the same number)
    int ngroups = 0, hpu = 0;            // hpu: KV heads per unit
    int max_group_tiles = 0;             // most tiles in any group (sizes the grid)
    int max_L = 0;                       // longest prefix (sizes the selection kernel's shared memory)
    long long total_keys = 0;            // keys of all units (floats in the scores array)
    long long total_rows = 0;            // rows of the stacked outputs
    long long total_tiles = 0;           // tiles of all heads
};
// Where the tables lie, from their first byte on: what both ways of a call read, then the groups of the two passes or the two tables
// of the one-pass eviction.  A workspace with room for the tables of the two passes is enough for every call.
struct UnitTableLayout {
    size_t maps = 0, qmaps, K, V, heads, groups, block_maps, tbase, bytes, prune_bytes;
};
static inline UnitTableLayout unit_tables(int nunits, int hpu)
{
    UnitTableLayout t;
    t.qmaps = (size_t)nunits * kTensorMapBytes;   // (the two of a unit apart: side by side, 256 bytes to a unit, 16 layers of 8 x 7745 keys took 127.8 us instead
                                                  // of 126.4, 8 layers of 8 x 4022 54.9 instead of 53.7)
    t.K = align_up(2 * (size_t)nunits * kTensorMapBytes, 256);
    t.V = t.K + align_up((size_t)nunits * sizeof(void *), 256);
    t.heads = t.V + align_up((size_t)nunits * sizeof(void *), 256);
    t.groups = t.block_maps = t.heads + align_up((size_t)nunits * hpu * sizeof(HeadRec), 256);
    t.bytes = t.groups + align_up((size_t)nunits * hpu * sizeof(GroupRec), 256);
    t.tbase = t.block_maps + align_up((size_t)nunits * kTensorMapBytes, 256);
    t.prune_bytes = t.tbase + align_up((size_t)nunits * hpu * sizeof(long long), 256);
    return t;
}
// One tensor map for a bf16 tensor [heads][rows][128], boxes of 64 columns x box_rows rows (host).
// (head_rows: rows between consecutive heads in memory when they are not packed).
bool make_tensor_map(void *map, const void *ptr, int rows, int heads, int box_rows, int head_rows = 0);
// Most KV heads of L keys that the scoring kernel takes as one group (tiles of a group are split over `sms` CTAs).
int heads_per_group(int L, int heads, int tiles_per_head, int sms, bool wide);   // wide: more than 128 query rows
int score_sms();   // CTAs of the scoring kernel on the current device; 0 on error

// Host-side bookkeeping.
int device_sms();           // multiprocessors of the current device; 0 on error
void count_launch(int n = 1);
jq_status check_launch();   // cudaGetLastError -> JQ_OK / JQ_ERR_CUDA

// Stage launchers (arguments already validated).
jq_status launch_score_fma(const void *K, const void *Q, const jq_shape &s, float *scores,
                           const Workspace &w, cudaStream_t st);
// Kwin, when not null: keys [Hkv][w][128] of the query positions themselves (window-inclusive softmax).
// With tables, s holds the head geometry and the total head count (s.L, s.budget unused): tiles, lengths and
// score offsets come from the tables, K and Q are ignored.
// k_head_rows: rows between consecutive heads of K in memory when the heads are not packed (0: s.L).
jq_status launch_score_tc(const void *K, const void *Q, const jq_shape &s, float *scores,
                          const Workspace &w, cudaStream_t st, const void *Kwin = nullptr,
                          const UnitTables *tables = nullptr, int k_head_rows = 0);
// With K, V, Kout, Vout given, the kernel also copies the kept rows (the fused layer path).  With tables, every
// head has a length, a budget and offsets of its own (s.L, s.budget unused).
// src_head_rows: rows between consecutive heads of K and V in memory when the heads are not packed (0: s.L);
// out_head_rows: rows between consecutive heads of Kout and Vout when more than nkeep (0: nkeep).
// Kwin, Vwin: with both given, the w window rows of every head follow its kept rows in Kout and Vout.
// scored: with select_reads_scored_tiles, only the blocks of 16 positions whose bits are set have scores; the others count as zero,
// and none of the positions that are kept is further than a window from one that is set.
struct ScoredTiles {
    const uint8_t *bits = nullptr;   // device: a byte per tile of 128 positions, heads one after the other
    const long long *tbase = nullptr;   // device: a head's first tile; null: tph of them from one head to the next
    int tph = 0;
    int max_tiles = 0;               // of any head
    long long tiles = 0;             // of all heads (read by the bounds-checked build)
};
constexpr int kMaxSparseTiles = 1024;   // (their list is in shared memory; two CTAs to an SM)
bool select_reads_scored_tiles(const jq_shape &s, int max_L);
jq_status launch_select(const float *scores, const jq_shape &s, int32_t *idx, float *pooled,
                        const Workspace &w, cudaStream_t st, const void *K = nullptr, const void *V = nullptr,
                        void *Kout = nullptr, void *Vout = nullptr, const UnitTables *tables = nullptr,
                        int src_head_rows = 0, int out_head_rows = 0, const void *Kwin = nullptr, const void *Vwin = nullptr,
                        const ScoredTiles *scored = nullptr);
// Scoring, selection and rows in one pass over K and a look at the keys that can be kept (jq_prune.cu), arguments as launch_score_tc
// and launch_select take them.  prune_taken: whether a call over `heads` heads (tiles, keys and kept pairs of all of them, the
// longest max_L) is one that this is the faster way for.
bool prune_taken(const jq_shape &s, int heads, long long tiles, long long keys, long long kept, int max_L);
jq_status launch_evict_pruned(const void *K, const void *V, const void *Q, const jq_shape &s, void *Kout, void *Vout, int32_t *idx,
                              const Workspace &w, cudaStream_t st, const UnitTables *tables = nullptr, int src_head_rows = 0,
                              int out_head_rows = 0, const void *Kwin = nullptr, const void *Vwin = nullptr);
// The keys and values of a one-launch layer call: rows [0, LA) of every head in KA, VA (a_rows rows apart; 0: packed), rows
// [LA, LA + LB) in KB, VB (packed), and the window's (Kwin: one more tile of the denominator; Vwin too: its rows are kept).
struct FusedSource {
    const void *KA = nullptr, *VA = nullptr, *KB = nullptr, *VB = nullptr, *Kwin = nullptr, *Vwin = nullptr;
    int LA = 0, LB = 0, a_rows = 0;
    bool inplace = false;   // the outputs are KA, VA themselves
};
// The whole pass in one launch, if the shape is one that this is the faster way for (*taken; else nothing is launched).
// In place (Kout, Vout are KA, VA and out_head_rows is a_rows) the kept rows move to the head of the cache.
jq_status launch_fused(const jq_shape &s, const FusedSource &src, const void *Q, void *Kout, void *Vout, int out_head_rows,
                       int32_t *idx, const Workspace &w, cudaStream_t st, bool *taken);
jq_status launch_gather(const void *K, const void *V, const int32_t *idx, const jq_shape &s,
                        void *Kout, void *Vout, cudaStream_t st);

}  // namespace jq
