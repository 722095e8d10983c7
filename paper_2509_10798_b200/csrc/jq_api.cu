// The C ABI: argument validation, workspace carve-up, stage sequencing.  See include/jq.h.
#include "jq_internal.cuh"
#include <algorithm>
#include <atomic>
#include <exception>
#include <vector>

namespace jq {

static std::atomic<unsigned long long> g_launches{0};
void count_launch(int n) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }

jq_status check_launch() { return cudaGetLastError() == cudaSuccess ? JQ_OK : JQ_ERR_CUDA; }

int device_sms()
{
    static std::atomic<int> sms[64];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if ((n = sms[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    sms[dev].store(n, std::memory_order_relaxed);
    return n;
}

static jq_status check_shape(const jq_shape *s)
{
    if (!s) return JQ_ERR_INVALID_ARG;
    if (s->Hkv < 1 || s->Hq < 1 || s->group < 1 || s->L < 1 || s->d < 1 || s->w < 1 || s->budget < 1 ||
        s->pool < 1)
        return JQ_ERR_INVALID_ARG;
    if ((long long)s->Hkv * s->group != (long long)s->Hq) return JQ_ERR_INVALID_ARG;
    if (s->pool % 2 == 0) return JQ_ERR_INVALID_ARG;
    if (s->d != kD) return JQ_ERR_UNSUPPORTED;
    if ((long long)s->group * s->w > kMaxR) return JQ_ERR_UNSUPPORTED;
    if (s->pool > 63) return JQ_ERR_UNSUPPORTED;
    if (s->L > (1 << 24)) return JQ_ERR_UNSUPPORTED;
    if (s->Hkv > 65535) return JQ_ERR_UNSUPPORTED;
    return JQ_OK;
}

static bool aligned16(const void *p) { return p && ((uintptr_t)p & 15u) == 0; }

static jq_status check_ws(const jq_shape *s, void *ws, size_t ws_bytes, Workspace *out)
{
    if (!aligned16(ws) || ((uintptr_t)ws & 255u)) return JQ_ERR_INVALID_ARG;
    *out = carve(ws, *s);
    return ws_bytes < out->bytes ? JQ_ERR_WORKSPACE : JQ_OK;
}

// Whether one pass over the keys and a look at the candidates is the faster way for a layer, and the workspace has room for it; it is
// then laid out for that (w.prune).
static bool layer_pruned(const jq_shape &s, void *ws, size_t ws_bytes, Workspace *w)
{
    const long long tiles = (long long)s.Hkv * ((s.L + 127) / 128), keys = (long long)s.Hkv * s.L;
    if (!prune_taken(s, s.Hkv, tiles, keys, (long long)s.Hkv * (s.budget < s.L ? s.budget : s.L), s.L)) return false;
    const Workspace p = carve_pruned(ws, (size_t)s.Hkv, (size_t)s.group * s.w, (size_t)keys);
    if (ws_bytes < p.bytes) return false;
    *w = p;
    return true;
}

// One layer that the one-launch pass does not take.  src_head_rows, out_head_rows: rows between consecutive heads of K and V / of Kout
// and Vout when they are not packed; Vwin: the window rows follow the kept ones.
static jq_status evict_in_steps(const void *K, const void *V, const void *Qwin, const jq_shape &s, void *Kout, void *Vout, int32_t *kept_idx,
                                const Workspace &w, cudaStream_t st, int src_head_rows = 0, int out_head_rows = 0,
                                const void *Kwin = nullptr, const void *Vwin = nullptr)
{
    if (w.prune)
        return launch_evict_pruned(K, V, Qwin, s, Kout, Vout, kept_idx, w, st, nullptr, src_head_rows, out_head_rows, Kwin, Vwin);
    const jq_status rc = launch_score_tc(K, Qwin, s, w.scores, w, st, Kwin, nullptr, src_head_rows);
    if (rc != JQ_OK) return rc;
    return launch_select(w.scores, s, kept_idx, nullptr, w, st, K, V, Kout, Vout, nullptr, src_head_rows, out_head_rows, Vwin ? Kwin : nullptr, Vwin);
}

}  // namespace jq

using namespace jq;

extern "C" {

jq_status jq_check_shape(const jq_shape *s) { return check_shape(s); }

size_t jq_workspace_bytes(const jq_shape *s)
{
    if (check_shape(s) != JQ_OK) return 0;
    return workspace_need(*s);
}

int jq_num_kept(const jq_shape *s)
{
    if (check_shape(s) != JQ_OK) return 0;
    return s->budget < s->L ? s->budget : s->L;
}

jq_status jq_workspace_init(void *ws, size_t ws_bytes, jq_stream_t stream)
{
    if (!aligned16(ws) || ((uintptr_t)ws & 255u)) return JQ_ERR_INVALID_ARG;
    if (ws_bytes < 256) return JQ_ERR_WORKSPACE;
    return cudaMemsetAsync(ws, 0, 256, (cudaStream_t)stream) == cudaSuccess ? JQ_OK : JQ_ERR_CUDA;
}

jq_status jq_score(const void *K, const void *Qwin, const jq_shape *s, float *scores, void *ws,
                   size_t ws_bytes, jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (!aligned16(K) || !aligned16(Qwin) || !aligned16(scores)) return JQ_ERR_INVALID_ARG;
    Workspace w;
    if ((rc = check_ws(s, ws, ws_bytes, &w)) != JQ_OK) return rc;
    return launch_score_tc(K, Qwin, *s, scores, w, (cudaStream_t)stream);
}

jq_status jq_score_windowed(const void *K, const void *Qwin, const void *Kwin, const jq_shape *s, float *scores,
                            void *ws, size_t ws_bytes, jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (s->w > 128) return JQ_ERR_UNSUPPORTED;   // the window keys of a head must fit one tile
    if (!aligned16(K) || !aligned16(Qwin) || !aligned16(Kwin) || !aligned16(scores)) return JQ_ERR_INVALID_ARG;
    Workspace w;
    if ((rc = check_ws(s, ws, ws_bytes, &w)) != JQ_OK) return rc;
    return launch_score_tc(K, Qwin, *s, scores, w, (cudaStream_t)stream, Kwin);
}

jq_status jq_evict_layer_windowed(const void *K, const void *V, const void *Qwin, const void *Kwin, const jq_shape *s,
                                  void *Kout, void *Vout, int32_t *kept_idx, void *ws, size_t ws_bytes,
                                  jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (s->w > 128) return JQ_ERR_UNSUPPORTED;   // the window keys of a head must fit one tile
    if (!aligned16(K) || !aligned16(V) || !aligned16(Qwin) || !aligned16(Kwin) || !aligned16(Kout) || !aligned16(Vout) ||
        !aligned16(kept_idx))
        return JQ_ERR_INVALID_ARG;
    Workspace w;
    if ((rc = check_ws(s, ws, ws_bytes, &w)) != JQ_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    FusedSource src;
    src.KA = K; src.VA = V; src.LA = s->L; src.Kwin = Kwin;
    bool taken = false;
    if (!layer_pruned(*s, ws, ws_bytes, &w) && ((rc = launch_fused(*s, src, Qwin, Kout, Vout, 0, kept_idx, w, st, &taken)) != JQ_OK || taken)) return rc;
    return evict_in_steps(K, V, Qwin, *s, Kout, Vout, kept_idx, w, st, 0, 0, Kwin);
}

jq_status jq_evict_layer_window_kept(const void *K, const void *V, const void *Qwin, const void *Kwin, const void *Vwin,
                                     const jq_shape *s, void *Kout, void *Vout, int32_t *kept_idx, void *ws, size_t ws_bytes,
                                     jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (s->w > 128) return JQ_ERR_UNSUPPORTED;                 // the window keys of a head must fit one tile
    if (s->budget <= s->w) return JQ_ERR_INVALID_ARG;          // the window alone would fill the budget
    if (!aligned16(K) || !aligned16(V) || !aligned16(Qwin) || !aligned16(Kwin) || !aligned16(Vwin) || !aligned16(Kout) ||
        !aligned16(Vout) || !aligned16(kept_idx))
        return JQ_ERR_INVALID_ARG;
    Workspace w;
    if ((rc = check_ws(s, ws, ws_bytes, &w)) != JQ_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    // prefix rows: the window-inclusive pass with budget - w; then the w window rows behind them, head by head
    jq_shape sp = *s;
    sp.budget = s->budget - s->w;
    const size_t np = (size_t)(sp.budget < s->L ? sp.budget : s->L), nt = np + (size_t)s->w;
    FusedSource src;
    src.KA = K; src.VA = V; src.LA = s->L; src.Kwin = Kwin; src.Vwin = Vwin;
    bool taken = false;
    if (!layer_pruned(sp, ws, ws_bytes, &w) && ((rc = launch_fused(sp, src, Qwin, Kout, Vout, (int)nt, kept_idx, w, st, &taken)) != JQ_OK || taken)) return rc;
    // the kept prefix rows of head kv go to rows [kv * nt, kv * nt + np) of the outputs, its window rows behind them
    return evict_in_steps(K, V, Qwin, sp, Kout, Vout, kept_idx, w, st, 0, (int)nt, Kwin, Vwin);
}

jq_status jq_score_fma(const void *K, const void *Qwin, const jq_shape *s, float *scores, void *ws,
                       size_t ws_bytes, jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (!aligned16(K) || !aligned16(Qwin) || !aligned16(scores)) return JQ_ERR_INVALID_ARG;
    Workspace w;
    if ((rc = check_ws(s, ws, ws_bytes, &w)) != JQ_OK) return rc;
    return launch_score_fma(K, Qwin, *s, scores, w, (cudaStream_t)stream);
}

jq_status jq_select_topk(const float *scores, const jq_shape *s, int32_t *kept_idx, float *pooled_or_null,
                         void *ws, size_t ws_bytes, jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (!aligned16(scores) || !aligned16(kept_idx)) return JQ_ERR_INVALID_ARG;
    if (pooled_or_null && !aligned16(pooled_or_null)) return JQ_ERR_INVALID_ARG;
    Workspace w;
    if ((rc = check_ws(s, ws, ws_bytes, &w)) != JQ_OK) return rc;
    return launch_select(scores, *s, kept_idx, pooled_or_null, w, (cudaStream_t)stream);
}

jq_status jq_compact_kv(const void *K, const void *V, const int32_t *kept_idx, const jq_shape *s,
                        void *Kout, void *Vout, jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (!aligned16(K) || !aligned16(V) || !aligned16(kept_idx) || !aligned16(Kout) || !aligned16(Vout))
        return JQ_ERR_INVALID_ARG;
    return launch_gather(K, V, kept_idx, *s, Kout, Vout, (cudaStream_t)stream);
}

jq_status jq_evict_layer(const void *K, const void *V, const void *Qwin, const jq_shape *s, void *Kout,
                         void *Vout, int32_t *kept_idx, void *ws, size_t ws_bytes, jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (!aligned16(K) || !aligned16(V) || !aligned16(Qwin) || !aligned16(Kout) || !aligned16(Vout) ||
        !aligned16(kept_idx))
        return JQ_ERR_INVALID_ARG;
    Workspace w;
    if ((rc = check_ws(s, ws, ws_bytes, &w)) != JQ_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    FusedSource src;
    src.KA = K; src.VA = V; src.LA = s->L;
    bool taken = false;
    if (!layer_pruned(*s, ws, ws_bytes, &w) && ((rc = launch_fused(*s, src, Qwin, Kout, Vout, 0, kept_idx, w, st, &taken)) != JQ_OK || taken)) return rc;
    return evict_in_steps(K, V, Qwin, *s, Kout, Vout, kept_idx, w, st);
}

// ---- units of one head geometry in buffers of their own: lengths, budgets and offsets per unit

namespace {

constexpr size_t kTablePiece = 60 * 1024;   // bytes of the tables per copy

struct RaggedPlan {
    jq_shape S;                 // head geometry with the total head count (L = longest prefix, budget = largest nkeep)
    size_t keys = 0;            // sum over units of Hkv * L
    long long rows = 0;         // sum over units of Hkv * nkeep
    int max_L = 0;
    bool uniform = true;        // one length and one number of kept rows for all units
};

// Validates the arguments the two ragged entry points share and sums the sizes.  L and budget may be NULL
// (then every unit has common->L / common->budget).
jq_status plan_ragged(const jq_shape *common, int nunits, const int *L, const int *budget, RaggedPlan *out)
{
    if (!common) return JQ_ERR_INVALID_ARG;
    if (nunits < 1) return JQ_ERR_INVALID_ARG;
    if (nunits > kMaxUnits) return JQ_ERR_UNSUPPORTED;
    RaggedPlan pl;
    int max_keep = 0, L0 = 0, keep0 = 0;
    for (int u = 0; u < nunits; ++u) {
        jq_shape su = *common;
        if (L) su.L = L[u];
        if (budget) su.budget = budget[u];
        const jq_status rc = check_shape(&su);
        if (rc != JQ_OK) return rc;
        const int nkeep = su.budget < su.L ? su.budget : su.L;
        pl.keys += (size_t)su.Hkv * su.L;
        pl.rows += (long long)su.Hkv * nkeep;
        if (u == 0) { L0 = su.L; keep0 = nkeep; }
        pl.uniform = pl.uniform && su.L == L0 && nkeep == keep0;
        if (su.L > pl.max_L) pl.max_L = su.L;
        if (nkeep > max_keep) max_keep = nkeep;
    }
    if ((long long)common->Hkv * nunits > 65535) return JQ_ERR_UNSUPPORTED;
    pl.S = *common;
    pl.S.Hkv = common->Hkv * nunits;
    pl.S.Hq = common->Hq * nunits;
    pl.S.L = pl.max_L;
    pl.S.budget = max_keep;
    *out = pl;
    return JQ_OK;
}

}  // namespace

size_t jq_ragged_workspace_bytes(const jq_shape *common, int nunits, const int *L)
{
    RaggedPlan pl;
    if (plan_ragged(common, nunits, L, nullptr, &pl) != JQ_OK) return 0;
    const UnitTableLayout at = unit_tables(nunits, common->Hkv);
    return workspace_need((size_t)pl.S.Hkv, (size_t)common->group * common->w, pl.keys, pl.max_L, at.bytes, at.prune_bytes);
}

long long jq_ragged_output_rows(const jq_shape *common, int nunits, const int *L, const int *budget)
{
    RaggedPlan pl;
    if (plan_ragged(common, nunits, L, budget, &pl) != JQ_OK) return 0;
    return pl.rows;
}

jq_status jq_evict_ragged(const void *const *K, const void *const *V, const void *const *Qwin, int nunits,
                          const jq_shape *common, const int *L, const int *budget, void *Kout, void *Vout,
                          int32_t *kept_idx, void *ws, size_t ws_bytes, jq_stream_t stream)
{
    RaggedPlan pl;
    jq_status rc = plan_ragged(common, nunits, L, budget, &pl);
    if (rc != JQ_OK) return rc;
    if (!K || !V || !Qwin || !aligned16(Kout) || !aligned16(Vout) || !aligned16(kept_idx)) return JQ_ERR_INVALID_ARG;
    for (int u = 0; u < nunits; ++u)
        if (!aligned16(K[u]) || !aligned16(V[u]) || !aligned16(Qwin[u])) return JQ_ERR_INVALID_ARG;
    if (!aligned16(ws) || ((uintptr_t)ws & 255u)) return JQ_ERR_INVALID_ARG;
    const int hpu = common->Hkv, R = common->group * common->w;
    Workspace w = carve(ws, (size_t)pl.S.Hkv, (size_t)R, pl.keys);
    const UnitTableLayout at = unit_tables(nunits, hpu);
    if (ws_bytes < w.bytes + at.bytes) return JQ_ERR_WORKSPACE;
    const int sms = score_sms();
    if (sms < 1) return JQ_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;

    // All tables are assembled in one host buffer of the library's own (so that the caller's arrays are only read
    // before the call returns, whatever memory they live in) and go to the device in as few copies as return at once.
    static thread_local std::vector<unsigned char> staging;
    static thread_local std::vector<int> order;           // the units by falling length
    static thread_local std::vector<long long> out_row;   // [unit] its first output row
    try {
        staging.assign(at.bytes > at.prune_bytes ? at.bytes : at.prune_bytes, 0);
        order.resize(nunits);
        out_row.resize(nunits);
    } catch (const std::exception &) {   // no host memory: nothing is thrown through the C interface
        return JQ_ERR_CUDA;
    }
    unsigned char *hb = staging.data();
    unsigned char *h_maps = hb + at.maps, *h_qmaps = hb + at.qmaps, *h_block_maps = hb + at.block_maps;
    const void **h_K = (const void **)(hb + at.K), **h_V = (const void **)(hb + at.V);
    HeadRec *h_head = (HeadRec *)(hb + at.heads);
    GroupRec *h_grp = (GroupRec *)(hb + at.groups);   // last: there are far fewer than there is room for
    long long *h_tbase = (long long *)(hb + at.tbase);
    UnitTables t;
    for (int u = 0; u < nunits; ++u) t.total_tiles += (long long)hpu * (((L ? L[u] : common->L) + 127) / 128);
    const Workspace wp = carve_pruned(ws, (size_t)pl.S.Hkv, (size_t)R, pl.keys);
    const bool pruned = prune_taken(*common, pl.S.Hkv, t.total_tiles, (long long)pl.keys, pl.rows, pl.max_L) && ws_bytes >= wp.bytes + at.prune_bytes;
    if (pruned) w = wp;
    // The tables hold the units by falling length (equal lengths as given), whatever the order of the call: the kernels that have a
    // CTA per head start the long heads first, and none of those is left to run by itself at the end.  Outputs stay in the call's
    // order.  (32 layers of prompts of 32768, 23212, 13655 and 4099 keys, 8 heads each, in the order of the layers: 1920 -> 1865 us,
    // by rising length 1937 -> 1862, by falling length 1862 either way; with few rows, which go the two-pass way, 2095 -> 1835, 1837
    // -> 1826 and 1833.)
    long long soff = 0, ooff = 0, tbase = 0;
    for (int u = 0; u < nunits; ++u) {
        const int Lu = L ? L[u] : common->L, Bu = budget ? budget[u] : common->budget;
        order[u] = u; out_row[u] = ooff;
        ooff += (long long)hpu * (Bu < Lu ? Bu : Lu);
    }
    if (L) std::stable_sort(order.begin(), order.end(), [L](int a, int b) { return L[a] > L[b]; });
    int ngroups = 0;
    for (int i = 0; i < nunits; ++i) {
        const int u = order[i];
        const int Lu = L ? L[u] : common->L, Bu = budget ? budget[u] : common->budget;
        const int nkeep = Bu < Lu ? Bu : Lu;
        const size_t m = (size_t)i * kTensorMapBytes;
        if (!make_tensor_map(h_maps + m, K[u], Lu, hpu, 128) || !make_tensor_map(h_qmaps + m, Qwin[u], R, hpu, R <= 128 ? 128 : 256) ||
            (pruned && !make_tensor_map(h_block_maps + m, K[u], Lu, hpu, 16)))
            return JQ_ERR_CUDA;
        h_K[i] = K[u]; h_V[i] = V[u];
        for (int h = 0; h < hpu; ++h) {
            HeadRec &r = h_head[i * hpu + h];
            r.L = Lu; r.nkeep = nkeep; r.unit = i; r.kv_in = h;
            r.soff = soff + (long long)h * Lu;
            r.ooff = out_row[u] + (long long)h * nkeep;
            if (pruned) h_tbase[i * hpu + h] = tbase + (long long)h * ((Lu + 127) / 128);
        }
        tbase += (long long)hpu * ((Lu + 127) / 128);
        soff += (long long)hpu * Lu;
    }
    // head groups of the scoring kernel: every run of consecutive units of one length is cut into groups of
    // at most 56 MiB of keys (short prefixes share a group across units, so that a group still has tiles for every CTA)
    for (int u0 = 0; u0 < nunits && !pruned;) {
        const int Lu = L ? L[order[u0]] : common->L, tph = (Lu + 127) / 128;
        int u1 = u0 + 1;
        while (u1 < nunits && (L ? L[order[u1]] : common->L) == Lu) ++u1;
        const int heads = (u1 - u0) * hpu, hpg = heads_per_group(Lu, heads, tph, sms, R > 128);
        for (int h0 = 0; h0 < heads; h0 += hpg) {
            GroupRec &g = h_grp[ngroups++];
            g.h0 = u0 * hpu + h0; g.nh = h0 + hpg <= heads ? hpg : heads - h0;
            g.tph = tph; g.L = Lu; g.unit = u0 + h0 / hpu; g.c20 = h0 % hpu;
            g.sbase = h_head[g.h0].soff; g.tph_magic = div_magic((uint32_t)tph); g.pad = 0;
            if (g.nh * tph > t.max_group_tiles) t.max_group_tiles = g.nh * tph;
        }
        u0 = u1;
    }
    char *tab = (char *)ws + w.bytes;
    // Copies from ordinary host memory return at once up to 64 KB; a larger one waits for the stream to reach it, which kept
    // the host from preparing one call while the GPU worked on the one before (128 units: 1.5 ms in the call, and a gap of
    // about 90 us per call of 2.6 ms).
    const size_t used = !pruned ? at.groups + (size_t)ngroups * sizeof(GroupRec) : pl.uniform ? at.tbase : at.prune_bytes;
    for (size_t off = 0; off < used; off += kTablePiece)
        if (cudaMemcpyAsync(tab + off, hb + off, used - off < kTablePiece ? used - off : kTablePiece, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return JQ_ERR_CUDA;
    t.maps = tab + at.maps;
    t.qmaps = tab + at.qmaps;
    t.K = (const void *const *)(tab + at.K);
    t.V = (const void *const *)(tab + at.V);
    t.heads = (const HeadRec *)(tab + at.heads);
    t.groups = (const GroupRec *)(tab + at.groups);
    t.block_maps = tab + at.block_maps;
    if (pruned && !pl.uniform) t.tbase = (const long long *)(tab + at.tbase);
    t.ngroups = ngroups; t.hpu = hpu; t.max_L = pl.max_L; t.total_keys = (long long)pl.keys; t.total_rows = pl.rows;
    if (pruned) return launch_evict_pruned(nullptr, nullptr, nullptr, pl.S, Kout, Vout, kept_idx, w, st, &t);
    if ((rc = launch_score_tc(nullptr, nullptr, pl.S, w.scores, w, st, nullptr, &t)) != JQ_OK) return rc;
    return launch_select(w.scores, pl.S, kept_idx, nullptr, w, st, nullptr, nullptr, Kout, Vout, &t);
}

size_t jq_layers_workspace_bytes(const jq_shape *layer, int nlayers)
{
    return jq_ragged_workspace_bytes(layer, nlayers, nullptr);
}

jq_status jq_evict_layers(const void *const *K, const void *const *V, const void *const *Qwin, int nlayers,
                          const jq_shape *layer, void *Kout, void *Vout, int32_t *kept_idx, void *ws, size_t ws_bytes,
                          jq_stream_t stream)
{
    return jq_evict_ragged(K, V, Qwin, nlayers, layer, nullptr, nullptr, Kout, Vout, kept_idx, ws, ws_bytes, stream);
}

// ---- streaming re-eviction: the pruned cache of a layer has grown during decoding

size_t jq_append_workspace_bytes(const jq_shape *s)
{
    if (check_shape(s) != JQ_OK) return 0;
    const size_t nkeep = (size_t)(s->budget < s->L ? s->budget : s->L);
    return workspace_need(*s) + 2 * align_up((size_t)s->Hkv * nkeep * s->d * 2, 256);
}

jq_status jq_evict_append(void *Kc, void *Vc, int cap, int n_old, const void *Knew, const void *Vnew, int n_new,
                          const void *Qrecent, const jq_shape *s, int32_t *kept_idx, void *ws, size_t ws_bytes,
                          jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (n_old < 0 || n_new < 0 || cap < 1 || (long long)n_old + n_new != (long long)s->L || s->L > cap) return JQ_ERR_INVALID_ARG;
    if (!aligned16(Kc) || !aligned16(Vc) || !aligned16(Qrecent) || !aligned16(kept_idx)) return JQ_ERR_INVALID_ARG;
    if (n_new > 0 && (!aligned16(Knew) || !aligned16(Vnew))) return JQ_ERR_INVALID_ARG;
    Workspace w;
    if ((rc = check_ws(s, ws, ws_bytes, &w)) != JQ_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t row = (size_t)s->d * 2, nkeep = (size_t)(s->budget < s->L ? s->budget : s->L), rows_bytes = align_up((size_t)s->Hkv * nkeep * row, 256);
    if (ws_bytes < w.bytes + 2 * rows_bytes) return JQ_ERR_WORKSPACE;
    // a short cache: one launch that reads the two parts where they are and moves the kept rows in place
    FusedSource src;
    src.KA = Kc; src.VA = Vc; src.LA = n_old; src.a_rows = cap; src.KB = Knew; src.VB = Vnew; src.LB = n_new; src.inplace = true;
    bool taken;
    if ((rc = launch_fused(*s, src, Qrecent, Kc, Vc, cap, kept_idx, w, st, &taken)) != JQ_OK || taken) return rc;
    layer_pruned(*s, ws, ws_bytes - 2 * rows_bytes, &w);
    char *const Ktmp = (char *)ws + w.bytes, *const Vtmp = Ktmp + rows_bytes;
    // 1. the new rows go behind the retained ones, head by head (the cache keeps `cap` rows per head)
    if (n_new > 0) {
        if (cudaMemcpy2DAsync((char *)Kc + (size_t)n_old * row, (size_t)cap * row, Knew, (size_t)n_new * row, (size_t)n_new * row,
                              (size_t)s->Hkv, cudaMemcpyDeviceToDevice, st) != cudaSuccess) return JQ_ERR_CUDA;
        if (cudaMemcpy2DAsync((char *)Vc + (size_t)n_old * row, (size_t)cap * row, Vnew, (size_t)n_new * row, (size_t)n_new * row,
                              (size_t)s->Hkv, cudaMemcpyDeviceToDevice, st) != cudaSuccess) return JQ_ERR_CUDA;
    }
    // 2. the pass over the L = n_old + n_new rows of every head, compacted into the workspace (a row may move
    //    onto a row that another thread still has to read, so the compaction cannot run in place)
    if ((rc = evict_in_steps(Kc, Vc, Qrecent, *s, Ktmp, Vtmp, kept_idx, w, st, cap)) != JQ_OK) return rc;
    // 3. back to the head of the cache
    if (cudaMemcpy2DAsync(Kc, (size_t)cap * row, Ktmp, nkeep * row, nkeep * row, (size_t)s->Hkv, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return JQ_ERR_CUDA;
    if (cudaMemcpy2DAsync(Vc, (size_t)cap * row, Vtmp, nkeep * row, nkeep * row, (size_t)s->Hkv, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return JQ_ERR_CUDA;
    return JQ_OK;
}

namespace {

constexpr int kHostChunks = 4;                 // most chunks of a call
constexpr size_t kHostChunkBytes = 8u << 20;   // least keys of a chunk of heads
constexpr size_t kHostIdxPad = 256;
static_assert(kHostChunks * 4 * sizeof(int32_t) + 16 <= kHostIdxPad, "room for the chunks' alignment");

// The stream beside the caller's and the events between the two: one set per host thread and device, made at the first call
// that uses it and released with the thread.  Calls of one thread on several streams share it (their side work then runs in
// the order of the calls).
struct HostPipe {
    cudaStream_t side = nullptr;
    cudaEvent_t in = nullptr, out = nullptr;
    ~HostPipe()
    {
        if (in) cudaEventDestroy(in);
        if (out) cudaEventDestroy(out);
        if (side) cudaStreamDestroy(side);
    }
};

HostPipe *host_pipe()
{
    static thread_local HostPipe pipes[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    HostPipe &p = pipes[dev];
    if ((!p.side && cudaStreamCreateWithFlags(&p.side, cudaStreamNonBlocking) != cudaSuccess) ||
        (!p.in && cudaEventCreateWithFlags(&p.in, cudaEventDisableTiming) != cudaSuccess) ||
        (!p.out && cudaEventCreateWithFlags(&p.out, cudaEventDisableTiming) != cudaSuccess)) {
        cudaGetLastError();
        return nullptr;   // the call then runs on the caller's stream alone
    }
    return &p;
}

// The device buffer of a call whose workspace, the last part of it, has ws_bytes.
size_t host_call_bytes(const jq_shape *s, size_t ws_bytes)
{
    const size_t row = (size_t)s->d * 2;
    const size_t nkeep = (size_t)(s->budget < s->L ? s->budget : s->L);
    size_t b = 0;
    b += 2 * align_up((size_t)s->Hkv * s->L * row, 256);      // K, V
    b += align_up((size_t)s->Hq * s->w * row, 256);           // Qwin
    b += 2 * align_up((size_t)s->Hkv * nkeep * row, 256);     // Kout, Vout
    b += align_up((size_t)s->Hkv * nkeep * 4, 256) + kHostIdxPad;   // kept_idx, with room to align every chunk's
    return b + ws_bytes;
}

}  // namespace

size_t jq_host_call_bytes(const jq_shape *s) { return check_shape(s) == JQ_OK ? host_call_bytes(s, workspace_need(*s)) : 0; }

jq_status jq_evict_layer_host(const void *hK, const void *hV, const void *hQwin, const jq_shape *s,
                              void *hKout, void *hVout, int32_t *hkept_idx, void *dev_buf,
                              size_t dev_buf_bytes, jq_stream_t stream)
{
    jq_status rc = check_shape(s);
    if (rc != JQ_OK) return rc;
    if (!hK || !hV || !hQwin || !hKout || !hVout || !hkept_idx) return JQ_ERR_INVALID_ARG;
    if (!dev_buf || ((uintptr_t)dev_buf & 255u)) return JQ_ERR_INVALID_ARG;
    if (dev_buf_bytes < host_call_bytes(s, carve(nullptr, *s).bytes)) return JQ_ERR_WORKSPACE;   // (what is enough for either way)
    cudaStream_t st = (cudaStream_t)stream;
    const size_t row = (size_t)s->d * 2;
    const size_t nkeep = (size_t)(s->budget < s->L ? s->budget : s->L);
    const size_t kvb = (size_t)s->Hkv * s->L * row, qb = (size_t)s->Hq * s->w * row;
    const size_t ob = (size_t)s->Hkv * nkeep * row, ib = (size_t)s->Hkv * nkeep * 4;
    char *p = (char *)dev_buf;
    char *dK = p;          p += align_up(kvb, 256);
    char *dV = p;          p += align_up(kvb, 256);
    char *dQ = p;          p += align_up(qb, 256);
    char *dKo = p;         p += align_up(ob, 256);
    char *dVo = p;         p += align_up(ob, 256);
    char *dI = p;          p += align_up(ib, 256) + kHostIdxPad;
    char *ws = p;
    const size_t wsb = dev_buf_bytes - (size_t)(ws - (char *)dev_buf);
    if (cudaMemsetAsync(ws, 0, 256, st) != cudaSuccess) return JQ_ERR_CUDA;
    if (cudaMemcpyAsync(dQ, hQwin, qb, cudaMemcpyHostToDevice, st) != cudaSuccess) return JQ_ERR_CUDA;
    // V is read at the kept rows only.  A page-locked host buffer is mapped into the device's address space: the
    // selection kernel then fetches those rows from it directly and the copy of all of V is skipped.
    const char *v_src = dV;
    cudaPointerAttributes pa;
    if (cudaPointerGetAttributes(&pa, hV) == cudaSuccess && pa.type == cudaMemoryTypeHost && pa.devicePointer &&
        !((uintptr_t)pa.devicePointer & 15u)) {
        v_src = (const char *)pa.devicePointer;
    } else {
        cudaGetLastError();
    }
    // The heads are taken in chunks: while one chunk's keys cross to the device on `stream`, the one before is evicted and
    // its results cross back on a stream beside it (the link carries both directions at once).  The copy of K, about 19 us
    // per MB, is what bounds the call; in one piece the pass and the copies back came on top of it.  Measured (us, one
    // piece, 2, 3, 4, 8 chunks): 8 heads x 32768 keys 1412, 1371, 1353, 1357, 1370; 4 x 65000, budget 4000, 1513, 1436,
    // 1443, 1409, 1435; 8 x 8000 480, 474, 483, 483, 483: each chunk's small copies back slow the keys down, so calls below
    // 32 MB stay in one piece.
    HostPipe *pipe = nullptr;
    int chunk = s->Hkv;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) return JQ_ERR_CUDA;
    const size_t head_bytes = (size_t)s->L * row;
    if (s->Hkv > 1 && kvb >= kHostChunks * kHostChunkBytes && cap == cudaStreamCaptureStatusNone && (pipe = host_pipe()) != nullptr) {
        chunk = (int)((kHostChunkBytes + head_bytes - 1) / head_bytes);
        const int least = (s->Hkv + kHostChunks - 1) / kHostChunks;
        if (chunk < least) chunk = least;
    }
    cudaStream_t side = pipe ? pipe->side : st;
    for (int h = 0, n = 0; h < s->Hkv; h += chunk, ++n) {
        jq_shape sc = *s;
        sc.Hkv = s->Hkv - h < chunk ? s->Hkv - h : chunk;
        sc.Hq = sc.Hkv * s->group;
        const size_t koff = (size_t)h * head_bytes, kb = (size_t)sc.Hkv * head_bytes, rows = (size_t)h * nkeep;
        const size_t cob = (size_t)sc.Hkv * nkeep * row;
        int32_t *const idx = (int32_t *)dI + align_up(rows, 4) + 4 * (size_t)n;   // 16-byte aligned, chunks apart
        if (cudaMemcpyAsync(dK + koff, (const char *)hK + koff, kb, cudaMemcpyHostToDevice, st) != cudaSuccess ||
            (v_src == dV && cudaMemcpyAsync(dV + koff, (const char *)hV + koff, kb, cudaMemcpyHostToDevice, st) != cudaSuccess) ||
            (pipe && (cudaEventRecord(pipe->in, st) != cudaSuccess || cudaStreamWaitEvent(side, pipe->in, 0) != cudaSuccess))) {
            rc = JQ_ERR_CUDA;
            break;
        }
        rc = jq_evict_layer(dK + koff, v_src + koff, dQ + (size_t)h * s->group * s->w * row, &sc, dKo + rows * row, dVo + rows * row, idx,
                            ws, wsb, (jq_stream_t)side);
        if (rc == JQ_OK &&
            (cudaMemcpyAsync(hkept_idx + rows, idx, (size_t)sc.Hkv * nkeep * 4, cudaMemcpyDeviceToHost, side) != cudaSuccess ||
             cudaMemcpyAsync((char *)hKout + rows * row, dKo + rows * row, cob, cudaMemcpyDeviceToHost, side) != cudaSuccess ||
             cudaMemcpyAsync((char *)hVout + rows * row, dVo + rows * row, cob, cudaMemcpyDeviceToHost, side) != cudaSuccess))
            rc = JQ_ERR_CUDA;
        if (rc != JQ_OK) break;
    }
    // whatever has been issued beside the stream belongs to the call (after an error too)
    if (pipe && (cudaEventRecord(pipe->out, side) != cudaSuccess || cudaStreamWaitEvent(st, pipe->out, 0) != cudaSuccess)) return JQ_ERR_CUDA;
    return rc;
}

jq_status jq_last_device_status(const void *ws, jq_stream_t stream)
{
    if (!ws) return JQ_ERR_INVALID_ARG;
    int word = 0;
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return JQ_ERR_CUDA;
    if (cudaMemcpy(&word, ws, sizeof word, cudaMemcpyDeviceToHost) != cudaSuccess) return JQ_ERR_CUDA;
    if (word < 0 || word > JQ_ERR_TIMEOUT) return JQ_ERR_CUDA;
    return (jq_status)word;
}

unsigned long long jq_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char *jq_status_string(jq_status s)
{
    switch (s) {
        case JQ_OK: return "ok";
        case JQ_ERR_INVALID_ARG: return "invalid argument";
        case JQ_ERR_UNSUPPORTED: return "unsupported shape";
        case JQ_ERR_WORKSPACE: return "workspace too small";
        case JQ_ERR_CUDA: return "CUDA error";
        case JQ_ERR_TIMEOUT: return "device-side wait timed out";
    }
    return "unknown status";
}

}  // extern "C"
