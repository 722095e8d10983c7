// One decoding step over the pruned cache (the step after the eviction pass: decoding continues with the
// retained pairs only).  Single-position GQA attention, out[h] = softmax_j(q[h] . Kc[kv,j] / sqrt(d)) Vc[kv].
//
// What bounds it: the single read of the two compacted arrays (2 * Hkv * n * 256 bytes) when there are many heads,
// and the latency of one such read plus the merge when there are few.  So a KV head is one thread-block CLUSTER of
// 1 to 16 CTAs of eight or twelve warps; a warp takes units of 16 keys, keeps a running softmax of its own and never waits for
// another warp before the merge, and both the K and the V rows of a unit go straight from global memory into
// matrix-instruction fragments (no staging in shared memory, no barrier in the loop: 16 independent 16-byte loads
// per lane and unit; one CTA to an SM: at 128 registers and two CTAs the spills cost more than they gave).
//   - logits: S[16 keys x 8 heads] = K q^T, mma.sync m16n8k16.  The order of the 128 dimensions within a dot product is
//     free, so a lane takes 16 contiguous bytes of a key row as the operands of two steps, and q is permuted alike.
//     bf16 products, fp32 accumulation.
//   - output: O^T[d x heads] += V^T P, V's rows paired by byte permutes, P transposed in registers (movmatrix).  P must not
//     be rounded to bf16: it is the sum of three bf16 numbers (24 bits), p = hi + mid + lo exactly to fp32 precision, one
//     product for each; groups of at most 4 heads repeat their heads in the other four columns and so carry two of the
//     three parts in one product.  (With FMAs the group's 2 x 128 multiply-adds per key and head would bind, and with the
//     heads as rows of the products, half of them empty, the loop took a quarter longer.)
//   - merge: the warps' (m, l, O) through shared memory, then every CTA pushes its share of each output to the
//     CTA of the cluster that writes it (distributed shared memory), one cluster barrier, and the sums are taken in
//     rank order: deterministic, one launch, no counters in memory.
// Measured (B200, back-to-back calls; before: one CTA per 64 keys staged in shared memory, FMAs, partials and a ticket in
// global memory): 8 KV heads x 1024 keys 12.3 -> 4.6 us (latency: 0.9 TB/s), 128 x 2048 186 -> 25.2 us (5.3 TB/s, 0.81 of
// the measured copy bandwidth).
#include <cuda_bf16.h>
#include <mutex>

#include "jq_internal.cuh"
#include "jq_debug.cuh"

namespace jq {
namespace {

constexpr int kDecChunk = 64;       // sizes the caller's workspace (part of the ABI; this kernel keeps its partials on chip)
constexpr int kDecWarps = 8, kDecManyWarps = 12;   // (decode_shape)
constexpr int kDecResident = 1;     // CTAs per SM
constexpr int kDecUnit = 16;        // keys a warp takes at a time
constexpr int kDecMaxGroup = 8;     // query heads per KV head
constexpr int kDecMaxCluster = 16;  // CTAs per KV head (more than 8 needs the kernel's opt-in)
constexpr int kPartial = kD + 2;    // floats per (chunk, head) of the caller's workspace
constexpr int kOPad = kD + 4;       // row pitch (floats) of a warp's output tile in shared memory

template <int kWarps>
struct DecSmem {
    __nv_bfloat16 q[kDecMaxGroup * kD];
    float O[kWarps][kDecMaxGroup][kOPad];
    float m[kWarps][kDecMaxGroup], l[kWarps][kDecMaxGroup];
    // what the cluster's CTAs push here: rank r's statistics of every head, and its share of the outputs written here
    float rm[kDecMaxCluster][kDecMaxGroup], rl[kDecMaxCluster][kDecMaxGroup];
    float rO[kDecMaxGroup * kD + kDecMaxCluster];   // [rank][share]: the shares of all ranks make up the head's outputs
};

__device__ __forceinline__ float dec_ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Read once: not kept in the L1.  (Not through the read-only path, which is for data that nobody writes during the kernel's
// life: the kernel may be set up while the one that writes the cache still runs.)
__device__ __forceinline__ uint4 ld_stream(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)   // lo in the low half
{
    const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *(const uint32_t *)&t;
}
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ void push_f32(float *local, uint32_t rank, float v)   // to the same variable of CTA `rank`
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

__device__ __forceinline__ uint32_t transpose8x8(uint32_t v)   // 8 x 8 matrix of 16-bit values over the warp, two per lane
{
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(v));
    return d;
}

// DUP (groups of at most 4 heads): columns 4 to 7 of the matrix products repeat the heads 0 to 3, so that one product
// carries two of the three parts of P.
template <bool DUP, int kWarps>
__global__ void __launch_bounds__(32 * kWarps, kDecResident)
decode_step(const uint4 *Kc, const uint4 *Vc, const __nv_bfloat16 *q, int n,
            int group, float scale_log2, float *__restrict__ out JQ_DBG_PARAM)
{
    extern __shared__ __align__(16) uint8_t dec_raw[];
    DecSmem<kWarps> &sm = *(DecSmem<kWarps> *)dec_raw;
    constexpr int kThreads = 32 * kWarps;
    uint32_t rank, C;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int kv = blockIdx.x / C;
    const int nunits = (n + kDecUnit - 1) / kDecUnit, stride = (int)C * kWarps;
    const long long n_rows = (long long)(gridDim.x / C) * n;   // extent, for the bounds-checked build
    (void)n_rows;
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // waited for before the first push
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();   // the stream's next kernel may be set up; it waits for this one's results

    const size_t head = (size_t)kv * n;
    int u = (int)rank * kWarps + warp;
    uint4 kf[8], vf[8];
    // K: rows g and 8 + g of the unit, 16-byte pieces t, 4 + t, 8 + t, 12 + t (rows past the end are masked below)
    auto load_k = [&](int uu) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int row = min(uu * kDecUnit + 8 * r + g, n - 1);
            const uint4 *src = Kc + (head + row) * 16 + t;
            const bool in = JQ_IN(head + row, n_rows, kDbgDecode, 1);
#pragma unroll
            for (int i = 0; i < 4; ++i) kf[4 * r + i] = in ? ld_stream(src + 4 * i) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    // V: rows 2t, 2t + 1, 2t + 8, 2t + 9 of the unit, 16-byte pieces g and 8 + g
    auto load_v = [&](int uu) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int row = min(uu * kDecUnit + 2 * t + (r & 1) + 8 * (r >> 1), n - 1);
            const uint4 *src = Vc + (head + row) * 16 + g;
            const bool in = JQ_IN(head + row, n_rows, kDbgDecode, 3);
            vf[2 * r] = in ? ld_stream(src) : make_uint4(0u, 0u, 0u, 0u);
            vf[2 * r + 1] = in ? ld_stream(src + 8) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    if (u < nunits) { load_k(u); load_v(u); }
    for (int i = tid; i < kDecMaxGroup * kD; i += kThreads) {   // (q may be aligned to 2 bytes only)
        const int src = DUP ? i & (4 * kD - 1) : i;
        sm.q[i] = src < group * kD && JQ_IN(kv * group * kD + src, (long long)(gridDim.x / C) * group * kD, kDbgDecode, 2)
                      ? q[(size_t)kv * group * kD + src] : __float2bfloat16(0.f);
    }
    __syncthreads();
    uint4 qf[4];                       // of head (column) g, permuted like the keys
#pragma unroll
    for (int i = 0; i < 4; ++i) qf[i] = *((const uint4 *)(sm.q + g * kD) + t + 4 * i);

    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};   // of columns 2t, 2t + 1: m is the warp's, l the lane's own part
    float o[8][4];                     // [i]: dimensions 8g + i (columns 2t, 2t + 1) and 64 + 8g + i (the same columns)
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
#pragma unroll 1
    for (; u < nunits; u += stride) {
        float sa[4] = {0.f, 0.f, 0.f, 0.f}, sb[4] = {0.f, 0.f, 0.f, 0.f};   // keys g and 8 + g, columns 2t and 2t + 1
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            mma_bf16(sa, kf[i].x, kf[4 + i].x, kf[i].y, kf[4 + i].y, qf[i].x, qf[i].y);
            mma_bf16(sb, kf[i].z, kf[4 + i].z, kf[i].w, kf[4 + i].w, qf[i].z, qf[i].w);
        }
        if (u + stride < nunits) load_k(u + stride);   // in flight while this unit is finished
        float x[4];                                    // [key g: 2 columns][key 8 + g: 2 columns]
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = (sa[i] + sb[i]) * scale_log2;
        if (u == nunits - 1) {
            const int j0 = u * kDecUnit + g;
            if (j0 >= n) x[0] = x[1] = -INFINITY;
            if (j0 + 8 >= n) x[2] = x[3] = -INFINITY;
        }
        float f[2], p[4];
        bool moved = false;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float mx = fmaxf(x[c], x[2 + c]);
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));   // a unit holds at least one key: finite
            const float mn = fmaxf(m[c], mx);
            moved |= mn > m[c];
            f[c] = dec_ex2(m[c] - mn);
            m[c] = mn;
            p[c] = dec_ex2(x[c] - mn);
            p[2 + c] = dec_ex2(x[2 + c] - mn);
            l[c] = fmaf(l[c], f[c], p[c] + p[2 + c]);
        }
        uint32_t hi[2], mid[2], lo[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            hi[r] = pack_bf16(p[2 * r], p[2 * r + 1]);
            const float r0 = p[2 * r] - bf16_lo(hi[r]), r1 = p[2 * r + 1] - bf16_hi(hi[r]);
            mid[r] = pack_bf16(r0, r1);
            lo[r] = pack_bf16(r0 - bf16_lo(mid[r]), r1 - bf16_hi(mid[r]));
            if (DUP && t >= 2) { hi[r] = mid[r]; lo[r] = 0u; }      // the repeated columns carry the middle part
            hi[r] = transpose8x8(hi[r]);
            lo[r] = transpose8x8(lo[r]);
            if (!DUP) mid[r] = transpose8x8(mid[r]);
        }
        if (__any_sync(0xffffffffu, moved)) {
#pragma unroll
            for (int i = 0; i < 8; ++i) { o[i][0] *= f[0]; o[i][1] *= f[1]; o[i][2] *= f[0]; o[i][3] *= f[1]; }
        }
        const uint32_t *v = (const uint32_t *)vf;      // [row r][half][4]: two dimensions each
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t sel = (i & 1) ? 0x7632u : 0x5410u;
            const uint32_t a0 = __byte_perm(v[i >> 1], v[8 + (i >> 1)], sel), a1 = __byte_perm(v[4 + (i >> 1)], v[12 + (i >> 1)], sel);
            const uint32_t a2 = __byte_perm(v[16 + (i >> 1)], v[24 + (i >> 1)], sel), a3 = __byte_perm(v[20 + (i >> 1)], v[28 + (i >> 1)], sel);
            mma_bf16(o[i], a0, a1, a2, a3, lo[0], lo[1]);
            if (!DUP) mma_bf16(o[i], a0, a1, a2, a3, mid[0], mid[1]);
            mma_bf16(o[i], a0, a1, a2, a3, hi[0], hi[1]);
        }
        if (u + stride < nunits) load_v(u + stride);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 4);
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 8);
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 16);
    }

    // ---- the warps of the CTA
    if (g == 0) {
        sm.m[warp][2 * t] = m[0]; sm.m[warp][2 * t + 1] = m[1];
        sm.l[warp][2 * t] = l[0]; sm.l[warp][2 * t + 1] = l[1];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float *dst = &sm.O[warp][2 * t + (c & 1)][64 * (c >> 1) + 8 * g];
        *(float4 *)dst = make_float4(o[0][c], o[1][c], o[2][c], o[3][c]);
        *(float4 *)(dst + 4) = make_float4(o[4][c], o[5][c], o[6][c], o[7][c]);
    }
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // every CTA of the cluster runs: its memory may be written
    const int items = group * kD, share = (items + (int)C - 1) / (int)C;
    for (int it = tid; it < items; it += kThreads) {
        const int h = it / kD, c = it - h * kD;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) M = fmaxf(M, sm.m[w][h]);
        float O = 0.f, Ls = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            // a warp without keys has m = -inf and adds nothing (M is -inf too when the whole CTA has none)
            const float f = sm.m[w][h] > -INFINITY ? dec_ex2(sm.m[w][h] - M) : 0.f;
            O = fmaf(DUP ? sm.O[w][h][c] + sm.O[w][h + 4][c] : sm.O[w][h][c], f, O);
            Ls = fmaf(sm.l[w][h], f, Ls);
        }
        const int to = it / share;
        push_f32(&sm.rO[(int)rank * share + (it - to * share)], (uint32_t)to, O);
        if (c < (int)C) { push_f32(&sm.rm[rank][h], (uint32_t)c, M); push_f32(&sm.rl[rank][h], (uint32_t)c, Ls); }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    for (int i = tid; i < share; i += kThreads) {
        const int it = (int)rank * share + i, h = it / kD;
        if (it >= items) break;
        float M = -INFINITY, O = 0.f, Ls = 0.f;
        for (int r = 0; r < (int)C; ++r) M = fmaxf(M, sm.rm[r][h]);
        for (int r = 0; r < (int)C; ++r) {
            const float f = sm.rm[r][h] > -INFINITY ? dec_ex2(sm.rm[r][h] - M) : 0.f;
            O = fmaf(sm.rO[r * share + i], f, O);
            Ls = fmaf(sm.rl[r][h], f, Ls);
        }
        if (JQ_IN((long long)kv * items + it, (long long)(gridDim.x / C) * items, kDbgDecode, 4)) out[(size_t)kv * items + it] = O / Ls;
    }
}

// CTAs per KV head: the cluster size that the estimate below finds fastest.  A cluster takes about 3.3 us of launch,
// merge and latency and 1 us for each unit its busiest warp walks through, and only so many clusters of a size are
// resident at a time (a cluster stays within a GPC: 148, 45, 33, 22, 15, 11, 7 of 1, 3, 4, 6, 8, 10, 16 CTAs; asked for once
// per device).
// Measured against it: 8 heads x 1024 keys 11.3, 7.5, 5.6, 4.3 us with 1, 2, 4, 8 CTAs; 128 x 2048 27, 30, 37, 56;
// 24 x 3000 30.5, 17.9, 11.8, 15.6 and 11.1 with 5; 20 x 3000 11.5, 9.6 with 4, 6; 36 x 2000 14.8, 12.8 with 2, 3; 7 x 4096
// 34, -, 11.7, 7.9 and 5.9 with 16.
struct DecPlan { int resident[kDecMaxCluster + 1] = {}; bool ready = false; };   // [C]: resident clusters of C CTAs

bool decode_plan(DecPlan *out)
{
    static DecPlan plans[64];
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lock(mu);
    DecPlan &p = plans[dev];
    if (!p.ready) {
        for (auto k : {decode_step<true, kDecWarps>, decode_step<false, kDecWarps>, decode_step<true, kDecManyWarps>, decode_step<false, kDecManyWarps>})
            if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
        for (auto k : {decode_step<true, kDecManyWarps>, decode_step<false, kDecManyWarps>})   // (eight warps need less than 48 KB)
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecSmem<kDecManyWarps>)) != cudaSuccess) return false;
        for (int C = 1; C <= kDecMaxCluster; ++C) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)C);
            cfg.blockDim = dim3(32 * kDecManyWarps);
            cfg.dynamicSmemBytes = sizeof(DecSmem<kDecManyWarps>);
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&p.resident[C], decode_step<true, kDecManyWarps>, &cfg) != cudaSuccess) { cudaGetLastError(); p.resident[C] = 0; }
        }
        if (p.resident[1] < 1) return false;
        p.ready = true;
    }
    *out = p;
    return true;
}

// A CTA has eight warps or twelve: with twelve more of the cache is on its way at a time, which pays where a warp walks through several
// units (the loop is bound by what a CTA has in flight, 8 KB per warp; a round of units then takes 1.3 times as long), and the merge
// is larger.  Measured with 8 and 12 warps: 128 heads x 2048 keys 27.2, 25.2 us, 100 x 3000 35.3, 30.1, 90 x 2048 25.8, 22.0,
// 140 x 4096 49.7, 46.7, 128 x 512 10.9, 10.7; 8 x 1024 5.1, 5.6, 149 x 256 13.1, 13.5.  (Ten: 26.0, 32.1, 23.3, 48.2.)
struct DecShape { int C; bool many; };
DecShape decode_shape(int Hkv, int n, const DecPlan &p)
{
    const int nunits = (n + kDecUnit - 1) / kDecUnit;
    DecShape best = {1, false};
    double best_cost = 1e30;
    for (int many = 0; many < 2; ++many)
        for (int C = 1; C <= kDecMaxCluster; ++C) {
            if (p.resident[C] < 1) continue;
            const int per = (many ? kDecManyWarps : kDecWarps) * C, units = (nunits + per - 1) / per, rounds = (Hkv + p.resident[C] - 1) / p.resident[C];
            const double cost = rounds * (many ? 3.35 + 1.3 * units : 3.3 + units) + (rounds > 1 ? 1.0 : 0.0);
            // (a second round of heads has a start and a merge of its own: 75, 80, 90 heads x 2048 keys take 20.9, 21.6, 21.7 us with a CTA
            // of twelve warps each, 21.4, 22.0, 23.1 with three in two rounds, which would win by a little without it;
            // at equal cost a power of two: the outputs then divide evenly over the CTAs)
            if (cost < best_cost || (cost == best_cost && (C & (C - 1)) == 0 && (best.C & (best.C - 1)) != 0)) { best = {C, many != 0}; best_cost = cost; }
            if (units == 1) break;   // (more CTAs have nothing to do)
        }
    return best;
}

}  // namespace
}  // namespace jq

extern "C" size_t jq_decode_workspace_bytes(int Hkv, int Hq, int n)
{
    if (Hkv < 1 || Hq < 1 || Hq % Hkv || Hq / Hkv > jq::kDecMaxGroup || n < 1) return 0;
    const size_t nsplit = ((size_t)n + jq::kDecChunk - 1) / jq::kDecChunk;
    return jq::align_up((size_t)Hq * nsplit * jq::kPartial * sizeof(float), 256) + jq::align_up((size_t)Hkv * sizeof(unsigned int), 256);
}

extern "C" jq_status jq_decode_attention(const void *Kc, const void *Vc, const void *q, int Hkv, int Hq, int n, float *out,
                                         void *workspace, size_t workspace_bytes, jq_stream_t stream)
{
    using namespace jq;
    if (!Kc || !Vc || !q || !out || Hkv < 1 || Hq < 1 || n < 1 || Hq % Hkv) return JQ_ERR_INVALID_ARG;
    if (((uintptr_t)Kc | (uintptr_t)Vc | (uintptr_t)out | (uintptr_t)workspace) & 15u) return JQ_ERR_INVALID_ARG;
    if (((uintptr_t)q) & 1u) return JQ_ERR_INVALID_ARG;
    const int group = Hq / Hkv;
    if (group > kDecMaxGroup || Hkv > 65535) return JQ_ERR_UNSUPPORTED;
    const size_t need = jq_decode_workspace_bytes(Hkv, Hq, n);
    if (!workspace || workspace_bytes < need) return JQ_ERR_WORKSPACE;
    DecPlan plan;
    if (!decode_plan(&plan)) return JQ_ERR_CUDA;
    const DecShape shape = decode_shape(Hkv, n, plan);
    const int C = shape.C;
    const bool many = shape.many;
    const float scale_log2 = 1.4426950408889634f / sqrtf((float)kD);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(Hkv * C));
    cfg.blockDim = dim3(32 * (many ? kDecManyWarps : kDecWarps));
    cfg.dynamicSmemBytes = many ? sizeof(DecSmem<kDecManyWarps>) : sizeof(DecSmem<kDecWarps>);
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // the kernel waits for the one before it in the stream
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, many ? (group <= 4 ? decode_step<true, kDecManyWarps> : decode_step<false, kDecManyWarps>)
                                         : (group <= 4 ? decode_step<true, kDecWarps> : decode_step<false, kDecWarps>), (const uint4 *)Kc, (const uint4 *)Vc, (const __nv_bfloat16 *)q, n, group, scale_log2,
                           out JQ_DBG_ARG) != cudaSuccess) {
        cudaGetLastError();
        return JQ_ERR_CUDA;
    }
    count_launch(1);
    return check_launch();
}
