// Wrappers and device functions that the two scoring kernels (jq_score_tc.cu, jq_fused.cu) share: mbarriers with
// bounded waits, TMA loads, tcgen05 issue, and the exponential stream with its row statistics.
#pragma once
#include <cuda.h>
#include "jq_internal.cuh"

namespace jq {
namespace {

constexpr long long kWaitCycles = 4000000000ll;  // about 2 s of SM clock per wait
constexpr int kWStatus = 0;                      // the status word of the workspace's status block

// ------------------------------------------------------------------ PTX wrappers

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// One look at the barrier, no waiting.
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  false: the wait ran out (status recorded) or another thread of the CTA aborted.
// A waiter that can afford it sleeps `sleep_ns` between polls: a spinning warp takes issue slots and
// queue entries of the shared-memory pipe away from the epilogue warps on its scheduler.  The clock is
// only consulted after many failed polls, so a normal wait never pays for it.
__device__ __noinline__ bool mbar_wait_slow(uint64_t *bar, uint32_t parity, int *abort_flag, int *status, uint32_t sleep_ns)
{
    if (*(volatile int *)abort_flag) return false;
    for (int i = 0; i < 2048; ++i) {
        if (mbar_try(bar, parity)) return true;
        if (sleep_ns) __nanosleep(sleep_ns);
    }
    const long long t0 = clock64();
    for (;;) {
        for (int i = 0; i < 64; ++i) {
            if (mbar_try(bar, parity)) return true;
            if (sleep_ns) __nanosleep(sleep_ns);
        }
        if (*(volatile int *)abort_flag) return false;
        if (clock64() - t0 > kWaitCycles) {
            *(volatile int *)abort_flag = 1;
            atomicMax(status + kWStatus, (int)JQ_ERR_TIMEOUT);
            return false;
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, int *abort_flag, int *status, uint32_t sleep_ns = 0)
{
    if (mbar_try(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, abort_flag, status, sleep_ns);
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

// The same with an L2 eviction policy (createpolicy).
__device__ __forceinline__ void tma_load_3d_hint(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
        ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "l"(policy) : "memory");
}

// A tensor map that the host wrote into global memory (with an ordinary copy) must be acquired by the
// tensor-map proxy before a TMA instruction of this CTA reads it.
__device__ __forceinline__ void tensormap_acquire(const CUtensorMap *map)
{
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Issued by ONE lane of a converged warp (the whole warp runs the issuing code so that its address
// arithmetic stays warp-uniform; only the tensor-core instructions themselves are predicated).
__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    __syncwarp();
    asm volatile(
        "{\n\t.reg .pred pe;\n\t"
        "elect.sync _|pe, 0xffffffff;\n\t"
        "@pe tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        ::"r"(smem_u32(bar)) : "memory");
}

// Instruction descriptor, kind::f16: D fp32, A and B bf16, both K-major, shape M x N.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float max3(float a, float b, float c)
{
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, rows of 128 bytes, 8-row groups 1024
// bytes apart (stride byte offset), leading byte offset 16 (unused for swizzled K-major), version 1.
// Only the low word depends on the address (in 16-byte units); the high word is a constant.
constexpr uint32_t kDescHi = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3fffu) | (1u << 16); }

// One accumulator block: D[tmem] = A[smem] * B[smem]^T over the whole head dimension (8 steps of 16),
// both operands K-major bf16 in two 64-column halves `a_half` / `b_half` bytes apart, fp32 accumulate.
// A single straight-line sequence run by the whole (converged) warp with one elected lane issuing: the
// warp shares its scheduler with epilogue warps, so every instruction it does not execute is time the
// tensor pipe does not wait.
__device__ __forceinline__ void tc_mma_block(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t a_half,
                                             uint32_t b_half, uint32_t idesc)
{
    const uint32_t a1 = a_lo + (a_half >> 4), b1 = b_lo + (b_half >> 4);
    __syncwarp();
    asm volatile(
        "{\n\t"
        ".reg .pred pz, po, pe;\n\t"
        ".reg .b64 da, db;\n\t"
        ".reg .b32 ta, tb;\n\t"
        "setp.ne.u32 pz, %0, %0;\n\t"
        "setp.eq.u32 po, %0, %0;\n\t"
        "elect.sync _|pe, 0xffffffff;\n\t"
        "mov.b64 da, {%1, %5};\n\t mov.b64 db, {%2, %5};\n\t"
        "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, pz;\n\t"
        "add.u32 ta, %1, 2;\n\t add.u32 tb, %2, 2;\n\t mov.b64 da, {ta, %5};\n\t mov.b64 db, {tb, %5};\n\t"
        "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, po;\n\t"
        "add.u32 ta, %1, 4;\n\t add.u32 tb, %2, 4;\n\t mov.b64 da, {ta, %5};\n\t mov.b64 db, {tb, %5};\n\t"
        "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, po;\n\t"
        "add.u32 ta, %1, 6;\n\t add.u32 tb, %2, 6;\n\t mov.b64 da, {ta, %5};\n\t mov.b64 db, {tb, %5};\n\t"
        "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, po;\n\t"
        "mov.b64 da, {%3, %5};\n\t mov.b64 db, {%4, %5};\n\t"
        "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, po;\n\t"
        "add.u32 ta, %3, 2;\n\t add.u32 tb, %4, 2;\n\t mov.b64 da, {ta, %5};\n\t mov.b64 db, {tb, %5};\n\t"
        "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, po;\n\t"
        "add.u32 ta, %3, 4;\n\t add.u32 tb, %4, 4;\n\t mov.b64 da, {ta, %5};\n\t mov.b64 db, {tb, %5};\n\t"
        "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, po;\n\t"
        "add.u32 ta, %3, 6;\n\t add.u32 tb, %4, 6;\n\t mov.b64 da, {ta, %5};\n\t mov.b64 db, {tb, %5};\n\t"
        "@pe tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, po;\n\t"
        "}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(a1), "r"(b1), "r"(kDescHi), "r"(idesc) : "memory");
}

// ------------------------------------------------------------------ exponentials

// acc += exp2(v * c + b) for two values.  All of them on the ex2 unit: a share on the FMA pipe (round, polynomial, exponent
// insertion) shortened the stream by itself, but sustained scoring runs at the GPU's power limit (1000 W), and the ten
// instructions of a polynomial pair cost more energy than they saved time: with 2 of 8 pairs on the FMA pipe 32 layers of
// 32768 keys took 1071 us, with 1 of 8 1055, with none 1037 (128K keys, 256 rows: 6292, 6230, 6258).
__device__ __forceinline__ void exp_acc2(float2 &acc, uint32_t v0, uint32_t v1, float2 cc, float2 b)
{
    const float2 x = __ffma2_rn(make_float2(__uint_as_float(v0), __uint_as_float(v1)), cc, b);
    acc = __fadd2_rn(acc, make_float2(ex2(x.x), ex2(x.y)));
}

// 16 values against 16 biases (pass 2: the negated row normalisers, from shared memory).
__device__ __forceinline__ void exp_acc16(float2 &a0, float2 &a1, const uint32_t (&v)[16], float2 cc, const float4 *bias)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 b = bias[i];
        exp_acc2(a0, v[4 * i], v[4 * i + 1], cc, make_float2(b.x, b.y));
        exp_acc2(a1, v[4 * i + 2], v[4 * i + 3], cc, make_float2(b.z, b.w));
    }
}

// 16 values against one bias (pass 1: minus the reference of the row).
__device__ __forceinline__ void exp_acc16(float2 &a0, float2 &a1, const uint32_t (&v)[16], float2 cc, float2 b)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        exp_acc2(a0, v[4 * i], v[4 * i + 1], cc, b);
        exp_acc2(a1, v[4 * i + 2], v[4 * i + 3], cc, b);
    }
}

__device__ __forceinline__ float max_of16(const uint32_t (&v)[16])
{
    float c0 = -INFINITY, c1 = -INFINITY;
#pragma unroll
    for (int t = 0; t < 16; t += 4) {
        c0 = max3(c0, __uint_as_float(v[t + 0]), __uint_as_float(v[t + 1]));
        c1 = max3(c1, __uint_as_float(v[t + 2]), __uint_as_float(v[t + 3]));
    }
    return fmaxf(c0, c1);
}

// Pass 1, 16 keys of a query row: online softmax statistics (m, l = sum_j exp2(c (s_j - m))).  Any
// reference m gives the same row normaliser c m + log2 l as long as nothing overflows, so m is not kept
// equal to the running max: it is raised (and l rescaled) only when the keys bring a value more than
// `lazy` above it, lazy = 64 / c, i.e. when an exponential would pass 2^64.  A warp of 32 rows restarts
// its statistics at every segment and would otherwise take the rescaling branch on most reads; now it
// takes it once per segment.  (exp2 arguments reach +64 at most, l stays below 2^64 times the keys of
// a segment: far inside fp32.)  The max runs on the ALU pipe and, unlike a check of the sum, does not
// wait for the exponentials in flight.  Keys at column >= valid are not keys (-inf).
struct RowState { float m; float2 l01, l23; };
__device__ __forceinline__ void p1_half(uint32_t (&v)[16], int c0, int valid, float c, float lazy, float2 cc, RowState &st)
{
    if (valid < c0 + 16) {
#pragma unroll
        for (int t = 0; t < 16; ++t) if (c0 + t >= valid) v[t] = 0xff800000u;
    }
    const float cm = max_of16(v);
    if (cm > st.m + lazy) {
        const float f = ex2(c * (st.m - cm));   // 0 for the first keys (m = -inf)
        st.l01 = make_float2(st.l01.x * f, st.l01.y * f);
        st.l23 = make_float2(st.l23.x * f, st.l23.y * f);
        st.m = cm;
    }
    const float nb = -st.m * c;
    exp_acc16(st.l01, st.l23, v, cc, make_float2(nb, nb));
}

// x / d for x < 2^25 with magic = ceil(2^32 / d) computed on the host: one multiplication and a correction
// instead of the compiler's division sequence (dozens of instructions and a reciprocal that would queue behind
// the exponentials in the special-function unit; every role runs the schedule arithmetic once per segment).
__device__ __forceinline__ uint32_t fast_div(uint32_t x, uint32_t d, uint32_t magic)
{
    uint32_t q = __umulhi(x, magic);
    if (q * d > x) --q;          // for d > 1 the estimate is never low and at most one high
    if ((q + 1) * d <= x) ++q;   // d == 1 (magic 2^32 - 1): one low
    return q;
}

}  // namespace
}  // namespace jq
