// Max-pooling and order keys, shared by the selection kernels (jq_select.cu, jq_fused.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace jq {
namespace {

// Order-preserving integer key of a score (float order == unsigned order).
__device__ __forceinline__ uint32_t order_key(float x)
{
    uint32_t b = __float_as_uint(x + 0.0f);  // -0 -> +0
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}

// Pooled order keys (and values) of the four positions of quad b, whose neighbours are a and c; radius <= 4.
__device__ __forceinline__ void pooled_quad(const float4 a, const float4 b, const float4 c, int radius, uint32_t (&key)[4], float (&best)[4])
{
    const float x[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
    if (radius == 3) {
        // window of 7: the four windows share x4..x7; the rest are running maxima of the three neighbours on either side
        const float core = fmaxf(max3f(x[4], x[5], x[6]), x[7]);
        const float l2 = fmaxf(x[2], x[3]), l1 = fmaxf(x[1], l2);
        const float r9 = fmaxf(x[8], x[9]), r10 = fmaxf(r9, x[10]);
        best[0] = fmaxf(core, l1);
        best[1] = max3f(core, l2, x[8]);
        best[2] = max3f(core, x[3], r9);
        best[3] = fmaxf(core, r10);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float m = x[4 + i];
#pragma unroll
            for (int u = 1; u <= 4; ++u) if (u <= radius) m = fmaxf(m, fmaxf(x[4 + i - u], x[4 + i + u]));
            best[i] = m;
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) key[i] = order_key(best[i]);
}

}  // namespace
}  // namespace jq
