// The copy of the kept rows, shared by the selection kernels (jq_select.cu, jq_prune.cu).
#pragma once
#include "jq_internal.cuh"
#include "jq_debug.cuh"

namespace jq {
namespace {

// Extents of what the kernel indexes (read by the bounds-checked build only).
struct SelExtents {
    long long scores;     // floats in the scores array (and keys in the global key array)
    long long out_rows;   // rows of the stacked outputs (kept indices, compacted K and V)
    long long src_heads;  // heads in one source buffer of K / V
};

// The window rows that follow every head's kept rows: K, V [Hkv][w] rows (w = 0: none).
struct WindowRows { const uint4 *K, *V; int w; };

// Rows [r0, r1) of a head's kept rows (256 bytes each: 16 lanes x 16 bytes), four rows of K and V in flight per 16 lanes.
// tid: of the `threads` that share the rows; kv_in: the head's index within the buffer the rows come from; orow: the head's first row in the outputs.
__device__ __forceinline__ void copy_rows(int tid, int threads, const int32_t *out, int r0, int r1, int kv_in, long long orow, int L, const uint4 *__restrict__ Kin,
                                          const uint4 *__restrict__ Vin, uint4 *__restrict__ Kout, uint4 *__restrict__ Vout, int src_rows,
                                          const SelExtents &ext JQ_DBG_PARAM)
{
    (void)ext;
    const int lane16 = tid & 15, grp = tid >> 4, ngrp = threads >> 4;
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

}  // namespace
}  // namespace jq
