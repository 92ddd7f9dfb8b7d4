// Sums over the entries of sparse rows, split by the rows' lengths.  A thread
// alone on a row pays about a memory latency per few entries, so a row of
// thousands of entries (a dense row of A) on one thread outlasts everything
// beside it, and a warp or CTA on a row of five entries idles.  One launch
// serves three classes by block range: rows of up to kWarpRow entries one
// thread each (in entry order), up to kLongColumn a warp each, longer ones a
// CTA each (lanes stride the entries, so the loads are coalesced; the lanes'
// sums are added in a fixed tree, so the result does not depend on
// scheduling).  On 40 block-angular blocks with 300 dense rows (rows of 303
// and of 16,000 entries) the residual takes 0.10 ms instead of 0.44.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "ipm_dev.h"

namespace ipm {
namespace rows {

constexpr int kThreads = 256;

// Blocks of a launch over all three classes; `shorts` rows are visited by the
// thread-per-row blocks (which skip the longer ones).
inline int grid(int32_t shorts, int32_t nmid, int32_t nlong) {
    const int s = (shorts + kThreads - 1) / kThreads;
    return nlong + (nmid + kThreads / 32 - 1) / (kThreads / 32) + (s < 1 ? 1 : s < 608 ? s : 608);
}

// What this block does: a long row's index in the list (cta), the first
// medium row of its eight warps (mid), or its place among the short blocks.
struct Part {
    int cta, mid, first, stride;
};
__device__ __forceinline__ Part part(int nmid, int nlong) {
    const int b = blockIdx.x, mb = (nmid + kThreads / 32 - 1) / (kThreads / 32);
    Part p{-1, -1, 0, 0};
    if (b < nlong) {
        p.cta = b;
    } else if (b < nlong + mb) {
        p.mid = (b - nlong) * (kThreads / 32) + (threadIdx.x >> 5);
    } else {
        p.first = (b - nlong - mb) * kThreads + threadIdx.x;
        p.stride = (gridDim.x - nlong - mb) * kThreads;
    }
    return p;
}

// a[0..NA) summed over the warp, every lane with the result.
template <int NA>
__device__ __forceinline__ void warp_add(double (&a)[NA]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < NA; c++) a[c] += __shfl_xor_sync(0xffffffffu, a[c], o);
}

// a[0..NA) summed over the CTA, thread 0 with the result (one CTA barrier).
template <int NA>
__device__ __forceinline__ void cta_add(double (&a)[NA], double (*sh)[NA]) {
    warp_add(a);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int c = 0; c < NA; c++) sh[threadIdx.x >> 5][c] = a[c];
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kThreads / 32; w++)
#pragma unroll
            for (int c = 0; c < NA; c++) a[c] += sh[w][c];
}

}  // namespace rows
}  // namespace ipm
