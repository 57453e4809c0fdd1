// Compensated FP64 sums of term values, shared by the result kernels of the
// sweep engine (kernels_reduce.cu) and of the general-noise path (generic.cu).
//
// A block adds each level's terms in a fixed order: lane-strided Neumaier
// sums, then pairs (sum, compensation) combined by error-free two-sums through
// shuffles and one shared-memory step.  What bounds this is the latency of
// dependent FP64 operations (the chip has few FP64 units): one thread adding
// the 256 partial sums of every level one after another took 221 us for the
// 1771 terms of three levels, the tree 10 us.  Levels of at most kWarpTerms
// terms are added by one warp each, all at once; longer ones by the whole
// block, one after another.
#pragma once

#include <cuda_runtime.h>

#include "../../include/nqs.h"

namespace nqs {

constexpr int kSumThreads = 256;
constexpr long long kWarpTerms = 512;

struct CompSum {
    double s, c;   // sum and its compensation
};

__device__ __forceinline__ void neumaier_add(CompSum& a, double x) {
    const double t = a.s + x;
    a.c += (fabs(a.s) >= fabs(x)) ? (a.s - t) + x : (x - t) + a.s;
    a.s = t;
}

__device__ __forceinline__ CompSum comp_join(CompSum a, CompSum b) {
    neumaier_add(a, b.s);
    a.c += b.c;
    return a;
}

__device__ __forceinline__ CompSum warp_join(CompSum a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        CompSum b;
        b.s = __shfl_down_sync(0xffffffffu, a.s, o);
        b.c = __shfl_down_sync(0xffffffffu, a.c, o);
        a = comp_join(a, b);
    }
    return a;   // lane 0 holds the whole warp's
}

// T[u] (shared memory) for every level; term(i) gives term i's value.  Called
// by a block of kSumThreads threads; ends with a barrier.
template <typename TermFn>
__device__ void level_sums(const long long* __restrict__ level_off, int level, TermFn term, double* T) {
    __shared__ double ps[kSumThreads / 32], pc[kSumThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int u = warp; u <= level; u += kSumThreads / 32) {
        const long long lo = level_off[u], hi = level_off[u + 1];
        if (hi - lo > kWarpTerms) continue;
        CompSum a{0.0, 0.0};
        for (long long i = lo + lane; i < hi; i += 32) neumaier_add(a, term(i));
        a = warp_join(a);
        if (lane == 0) T[u] = a.s + a.c;
    }
    for (int u = 0; u <= level; ++u) {
        const long long lo = level_off[u], hi = level_off[u + 1];
        if (hi - lo <= kWarpTerms) continue;
        CompSum a{0.0, 0.0};
        for (long long i = lo + tid; i < hi; i += kSumThreads) neumaier_add(a, term(i));
        a = warp_join(a);
        if (lane == 0) {
            ps[warp] = a.s;
            pc[warp] = a.c;
        }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < kSumThreads / 32; ++w) a = comp_join(a, CompSum{ps[w], pc[w]});
            T[u] = a.s + a.c;
        }
        __syncthreads();
    }
    __syncthreads();
}

// F and the per-level sums of a result record (one thread)
__device__ __forceinline__ void store_levels(nqs_result* res, const double* T, int level) {
    CompSum f{0.0, 0.0};
    for (int u = 0; u <= NQS_MAX_LEVEL; ++u) {
        res->T[u] = u <= level ? T[u] : 0.0;
        if (u <= level) neumaier_add(f, T[u]);
    }
    res->F = f.s + f.c;
}

}  // namespace nqs
