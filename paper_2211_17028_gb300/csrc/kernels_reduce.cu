// Reductions and bookkeeping kernels: the standalone reduced-matrix kernel,
// the fixed-order finishers that turn per-block partial sums into term
// values, the Neumaier-compensated per-level sums, and the basis-state fill.
#include "level_sum.cuh"
#include "sweep_types.h"
#include "nqs_internal.h"

namespace nqs {

// Standalone reduced-matrix kernel (nqs_reduced_matrix and the N = 0 path):
// grid-stride over amplitude pairs of qubit q.
__global__ void __launch_bounds__(kThreads) reduce2x2_kernel(const float2* __restrict__ phi,
                                                             const float2* __restrict__ chi, int n, int q,
                                                             double* __restrict__ partials) {
    __shared__ double acc[kWarps][8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < kWarps * 8) (&acc[0][0])[tid] = 0.0;
    __syncthreads();
    const long long npairs = 1ll << (n - 1);
    const long long bit = 1ll << q;
    const long long stride = (long long)gridDim.x * kThreads;
    long long p = (long long)blockIdx.x * kThreads + tid;
    while (__any_sync(0xffffffffu, p < npairs)) {
        float r[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int it = 0; it < 16 && p < npairs; ++it, p += stride) {
            long long lo = p & (bit - 1);
            long long i0 = ((p - lo) << 1) | lo, i1 = i0 | bit;
            float2 f0 = __ldcs(phi + i0), f1 = __ldcs(phi + i1);
            float2 x0 = __ldcs(chi + i0), x1 = __ldcs(chi + i1);
            r[0] += f0.x * x0.x + f0.y * x0.y;  r[1] += f0.x * x0.y - f0.y * x0.x;
            r[2] += f0.x * x1.x + f0.y * x1.y;  r[3] += f0.x * x1.y - f0.y * x1.x;
            r[4] += f1.x * x0.x + f1.y * x0.y;  r[5] += f1.x * x0.y - f1.y * x0.x;
            r[6] += f1.x * x1.x + f1.y * x1.y;  r[7] += f1.x * x1.y - f1.y * x1.x;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float v = r[e];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane == 0) acc[warp][e] += (double)v;
        }
    }
    __syncthreads();
    if (tid < 8) {
        double v = 0.0;
        for (int w = 0; w < kWarps; ++w) v += acc[w][tid];
        partials[(size_t)blockIdx.x * 8 + tid] = v;
    }
}

// One warp per reduction slot: the per-block partial sums in a fixed order
// (lane l takes component l % 8 of blocks l / 8, l / 8 + 4, ...: whole 64-byte
// rows per load, four loads in flight; two shuffles join the four rows), then
// X = |sum_ab K[a][b] R[a][b]|^2 for each factor of the slot.  Latency-bound;
// one launch serves all reductions since the last one (as a launch behind
// every pass it was 109 launches of 8.4 us in a 20-qubit level-2 call).
__device__ __forceinline__ void finish_slot(const double* __restrict__ partials, const FinishSlot& s,
                                            const double* __restrict__ kmats, double* __restrict__ term_vals,
                                            double* R) {
    const int lane = threadIdx.x & 31;
    const double* const part = partials + s.part + (lane & 7);
    double v = 0.0;
    int b = lane >> 3;
    for (; b + 12 < s.grid; b += 16) {
        const double p0 = part[(size_t)b * 8], p1 = part[(size_t)(b + 4) * 8];
        const double p2 = part[(size_t)(b + 8) * 8], p3 = part[(size_t)(b + 12) * 8];
        v += (p0 + p1) + (p2 + p3);
    }
    for (; b < s.grid; b += 4) v += part[(size_t)b * 8];
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    if (lane < 8) R[lane] = v;
    __syncwarp();
    if (lane < 4) {
        const FinishDesc d = s.d[lane];
        if (d.rank >= 0) {
            const double* K = kmats + d.kmat;
            double re = 0, im = 0;
            for (int e = 0; e < 4; ++e) {
                double kr = K[2 * e], ki = K[2 * e + 1], rr = R[2 * e], ri = R[2 * e + 1];
                re += kr * rr - ki * ri;
                im += kr * ri + ki * rr;
            }
            term_vals[d.rank] = re * re + im * im;
        }
    }
}

__global__ void __launch_bounds__(kThreads) finish_kernel(const double* __restrict__ partials,
                                                          const FinishSlot* __restrict__ slots,
                                                          const double* __restrict__ kmats,
                                                          double* __restrict__ term_vals, int n_slots) {
    __shared__ double R[kWarps][8];
    const int warp = threadIdx.x >> 5, slot = blockIdx.x * kWarps + warp;
    if (slot < n_slots) finish_slot(partials, slots[slot], kmats, term_vals, R[warp]);
}

// finishers of many circuits: unit u owns blocks [blk_begin[u], blk_begin[u+1])
__global__ void __launch_bounds__(kThreads) finish_kernel_batched(const FinishUnit* __restrict__ units,
                                                                  const int* __restrict__ blk_begin, int n_units) {
    __shared__ double R[kWarps][8];
    int lo = 0, hi = n_units;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (blk_begin[mid] <= (int)blockIdx.x) lo = mid;
        else hi = mid;
    }
    const FinishUnit u = units[lo];
    const int warp = threadIdx.x >> 5, slot = ((int)blockIdx.x - blk_begin[lo]) * kWarps + warp;
    if (slot < u.n_slots) finish_slot(u.partials, u.slots[slot], u.kmats, u.vals, R[warp]);
}

// One block: fixed-order sum of per-block partials into 8 doubles.
__global__ void __launch_bounds__(kThreads) partials_sum_kernel(const double* __restrict__ part, int grid,
                                                                double* __restrict__ R) {
    // thread t takes component t % 8 of blocks t / 8, t / 8 + 32, ...; two
    // shuffles join the rows of a warp, eight threads add the warps' sums
    __shared__ double scratch[kWarps][8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double v = 0.0;
    for (int b = tid >> 3; b < grid; b += kThreads / 8) v += part[(size_t)b * 8 + (tid & 7)];
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    if (lane < 8) scratch[warp][lane] = v;
    __syncthreads();
    if (tid < 8) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) t += scratch[w][tid];
        R[tid] = t;
    }
}

// Neumaier-compensated per-level sums (level_sum.cuh), one block.
__device__ __forceinline__ void level_sum_body(const double* __restrict__ vals,
                                               const long long* __restrict__ level_off, int level,
                                               nqs_result* __restrict__ res, double bound, long long n_terms,
                                               const int* __restrict__ err, nqs_result* __restrict__ copy) {
    __shared__ double T[NQS_MAX_LEVEL + 1];
    level_sums(level_off, level, [&](long long i) { return vals[i]; }, T);
    if (threadIdx.x == 0) {
        store_levels(res, T, level);
        res->imag_residual = 0.0;
        res->n_terms = (uint64_t)n_terms;
        res->bound = bound;
        res->level = level;
        res->status = (err && *err) ? *err : NQS_OK;
        if (copy) *copy = *res;
    }
}

__global__ void __launch_bounds__(kThreads) level_sum_kernel(const double* __restrict__ vals,
                                                             const long long* __restrict__ level_off, int level,
                                                             nqs_result* __restrict__ res, double bound,
                                                             long long n_terms, const int* __restrict__ err) {
    level_sum_body(vals, level_off, level, res, bound, n_terms, err, nullptr);
}

// per-level sums of many circuits, one block each; results also gathered into one array
__global__ void __launch_bounds__(kThreads) level_sum_kernel_batched(const SumUnit* __restrict__ units) {
    const SumUnit u = units[blockIdx.x];
    level_sum_body(u.vals, u.level_off, u.level, u.res, u.bound, u.n_terms, u.err, u.copy);
}

// basis-state fills of many circuits: blockIdx.y selects the unit
__global__ void basis_fill_kernel_batched(const FillUnit* __restrict__ units) {
    const FillUnit u = units[blockIdx.y];
    long long stride = (long long)gridDim.x * blockDim.x;
    float4* o4 = reinterpret_cast<float4*>(u.dst);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (u.dim >> 1); i += stride) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if ((unsigned long long)(2 * i) == u.bits) v.x = 1.f;
        if ((unsigned long long)(2 * i + 1) == u.bits) v.z = 1.f;
        o4[i] = v;
    }
}

__global__ void basis_fill_kernel(float2* out, long long dim, unsigned long long bits) {
    long long stride = (long long)gridDim.x * blockDim.x;
    float4* o4 = reinterpret_cast<float4*>(out);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (dim >> 1); i += stride) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if ((unsigned long long)(2 * i) == bits) v.x = 1.f;
        if ((unsigned long long)(2 * i + 1) == bits) v.z = 1.f;
        o4[i] = v;
    }
}


cudaError_t launch_reduce2x2(const float2* phi, const float2* chi, int n, int q, double* partials, int grid,
                             cudaStream_t st) {
    reduce2x2_kernel<<<grid, kThreads, 0, st>>>(phi, chi, n, q, partials);
    return cudaGetLastError();
}

int finish_blocks(int n_slots) { return (n_slots + kWarps - 1) / kWarps; }

cudaError_t launch_finish(const double* partials, const FinishSlot* slots, const double* kmats, double* vals,
                          int n_slots, cudaStream_t st) {
    finish_kernel<<<finish_blocks(n_slots), kThreads, 0, st>>>(partials, slots, kmats, vals, n_slots);
    return cudaGetLastError();
}

// v <- v / ||v||, the norm from the per-block partials of reduce2x2_kernel(v,
// v, qubit 0): ||v||^2 = Re R00 + Re R11, summed in a fixed order by every
// block.  The noiseless circuit keeps the norm of a basis state, 1; complex64
// gates lose a little of it, and v enters F twice.  Bound by HBM (16 B per
// amplitude); every block's first warp adds the partials in parallel (one
// thread adding 608 of them took longer than the copy: 155 us at 24 qubits,
// 45 us so).
__global__ void __launch_bounds__(kThreads) normalize_kernel(float4* __restrict__ v, long long dim2,
                                                             const double* __restrict__ part, int grid) {
    __shared__ float scale;
    if (threadIdx.x < 32) {
        double a = 0.0;
        for (int g = threadIdx.x; g < grid; g += 32) a += part[(size_t)g * 8] + part[(size_t)g * 8 + 6];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (threadIdx.x == 0) scale = a > 0.0 ? (float)(1.0 / sqrt(a)) : 1.0f;
    }
    __syncthreads();
    const float f = scale;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < dim2; i += stride) {
        const float4 x = v[i];
        v[i] = make_float4(x.x * f, x.y * f, x.z * f, x.w * f);
    }
}

cudaError_t launch_normalize(float2* v, long long dim, const double* partials, int red_grid, int grid,
                             cudaStream_t st) {
    normalize_kernel<<<grid, kThreads, 0, st>>>(reinterpret_cast<float4*>(v), dim >> 1, partials, red_grid);
    return cudaGetLastError();
}

// out = x + c y for basis or dense x, y (the superposed states of the
// polarization identity); a basis state is |bits> (kind 0), dense ones are
// read from device memory (kind 1)
__global__ void __launch_bounds__(kThreads) combine_kernel(float2* __restrict__ out, long long dim, int xk,
                                                           unsigned long long xb, const float2* __restrict__ xd,
                                                           int yk, unsigned long long yb,
                                                           const float2* __restrict__ yd, float cre, float cim) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < dim; i += stride) {
        const float2 a = xk ? xd[i] : make_float2((unsigned long long)i == xb ? 1.f : 0.f, 0.f);
        const float2 b = yk ? yd[i] : make_float2((unsigned long long)i == yb ? 1.f : 0.f, 0.f);
        out[i] = make_float2(a.x + cre * b.x - cim * b.y, a.y + cre * b.y + cim * b.x);
    }
}

cudaError_t launch_combine(float2* out, long long dim, int xk, unsigned long long xb, const float2* xd, int yk,
                           unsigned long long yb, const float2* yd, float cre, float cim, int grid, cudaStream_t st) {
    combine_kernel<<<grid, kThreads, 0, st>>>(out, dim, xk, xb, xd, yk, yb, yd, cre, cim);
    return cudaGetLastError();
}

cudaError_t launch_partials_sum(const double* part, int grid, double* R, cudaStream_t st) {
    partials_sum_kernel<<<1, kThreads, 0, st>>>(part, grid, R);
    return cudaGetLastError();
}

cudaError_t launch_level_sum(const double* vals, const long long* level_off, int level, nqs_result* res,
                             double bound, long long n_terms, const int* err, cudaStream_t st) {
    level_sum_kernel<<<1, kThreads, 0, st>>>(vals, level_off, level, res, bound, n_terms, err);
    return cudaGetLastError();
}

cudaError_t launch_basis_fill(float2* out, long long dim, unsigned long long bits, int grid, cudaStream_t st) {
    basis_fill_kernel<<<grid, kThreads, 0, st>>>(out, dim, bits);
    return cudaGetLastError();
}

cudaError_t launch_finish_batched(const FinishUnit* units, const int* blk_begin, int n_units, int total_blocks,
                                  cudaStream_t st) {
    finish_kernel_batched<<<total_blocks, kThreads, 0, st>>>(units, blk_begin, n_units);
    return cudaGetLastError();
}

cudaError_t launch_level_sum_batched(const SumUnit* units, int n_units, cudaStream_t st) {
    level_sum_kernel_batched<<<n_units, kThreads, 0, st>>>(units);
    return cudaGetLastError();
}

cudaError_t launch_fill_batched(const FillUnit* units, int n_units, cudaStream_t st) {
    basis_fill_kernel_batched<<<dim3(64, n_units), kThreads, 0, st>>>(units);
    return cudaGetLastError();
}

}  // namespace nqs
