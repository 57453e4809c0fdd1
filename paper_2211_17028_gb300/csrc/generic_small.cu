// General-noise expansions of circuits of at most 14 qubits, in four launches.
//
// A state fits in the shared memory of one block, so a whole sweep is one
// block's loop over the gates.  (1) Two blocks make the checkpoints: phi_s from
// v backwards, chi_s from psi forwards.  (2) One block per prefix of insertions
// starts from chi of its first site, repeats the way to its last one and
// stores its state at every later site.  (3) All reductions at once: the
// reduced matrix of phi_t and each stored state in FP64, several blocks per
// reduction.  (4) Amplitudes of every factor from the reduced matrices.
//
// The sweeps are bound by the latency of one gate after another (shared
// memory, a few multiply-adds, a barrier), the reductions by the chip's few
// FP64 units: 64 FP64 multiply-adds per four amplitudes and pair of states,
// which is why they are spread over all SMs instead of staying in the sweeping
// blocks.  A 12-qubit level-2 call with four two-qubit noises (1411 terms)
// was 1950 launches and 94 host synchronisations, one gate or reduction each.
#include "generic_small.h"

#include <algorithm>

#include "generic_gates.cuh"

namespace nqs {

namespace {

constexpr int kChunk = 32;
constexpr int kMat = 16;
constexpr int kRedThreads = 256;

struct GShared {
    GOp ops[2][kChunk];
    float2 mats[2][kChunk * kMat];
};

__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}

// chunk c of an operation list into buffer c & 1 (the lists are padded to whole chunks)
__device__ __forceinline__ void fetch_chunk(GShared& sh, const GOp* ops, const float2* mats, int c) {
    for (int i = threadIdx.x; i < kChunk; i += blockDim.x) cp16(&sh.ops[c & 1][i], ops + (size_t)c * kChunk + i);
    for (int i = threadIdx.x; i < kChunk * kMat / 2; i += blockDim.x)
        cp16(&sh.mats[c & 1][2 * i], mats + (size_t)c * kChunk * kMat + 2 * i);
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ int pair_index(int p, int q) { return ((p >> q) << (q + 1)) | (p & ((1 << q) - 1)); }

__device__ __forceinline__ void apply_dense(float2* x, int n, int nq, int q0, int q1, const float2* m) {
    if (nq == 1) {
        const float2 m0 = m[0], m1 = m[1], m2 = m[2], m3 = m[3];
        for (int p = threadIdx.x; p < (1 << (n - 1)); p += blockDim.x) {
            const int i0 = pair_index(p, q0), i1 = i0 | (1 << q0);
            float2 a = x[i0], b = x[i1];
            gate2(m0, m1, m2, m3, a, b);
            x[i0] = a;
            x[i1] = b;
        }
    } else {
        for (int p = threadIdx.x; p < (1 << (n - 2)); p += blockDim.x) {
            long long idx[4];
            quad_index(p, q0, q1, idx);
            float2 v[4] = {x[idx[0]], x[idx[1]], x[idx[2]], x[idx[3]]};
            gate4(m, v);
#pragma unroll
            for (int k = 0; k < 4; ++k) x[idx[k]] = v[k];
        }
    }
}

// CZ and CX touch a quarter or half of the amplitudes: as dense 4x4 gates
// their products with 0 and 1 are exact, so signs and exchanges are the same
__device__ __forceinline__ void apply_gate(float2* x, int n, const GOp& op, const float2* m) {
    if (op.type == GO_ONE) {
        apply_dense(x, n, 1, op.a, 0, m);
        return;
    }
    for (int p = threadIdx.x; p < (1 << (n - 2)); p += blockDim.x) {
        long long idx[4];
        quad_index(p, op.a, op.b, idx);
        if (op.type == GO_CZ) {
            const float2 v = x[idx[3]];
            x[idx[3]] = make_float2(-v.x, -v.y);
        } else {
            const float2 v = x[idx[2]];
            x[idx[2]] = x[idx[3]];
            x[idx[3]] = v;
        }
    }
}

// operations [begin, end) of a list; at_site(op, matrix of K_0) for sites
template <typename SiteFn>
__device__ void run_ops(GShared& sh, float2* x, int n, const GOp* ops, const float2* mats, int begin, int end,
                        SiteFn at_site) {
    if (begin >= end) return;
    const int c0 = begin / kChunk, c1 = (end - 1) / kChunk;
    __syncthreads();
    fetch_chunk(sh, ops, mats, c0);
    if (c1 > c0) fetch_chunk(sh, ops, mats, c0 + 1);
    for (int c = c0; c <= c1; ++c) {
        if (c < c1) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const int oe = min(end - c * kChunk, kChunk);
        for (int o = max(begin - c * kChunk, 0); o < oe; ++o) {
            const GOp op = sh.ops[c & 1][o];
            const float2* const m = sh.mats[c & 1] + o * kMat;
            if (op.type == GO_SITE) at_site(op, m);
            else apply_gate(x, n, op, m);
            __syncthreads();
        }
        if (c + 2 <= c1) fetch_chunk(sh, ops, mats, c + 2);   // every thread is past this chunk
    }
}

__device__ __forceinline__ void load_state(float2* x, int n, int kind, unsigned long long bits, const float2* dev) {
    for (int j = threadIdx.x; j < (1 << n); j += blockDim.x)
        x[j] = kind == NQS_STATE_DENSE ? dev[j] : make_float2((unsigned long long)j == bits ? 1.f : 0.f, 0.f);
    __syncthreads();
}

__device__ __forceinline__ void copy_state(float2* dst, const float2* src, int n) {
    for (int j = threadIdx.x; j < (1 << n); j += blockDim.x) dst[j] = src[j];
}

__global__ void __launch_bounds__(1024) gs_checkpoints_kernel(const GSmallArgs A) {
    extern __shared__ __align__(16) float2 x[];
    __shared__ __align__(16) GShared sh;
    const int n = A.n;
    if (blockIdx.x == 1) {
        load_state(x, n, A.psi_kind, A.psi_bits, A.psi_dev);
        run_ops(sh, x, n, A.fwd, A.fwd_mats, 0, A.fwd_ops, [&](const GOp& op, const float2* m) {
            copy_state(A.chi + ((size_t)op.site << n), x, n);
            __syncthreads();
            apply_dense(x, n, op.nq, op.a, op.b, m);
        });
        return;
    }
    if (A.v_kind == NQS_STATE_IDEAL) {
        load_state(x, n, A.psi_kind, A.psi_bits, A.psi_dev);
        run_ops(sh, x, n, A.fwd, A.fwd_mats, 0, A.all_ops, [](const GOp&, const float2*) {});
    } else {
        load_state(x, n, A.v_kind, A.v_bits, A.v_dev);
    }
    run_ops(sh, x, n, A.bwd, A.bwd_mats, 0, A.bwd_ops, [&](const GOp& op, const float2* m) {
        copy_state(A.phi + ((size_t)op.site << n), x, n);
        __syncthreads();
        apply_dense(x, n, op.nq, op.a, op.b, m);
    });
}

__global__ void __launch_bounds__(1024) gs_units_kernel(const GSmallArgs A) {
    extern __shared__ __align__(16) float2 x[];
    __shared__ __align__(16) GShared sh;
    const int n = A.n;
    const GUnit* const u = A.units + blockIdx.x;
    const int depth = u->depth, first = u->site[0];
    copy_state(x, A.chi + ((size_t)first << n), n);
    __syncthreads();
    const GOp op0 = A.fwd[A.site_op[first]];
    apply_dense(x, n, op0.nq, op0.a, op0.b, A.factors + (size_t)(first * 16 + u->factor[0]) * kMat);
    int k = 1, slot = u->out;
    run_ops(sh, x, n, A.fwd, A.fwd_mats, A.site_op[first] + 1, A.fwd_ops, [&](const GOp& op, const float2* m) {
        if (k < depth && op.site == u->site[k]) {
            apply_dense(x, n, op.nq, op.a, op.b, A.factors + (size_t)(op.site * 16 + u->factor[k]) * kMat);
            ++k;
            return;
        }
        if (k == depth) {
            copy_state(A.out + ((size_t)slot << n), x, n);
            ++slot;
            __syncthreads();
        }
        apply_dense(x, n, op.nq, op.a, op.b, m);
    });
}

// per-block FP64 partials of R[a][b] of a pair: blockIdx.x pair, blockIdx.y part
__global__ void __launch_bounds__(kRedThreads) gs_reduce_kernel(const GSmallArgs A) {
    const GPair pr = A.pairs[blockIdx.x];
    const GOp op = A.fwd[A.site_op[pr.site]];
    const float2* const phi = A.phi + ((size_t)pr.site << A.n);
    const float2* const w = pr.slot < 0 ? A.chi + ((size_t)pr.site << A.n) : A.out + ((size_t)pr.slot << A.n);
    double acc[32];
#pragma unroll
    for (int e = 0; e < 32; ++e) acc[e] = 0.0;
    const int count = 1 << (A.n - op.nq), stride = gridDim.y * kRedThreads;
    for (int p = blockIdx.y * kRedThreads + threadIdx.x; p < count; p += stride) {
        if (op.nq == 1) {
            const int i0 = pair_index(p, op.a), i1 = i0 | (1 << op.a);
            const float2 f[2] = {phi[i0], phi[i1]}, x[2] = {w[i0], w[i1]};
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    acc[2 * (2 * a + b)] += (double)f[a].x * x[b].x + (double)f[a].y * x[b].y;
                    acc[2 * (2 * a + b) + 1] += (double)f[a].x * x[b].y - (double)f[a].y * x[b].x;
                }
        } else {
            long long idx[4];
            quad_index(p, op.a, op.b, idx);
            float2 f[4], x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                f[k] = phi[idx[k]];
                x[k] = w[idx[k]];
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    acc[2 * (4 * a + b)] += (double)f[a].x * x[b].x + (double)f[a].y * x[b].y;
                    acc[2 * (4 * a + b) + 1] += (double)f[a].x * x[b].y - (double)f[a].y * x[b].x;
                }
        }
    }
    __shared__ double sm[kRedThreads / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    sm[warp][lane] = warp_scatter32(acc, lane);
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < kRedThreads / 32; ++k) v += sm[k][threadIdx.x];
        A.part[((size_t)blockIdx.x * gridDim.y + blockIdx.y) * 32 + threadIdx.x] = v;
    }
}

// one warp per pair: R from its parts, then sum_ab K_j[a][b] R[a][b]
__global__ void __launch_bounds__(32) gs_finish_kernel(const GSmallArgs A) {
    __shared__ double R[32];
    const GPair pr = A.pairs[blockIdx.x];
    double v = 0.0;
    for (int k = 0; k < A.parts; ++k) v += A.part[((size_t)blockIdx.x * A.parts + k) * 32 + threadIdx.x];
    R[threadIdx.x] = v;
    __syncwarp();
    const int m = A.n_factors[pr.site], j = threadIdx.x;
    if (j >= m) return;
    const long long rank = j == 0 ? pr.rank0 : pr.rank >= 0 ? pr.rank + j - 1 : -1;
    if (rank < 0) return;
    const int dd = A.fwd[A.site_op[pr.site]].nq == 1 ? 4 : 16;
    const double2* const k = A.kmats + A.kofs[pr.site] + (size_t)j * dd;
    double re = 0.0, im = 0.0;
    for (int e = 0; e < dd; ++e) {
        re += k[e].x * R[2 * e] - k[e].y * R[2 * e + 1];
        im += k[e].x * R[2 * e + 1] + k[e].y * R[2 * e];
    }
    A.amps[rank] = make_double2(re, im);
}

}  // namespace

int generic_small_parts(int n, int n_pairs, int sms) {
    const int most = std::max(1, (1 << std::max(0, n - 2)) / kRedThreads);
    return std::max(1, std::min(most, (4 * sms + n_pairs - 1) / std::max(1, n_pairs)));
}

cudaError_t launch_generic_small(const GSmallArgs& a, cudaStream_t st) {
    const int threads = std::min(1024, std::max(32, 1 << std::max(0, a.n - 2)));
    const size_t smem = sizeof(float2) << a.n;
    cudaError_t e = cudaSuccess;
    if (smem > (size_t)(32 << 10)) {
        e = allow_dynamic_smem((const void*)gs_checkpoints_kernel);
        if (e == cudaSuccess) e = allow_dynamic_smem((const void*)gs_units_kernel);
        if (e != cudaSuccess) return e;
    }
    gs_checkpoints_kernel<<<2, threads, smem, st>>>(a);
    if (a.n_units > 0) gs_units_kernel<<<a.n_units, threads, smem, st>>>(a);
    gs_reduce_kernel<<<dim3(a.n_pairs, a.parts), kRedThreads, 0, st>>>(a);
    gs_finish_kernel<<<a.n_pairs, 32, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace nqs
