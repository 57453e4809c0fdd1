// Expansions of circuits of at most 11 qubits, in two launches.
//
// A whole state (at most 16 KiB) lives in the shared memory of one block, so
// a sweep needs no passes, and every kept prefix of the expansion is a block of
// its own: the first launch sweeps the test state backwards and the input
// state forwards (two blocks), storing phi_s and chi_s at every site; the
// second has one block per site (levels 0 and 1 from phi_s and chi_s alone)
// and one per prefix of insertions, which starts from chi of its first site
// and repeats the way to its last one instead of waiting for another block.
// Term values come straight out of the block that reduced them.
//
// What bounds it is the latency of one operation after another: matrix and
// record from shared memory, two amplitudes, eight multiply-adds, a barrier.
// Operations come in chunks of 32 by cp.async two ahead of use, and the next
// record and matrix are read before the barrier.  The 6-qubit level-4 call
// (256 terms, 175 prefixes) took 54 three-state launches of 27 us one after
// another, chains of dependent global reads: 1.94 ms, and 59 us so.
#include "small.h"

#include <algorithm>

#include "sweep_types.h"

namespace nqs {

namespace {

constexpr int kChunk = 32;        // operations per chunk
constexpr int kMat = 16;          // float2 per operation
constexpr int kAccSites = 32;     // reductions collected before they become terms

struct SmallShared {
    SmallOp ops[2][kChunk];
    float2 mats[2][kChunk * kMat];
    double acc[kAccSites][8][8];  // [reduction][warp][component]
    double R[kAccSites][8];
    double norm[8];
};

__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}

// chunk c of an operation list into buffer c & 1 (whole chunks: the lists are padded)
__device__ __forceinline__ void fetch_chunk(SmallShared& sh, const SmallOp* ops, const float2* mats, int c) {
    SmallOp* const od = sh.ops[c & 1];
    float2* const md = sh.mats[c & 1];
    for (int i = threadIdx.x; i < kChunk; i += blockDim.x) cp16(od + i, ops + (size_t)c * kChunk + i);
    for (int i = threadIdx.x; i < kChunk * kMat / 2; i += blockDim.x)
        cp16(md + 2 * i, mats + (size_t)c * kChunk * kMat + 2 * i);
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// sums of v[0..7] over the warp; lane l with l % 4 == 0 ends with component
// ((l >> 4) & 1) * 4 + ((l >> 3) & 1) * 2 + ((l >> 2) & 1) in v[0]
__device__ __forceinline__ void warp_scatter(float (&v)[8], int lane) {
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1) {
        const bool hi = lane & (4 * w);
#pragma unroll
        for (int e = 0; e < w; ++e) {
            const float send = hi ? v[e] : v[e + w];
            const float keep = hi ? v[e + w] : v[e];
            v[e] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * w);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// R[a][b] += conj(phi_a) chi_b over the pairs of qubit q, into acc[warp]
__device__ __forceinline__ void reduce_site(const float2* __restrict__ phi, const float2* x, int n, int q,
                                            double (*acc)[8]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float r[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int p = threadIdx.x; p < (1 << (n - 1)); p += blockDim.x) {
        const int j0 = insert0(p, q), j1 = j0 | (1 << q);
        const float2 f0 = phi[j0], f1 = phi[j1], x0 = x[j0], x1 = x[j1];
        r[0] += f0.x * x0.x + f0.y * x0.y;  r[1] += f0.x * x0.y - f0.y * x0.x;
        r[2] += f0.x * x1.x + f0.y * x1.y;  r[3] += f0.x * x1.y - f0.y * x1.x;
        r[4] += f1.x * x0.x + f1.y * x0.y;  r[5] += f1.x * x0.y - f1.y * x0.x;
        r[6] += f1.x * x1.x + f1.y * x1.y;  r[7] += f1.x * x1.y - f1.y * x1.x;
    }
    warp_scatter(r, lane);
    if ((lane & 3) == 0)
        acc[warp][((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = (double)r[0];
}

// |sum_ab K[a][b] R[a][b]|^2
__device__ __forceinline__ double term_value(const double* __restrict__ K, const double* R) {
    double re = 0, im = 0;
    for (int e = 0; e < 4; ++e) {
        re += K[2 * e] * R[2 * e] - K[2 * e + 1] * R[2 * e + 1];
        im += K[2 * e] * R[2 * e + 1] + K[2 * e + 1] * R[2 * e];
    }
    return re * re + im * im;
}

// one operation on the state x
__device__ __forceinline__ void apply_op(float2* x, int n, const SmallOp& op, const float2* m, const float2 (&m4)[4]) {
    const int T = 1 << n;
    if (op.type == OP_G1) {
        for (int p = threadIdx.x; p < (T >> 1); p += blockDim.x) {
            const int j0 = insert0(p, op.a), j1 = j0 | (1 << op.a);
            const float2 x0 = x[j0], x1 = x[j1];
            x[j0] = cfma(m4[0], x0, cmul(m4[1], x1));
            x[j1] = cfma(m4[2], x0, cmul(m4[3], x1));
        }
    } else if (op.type == OP_D1) {
        for (int j = threadIdx.x; j < T; j += blockDim.x) x[j] = cmul(((j >> op.a) & 1) ? m4[3] : m4[0], x[j]);
    } else if (op.type == OP_D2) {
        for (int j = threadIdx.x; j < T; j += blockDim.x)
            x[j] = cmul(m[5 * (2 * ((j >> op.a) & 1) + ((j >> op.b) & 1))], x[j]);
    } else if (op.type == OP_G2) {
        const int lo = min(op.a, op.b), hi = max(op.a, op.b), ba = 1 << op.a, bb = 1 << op.b;
        for (int p = threadIdx.x; p < (T >> 2); p += blockDim.x) {
            const int j = insert0(insert0(p, lo), hi);
            const int idx[4] = {j, j | bb, j | ba, j | ba | bb};
            float2 v[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r] = x[idx[r]];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float2 y = cmul(m[4 * r], v[0]);
                y = cfma(m[4 * r + 1], v[1], y);
                y = cfma(m[4 * r + 2], v[2], y);
                x[idx[r]] = cfma(m[4 * r + 3], v[3], y);
            }
        }
    }
}

// K of a site: K_0 (products only, when diagonal) or a kept factor
__device__ __forceinline__ void apply_factor(float2* x, int n, const SmallOp& op, const float2* K, bool diag) {
    const float2 k0 = K[0], k1 = K[1], k2 = K[2], k3 = K[3];
    for (int p = threadIdx.x; p < (1 << (n - 1)); p += blockDim.x) {
        const int j0 = insert0(p, op.a), j1 = j0 | (1 << op.a);
        const float2 x0 = x[j0], x1 = x[j1];
        x[j0] = diag ? cmul(k0, x0) : cfma(k0, x0, cmul(k1, x1));
        x[j1] = diag ? cmul(k3, x1) : cfma(k2, x0, cmul(k3, x1));
    }
}

// Operations [begin, end) of a list, calling at_site(op, matrices) for sites
// (the state is complete there; it returns whether it ends with a barrier due).
template <typename SiteFn>
__device__ void run_ops(SmallShared& sh, float2* x, int n, const SmallOp* ops, const float2* mats, int begin, int end,
                        SiteFn at_site) {
    if (begin >= end) return;
    const int c0 = begin / kChunk, c1 = (end - 1) / kChunk;
    __syncthreads();   // the buffers are free
    fetch_chunk(sh, ops, mats, c0);
    if (c1 > c0) fetch_chunk(sh, ops, mats, c0 + 1);
    for (int c = c0; c <= c1; ++c) {
        if (c < c1) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const SmallOp* const os = sh.ops[c & 1];
        const float2* const ms = sh.mats[c & 1];
        int o = max(begin - c * kChunk, 0);
        const int oe = min(end - c * kChunk, kChunk);
        SmallOp next = os[o];
        float2 nm[4] = {ms[o * kMat], ms[o * kMat + 1], ms[o * kMat + 2], ms[o * kMat + 3]};
        for (; o < oe; ++o) {
            const SmallOp op = next;
            const float2 m4[4] = {nm[0], nm[1], nm[2], nm[3]};
            const float2* const m = ms + o * kMat;
            const int w = min(o + 1, oe - 1);
            next = os[w];
#pragma unroll
            for (int e = 0; e < 4; ++e) nm[e] = ms[w * kMat + e];
            if (op.type == OP_SITE) at_site(op, m);
            else apply_op(x, n, op, m, m4);
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

__device__ __forceinline__ void store_state(float2* dst, const float2* x, int n) {
    for (int j = threadIdx.x; j < (1 << n); j += blockDim.x) dst[j] = x[j];
}

// block 0: phi_s from v backwards (v = U |psi> first when asked for); block 1:
// chi_s from psi forwards
__global__ void __launch_bounds__(256) small_checkpoints_kernel(const SmallArgs A) {
    extern __shared__ __align__(16) float2 x[];
    __shared__ __align__(16) SmallShared sh;
    const int n = A.n;
    if (blockIdx.x == 1) {
        load_state(x, n, A.psi_kind, A.psi_bits, A.psi_dev);
        run_ops(sh, x, n, A.fwd, A.fwd_mats, 0, A.fwd_ops, [&](const SmallOp& op, const float2* m) {
            store_state(A.chi + ((size_t)op.site << n), x, n);
            __syncthreads();
            apply_factor(x, n, op, m, op.diag);
        });
        return;
    }
    if (A.v_kind == NQS_STATE_IDEAL) {
        load_state(x, n, A.psi_kind, A.psi_bits, A.psi_dev);
        run_ops(sh, x, n, A.fwd, A.fwd_mats, 0, A.all_ops, [](const SmallOp&, const float2*) {});
        if (A.psi_kind == NQS_STATE_BASIS) {
            // the computed state has the norm of the basis state, 1
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            double s = 0.0;
            for (int j = threadIdx.x; j < (1 << n); j += blockDim.x)
                s += (double)x[j].x * x[j].x + (double)x[j].y * x[j].y;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) sh.norm[warp] = s;
            __syncthreads();
            double t = 0.0;
            for (int w = 0; w < (int)blockDim.x / 32; ++w) t += sh.norm[w];
            const float f = t > 0.0 ? (float)(1.0 / sqrt(t)) : 1.0f;
            for (int j = threadIdx.x; j < (1 << n); j += blockDim.x) x[j] = make_float2(x[j].x * f, x[j].y * f);
            __syncthreads();
        }
    } else {
        load_state(x, n, A.v_kind, A.v_bits, A.v_dev);
    }
    run_ops(sh, x, n, A.bwd, A.bwd_mats, 0, A.bwd_ops, [&](const SmallOp& op, const float2* m) {
        store_state(A.phi + ((size_t)op.site << n), x, n);
        __syncthreads();
        apply_factor(x, n, op, m, op.diag);
    });
}

// terms of `count` collected reductions: site[k] and the rank of the first
// factor's term
template <typename SiteRankFn>
__device__ void write_terms(const SmallArgs& A, SmallShared& sh, int count, SiteRankFn at) {
    __syncthreads();
    for (int i = threadIdx.x; i < count * 8; i += blockDim.x) {
        double v = 0.0;
        for (int w = 0; w < (int)blockDim.x / 32; ++w) v += sh.acc[i >> 3][w][i & 7];
        sh.R[i >> 3][i & 7] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < count * 3; i += blockDim.x) {
        const int k = i / 3, f = i % 3;
        int site;
        long long rank;
        at(k, site, rank);
        if (rank >= 0 && f < A.n_factors[site])
            A.term_vals[rank + f] = term_value(A.kmats + site * 32 + A.keep[3 * site + f] * 8, sh.R[k]);
    }
    __syncthreads();
}

// blocks 0 .. n_sites - 1: levels 0 and 1 of one site; the others: one unit each
__global__ void __launch_bounds__(256) small_units_kernel(const SmallArgs A) {
    extern __shared__ __align__(16) float2 x[];
    __shared__ __align__(16) SmallShared sh;
    const int n = A.n;
    if ((int)blockIdx.x < A.n_sites) {
        const int s = blockIdx.x;
        if (A.pair_rank[s] < 0 && !(s == 0 && A.level0 >= 0)) return;
        const int q = A.fwd[A.site_op[s]].a;
        reduce_site(A.phi + ((size_t)s << n), A.chi + ((size_t)s << n), n, q, sh.acc[0]);
        write_terms(A, sh, 1, [&](int, int& site, long long& rank) {
            site = s;
            rank = A.pair_rank[s];
        });
        if (s == 0 && A.level0 >= 0 && threadIdx.x == 0)
            A.term_vals[A.level0] = term_value(A.kmats, sh.R[0]);
        return;
    }
    const SmallUnit* const u = A.units + (blockIdx.x - A.n_sites);
    const int depth = u->depth, first = u->site[0], last = u->site[depth - 1];
    store_state(x, A.chi + ((size_t)first << n), n);
    __syncthreads();
    // the first insertion
    {
        const int o = A.site_op[first];
        const SmallOp op = A.fwd[o];
        apply_factor(x, n, op, A.fwd_mats + (size_t)o * kMat + 4 * (u->factor[0] + 1), false);
    }
    int k = 1, count = 0, t0 = last + 1;
    const long long* const ranks = A.ranks + u->rank;
    run_ops(sh, x, n, A.fwd, A.fwd_mats, A.site_op[first] + 1, A.fwd_ops, [&](const SmallOp& op, const float2* m) {
        if (k < depth && op.site == u->site[k]) {
            apply_factor(x, n, op, m + 4 * (u->factor[k] + 1), false);
            ++k;
            return;
        }
        if (k == depth) {
            reduce_site(A.phi + ((size_t)op.site << n), x, n, op.a, sh.acc[count]);
            if (++count == kAccSites) {
                write_terms(A, sh, count, [&](int j, int& site, long long& rank) {
                    site = t0 + j;
                    rank = ranks[site - last - 1];
                });
                t0 += count;
                count = 0;
            } else {
                __syncthreads();
            }
        }
        apply_factor(x, n, op, m, op.diag);
    });
    if (count > 0)
        write_terms(A, sh, count, [&](int j, int& site, long long& rank) {
            site = t0 + j;
            rank = ranks[site - last - 1];
        });
}

}  // namespace

cudaError_t launch_small(const SmallArgs& a, cudaStream_t st) {
    const int threads = a.n <= 6 ? 32 : std::min(256, 1 << (a.n - 1));
    const size_t smem = sizeof(float2) << a.n;
    small_checkpoints_kernel<<<2, threads, smem, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    small_units_kernel<<<a.n_sites + a.n_units, threads, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace nqs
