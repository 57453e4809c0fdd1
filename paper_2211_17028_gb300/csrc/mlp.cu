// Proposal network of the importance-sampled level-l estimate: a small MLP
// (ReLU hidden layers, linear scalar output) whose weights are used in bf16
// with fp32 accumulation, trained on the GPU by the kernels below (forward,
// backward, Adam on fp32 master weights, mean-squared-error loss).  The
// matrix products run on the bf16 tensor cores (warp-level mma.sync).
//
// Parameters, flattened in this order: for each layer l, W_l (out x in,
// row-major) then b_l (out).  The bf16 copy of every W_l is what the forward
// and backward passes read; gradients flow to the fp32 masters.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <vector>

#include "nqs_internal.h"

namespace nqs {

namespace {

// Matrix products on the bf16 tensor cores (mma.sync m16n8k16, fp32
// accumulation).  Both MMA operands are bf16, so an fp32 operand x enters as
// two bf16 parts, x_hi = bf16(x) and x_lo = bf16(x - x_hi) (x = x_hi + x_lo to
// about 2^-16 of |x|): A_hi B + A_lo B for bf16 weights, A_hi B_hi + A_lo B_hi +
// A_hi B_lo when both are fp32 (the lo * lo product is below fp32 resolution).
//
// The layers are 256 wide and a batch is about a thousand rows, so a product is
// a hundred blocks of a few microseconds: what bounds it is the latency of the
// k-steps and the number of launches, not the tensor cores.  Hence small tiles
// (64 x 32, k-step 64), the next step's operands in registers while the
// current one multiplies (float4 loads, split on the way into shared memory),
// fragments by ldmatrix, and everything elementwise in the epilogues: bias and
// ReLU forward, the ReLU mask backward, bias gradients in the blocks that read
// dY anyway; the input gradient and the weight gradient of a layer share one
// launch.  Loss and gradient through 8 -> 256 x 3 -> 1, with the gradient's copy
// to the host: 1024 rows 8 launches instead of 25, 435 -> 117 us (k-step 32:
// 128 us); 8192 rows 925 -> 238 us (249 us); 4096 rows through three layers of
// 1024 4.24 -> 1.13 ms.
constexpr int kBM = 64, kBN = 32, kBK = 64;
constexpr int kGemmThreads = 128;

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16* p) {
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(a));
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(a));
}

// A ROWS x COLS piece of a row-major matrix, four consecutive columns per
// thread and step; VEC: rows and pointers aligned for vector loads.
template <typename T, int ROWS, int COLS, bool VEC>
struct Tile {
    static constexpr int N = ROWS * COLS / 4 / kGemmThreads;
    float v[N][4];
    __device__ __forceinline__ void load(const T* __restrict__ src, int ld, int r0, int c0, int r_end, int c_end) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int e = threadIdx.x + i * kGemmThreads;
            const int r = r0 + e / (COLS / 4), c = c0 + 4 * (e % (COLS / 4));
            const T* const p = src + (size_t)r * ld + c;
            if (VEC && r < r_end && c + 3 < c_end) {
                if constexpr (std::is_same<T, float>::value) {
                    const float4 q = *reinterpret_cast<const float4*>(p);
                    v[i][0] = q.x;
                    v[i][1] = q.y;
                    v[i][2] = q.z;
                    v[i][3] = q.w;
                } else {
                    const uint2 q = *reinterpret_cast<const uint2*>(p);
                    const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x));
                    const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y));
                    v[i][0] = x.x;
                    v[i][1] = x.y;
                    v[i][2] = y.x;
                    v[i][3] = y.y;
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) v[i][k] = (r < r_end && c + k < c_end) ? (float)p[k] : 0.f;
            }
        }
    }
    // into shared memory (row pitch LD), high and low bf16 parts (LO: both)
    template <bool LO, int LD>
    __device__ __forceinline__ void store(__nv_bfloat16* hi, __nv_bfloat16* lo) const {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int e = threadIdx.x + i * kGemmThreads;
            const int at = (e / (COLS / 4)) * LD + 4 * (e % (COLS / 4));
            __nv_bfloat162 h[2], l[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                h[k] = __floats2bfloat162_rn(v[i][2 * k], v[i][2 * k + 1]);
                const float2 f = __bfloat1622float2(h[k]);
                if (LO) l[k] = __floats2bfloat162_rn(v[i][2 * k] - f.x, v[i][2 * k + 1] - f.y);
            }
            *reinterpret_cast<uint2*>(hi + at) = *reinterpret_cast<const uint2*>(h);
            if (LO) *reinterpret_cast<uint2*>(lo + at) = *reinterpret_cast<const uint2*>(l);
        }
    }
};

struct alignas(16) GemmShared {
    // rows padded by 8 (conflict-free ldmatrix): A [m][k] or [k][m], B [n][k] or [k][n]
    __nv_bfloat16 ah[kBM * (kBK + 8)], al[kBM * (kBK + 8)], bh[kBK * (kBN + 8)], bl[kBK * (kBN + 8)];
};

enum GemmMode { GM_FWD, GM_DX, GM_DW };

// One 64 x 32 output tile.
//   GM_FWD: C[M x N] = act(A[M x K] W[N x K]^T + bias), act = ReLU or none
//   GM_DX:  C[M x N] = A[M x K] W[K x N], zero where mask[M x N] <= 0
//   GM_DW:  part[M x N] = sum over k in [k0, k1) of A[k x M] X[k x N], and
//           bias_part[M] = the column sums of A (tiles of the first N columns)
template <int MODE, bool VEC>
__device__ __forceinline__ void gemm_tile(GemmShared& sh, int M, int N, int K, int k0, int k1, const float* __restrict__ A,
                                          const void* __restrict__ Bv, float* __restrict__ C,
                                          const float* __restrict__ extra, int relu, float* __restrict__ bias_part,
                                          int m0, int n0) {
    constexpr bool DW = MODE == GM_DW;
    constexpr int LDA = (DW ? kBM : kBK) + 8, LDB = (MODE == GM_FWD ? kBK : kBN) + 8;
    static_assert(kBM == kBK, "tiles of A have one size");
    typedef typename std::conditional<DW, float, __nv_bfloat16>::type TB;
    const TB* const B = (const TB*)Bv;
    Tile<float, DW ? kBK : kBM, DW ? kBM : kBK, VEC> ta;
    Tile<TB, MODE == GM_FWD ? kBN : kBK, MODE == GM_FWD ? kBK : kBN, VEC> tb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto load = [&](int k) {
        if (DW) ta.load(A, M, k, m0, k1, M);
        else ta.load(A, K, m0, k, M, k1);
        if (MODE == GM_FWD) tb.load(B, K, n0, k, N, k1);
        else tb.load(B, N, k, n0, k1, N);
    };
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
    // bias gradient: thread t sums column 4 (t % 16) .. + 3 of the rows it stages
    float bsum[4] = {0.f, 0.f, 0.f, 0.f};
    const int sub = lane >> 3, row = lane & 7;   // ldmatrix: matrix of the lane's address, its row
    if (k0 < k1) load(k0);
    for (int k = k0; k < k1; k += kBK) {
        __syncthreads();
        ta.template store<true, LDA>(sh.ah, sh.al);
        tb.template store<DW, LDB>(sh.bh, sh.bl);
        if (DW && bias_part && n0 == 0)
#pragma unroll
            for (int i = 0; i < ta.N; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) bsum[e] += ta.v[i][e];
        __syncthreads();
        if (k + kBK < k1) load(k + kBK);
#pragma unroll
        for (int kk = 0; kk < kBK; kk += 16) {
            uint32_t ah[4], al[4], bh[2][4], bl[2][4];
            // A matrices: (m 0-7, k 0-7), (m 8-15, k 0-7), (m 0-7, k 8-15), (m 8-15, k 8-15)
            const int am = 16 * warp + 8 * (sub & 1), ak = kk + 8 * (sub >> 1);
            const int at = DW ? (ak + row) * LDA + am : (am + row) * LDA + ak;
            ldsm4<DW>(ah, sh.ah + at);
            ldsm4<DW>(al, sh.al + at);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                // B matrices: (n 0-7, k 0-7), (n 0-7, k 8-15), (n 8-15, k 0-7), (n 8-15, k 8-15)
                const int bn = 16 * j + 8 * (sub >> 1), bk = kk + 8 * (sub & 1);
                const int bt = MODE == GM_FWD ? (bn + row) * LDB + bk : (bk + row) * LDB + bn;
                ldsm4<MODE != GM_FWD>(bh[j], sh.bh + bt);
                if (DW) ldsm4<true>(bl[j], sh.bl + bt);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                mma_bf16(acc[j], ah, bh[j >> 1] + 2 * (j & 1));
                mma_bf16(acc[j], al, bh[j >> 1] + 2 * (j & 1));
                if (DW) mma_bf16(acc[j], ah, bl[j >> 1] + 2 * (j & 1));
            }
        }
    }
    // accumulator element e of the 16 x 8 tile: row g (+8 for e >= 2), column 2t + (e & 1)
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int m = m0 + 16 * warp + g + (e >= 2 ? 8 : 0);
            const int n = n0 + 8 * j + 2 * t + (e & 1);
            if (m >= M || n >= N) continue;
            float v = acc[j][e];
            if (MODE == GM_FWD) {
                v += extra[n];
                if (relu) v = fmaxf(v, 0.f);
            }
            if (MODE == GM_DX && extra[(size_t)m * N + n] <= 0.f) v = 0.f;
            C[(size_t)m * N + n] = v;
        }
    if (DW && bias_part && n0 == 0) {
        // the eight rows of threads that share a column, in a fixed order
        __syncthreads();
        float* const s = reinterpret_cast<float*>(sh.ah);
        constexpr int CG = kBM / 4;   // threads along a row
#pragma unroll
        for (int e = 0; e < 4; ++e) s[(threadIdx.x / CG) * kBM + 4 * (threadIdx.x % CG) + e] = bsum[e];
        __syncthreads();
        if (threadIdx.x < kBM && m0 + (int)threadIdx.x < M) {
            float v = 0.f;
#pragma unroll
            for (int r = 0; r < kGemmThreads / CG; ++r) v += s[r * kBM + threadIdx.x];
            bias_part[m0 + threadIdx.x] = v;
        }
    }
}

template <bool VEC>
__global__ void __launch_bounds__(kGemmThreads) mlp_forward_kernel(int M, int N, int K, const float* __restrict__ A,
                                                                   const __nv_bfloat16* __restrict__ W,
                                                                   float* __restrict__ C, const float* __restrict__ bias,
                                                                   int relu) {
    __shared__ GemmShared sh;
    gemm_tile<GM_FWD, VEC>(sh, M, N, K, 0, K, A, W, C, bias, relu, nullptr, blockIdx.y * kBM, blockIdx.x * kBN);
}

// Backward of one layer (out x in weights, B rows): blocks [0, dx_tiles) the
// input gradient dX = (dY W) masked by the input's ReLU, the others the weight
// gradient's partial products over `chunk` rows each (z-major) with the bias sums.
struct LayerBack {
    int B, out, in, dx_tiles, splits, chunk;
    const float* dY;
    const float* X;               // the layer's input (activations, post-ReLU)
    const __nv_bfloat16* W;
    float* dX;
    float* part;                  // [split][out * in + out]
};

template <bool VEC>
__global__ void __launch_bounds__(kGemmThreads) mlp_backward_kernel(const LayerBack L) {
    __shared__ GemmShared sh;
    int b = blockIdx.x;
    if (b < L.dx_tiles) {
        const int nt = (L.in + kBN - 1) / kBN;
        gemm_tile<GM_DX, VEC>(sh, L.B, L.in, L.out, 0, L.out, L.dY, L.W, L.dX, L.X, 0, nullptr, (b / nt) * kBM,
                              (b % nt) * kBN);
        return;
    }
    b -= L.dx_tiles;
    const int nt = (L.in + kBN - 1) / kBN, tiles = ((L.out + kBM - 1) / kBM) * nt;
    const int z = b / tiles, tile = b % tiles;
    float* const part = L.part + (size_t)z * ((size_t)L.out * L.in + L.out);
    gemm_tile<GM_DW, VEC>(sh, L.out, L.in, L.B, z * L.chunk, min(L.B, (z + 1) * L.chunk), L.dY, L.X, part, nullptr, 0,
                          part + (size_t)L.out * L.in, (tile / nt) * kBM, (tile % nt) * kBN);
}

// The linear output of every row, a warp per row: pred = act . w + b.  With
// targets also the loss's partial sums, dY = 2 (pred - y) / B, the masked
// gradient of the activations and the block's share of the layer's gradient.
constexpr int kHeadRows = 16, kHeadThreads = 256, kHeadBlocks = 256;

__global__ void __launch_bounds__(kHeadThreads) mlp_head_kernel(int B, int K, int rows_per_block, const float* __restrict__ act,
                                                                const __nv_bfloat16* __restrict__ w,
                                                                const float* __restrict__ bias, float* __restrict__ pred,
                                                                const float* __restrict__ y, float* __restrict__ dact,
                                                                double* __restrict__ loss_part,
                                                                float* __restrict__ part, int mask) {
    __shared__ float d[kHeadRows];
    __shared__ double sq[kHeadRows];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int first = blockIdx.x * rows_per_block, end = min(B, first + rows_per_block);
    float* const grad = part + (size_t)blockIdx.x * (K + 1);
    double loss = 0.0;
    float bsum = 0.f;
    for (int r0 = first; r0 < end; r0 += kHeadRows) {
        const int rows = min(kHeadRows, end - r0);
        for (int i = warp; i < rows; i += kHeadThreads / 32) {
            const int r = r0 + i;
            float s = 0.f;
            for (int k = lane; k < K; k += 32) s = fmaf(act[(size_t)r * K + k], __bfloat162float(w[k]), s);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) {
                const float p = s + bias[0];
                pred[r] = p;
                const float e = y ? p - y[r] : 0.f;
                d[i] = 2.f * e / (float)B;
                sq[i] = (double)e * e;
            }
        }
        if (!y) continue;
        __syncthreads();
        if (threadIdx.x == 0)
            for (int i = 0; i < rows; ++i) {
                loss += sq[i];
                bsum += d[i];
            }
        // the same thread has the same columns in every group of rows
        for (int k = threadIdx.x; k < K; k += kHeadThreads) {
            const float wk = __bfloat162float(w[k]);
            float s = r0 == first ? 0.f : grad[k];
            for (int i = 0; i < rows; ++i) {
                const float a = act[(size_t)(r0 + i) * K + k];
                s = fmaf(d[i], a, s);
                dact[(size_t)(r0 + i) * K + k] = (mask && a <= 0.f) ? 0.f : d[i] * wk;
            }
            grad[k] = s;
        }
        __syncthreads();
    }
    if (y && threadIdx.x == 0) {
        loss_part[blockIdx.x] = loss;
        grad[K] = bsum;
    }
}

// Gradients from the partial sums of every layer, in a fixed order; block 0
// also adds the loss.
struct LayerSum {
    const float* part;
    int splits;
    int count;                    // parameters of the layer (weights, then biases)
    int first;                    // their offset
};
struct GradSums {
    LayerSum layer[9];
    int layers, loss_parts, B;
    const double* loss_part;
    double* loss;
};

__global__ void __launch_bounds__(256) mlp_gradient_kernel(GradSums S, float* __restrict__ g, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int l = 0;
        while (l + 1 < S.layers && i >= S.layer[l + 1].first) ++l;
        const LayerSum& L = S.layer[l];
        const float* const p = L.part + (i - L.first);
        if (L.splits == 0) continue;   // written there already
        float v = 0.f;
        int z = 0;
        for (; z + 8 <= L.splits; z += 8) {   // eight loads in flight
            float x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = p[(size_t)(z + k) * L.count];
#pragma unroll
            for (int k = 0; k < 8; ++k) v += x[k];
        }
        for (; z < L.splits; ++z) v += p[(size_t)z * L.count];
        g[i] = v;
    }
    if (blockIdx.x == 0) {
        __shared__ double s[256];
        double t = 0.0;
        for (int k = threadIdx.x; k < S.loss_parts; k += 256) t += S.loss_part[k];
        s[threadIdx.x] = t;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if ((int)threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) *S.loss = s[0] / S.B;
    }
}

__global__ void to_bf16_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) wb[i] = __float2bfloat16(w[i]);
}

// Adam on the fp32 masters; the bf16 copies follow
__global__ void adam_kernel(float* __restrict__ w, __nv_bfloat16* __restrict__ wb, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        wb[i] = __float2bfloat16(wi);
    }
}

// rows of (X, y) picked by a counter-based generator (SplitMix64 of seed + step*B + i)
__device__ __forceinline__ unsigned long long splitmix(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void gather_batch_kernel(const float* __restrict__ X, const float* __restrict__ y, int n, int in,
                                    float* __restrict__ Xb, float* __restrict__ yb, int B, unsigned long long seed,
                                    long long step) {
    const int i = blockIdx.x;
    if (i >= B) return;
    const unsigned long long r = splitmix(seed + (unsigned long long)step * B + i);
    const int src = (int)(r % (unsigned long long)n);
    for (int k = threadIdx.x; k < in; k += blockDim.x) Xb[(size_t)i * in + k] = X[(size_t)src * in + k];
    if (threadIdx.x == 0) yb[i] = y[src];
}

}  // namespace

struct Mlp {
    std::vector<int> dims;        // in, hidden..., 1
    size_t n_params = 0;
    std::vector<size_t> w_off, b_off;
    float* w = nullptr;           // fp32 masters
    __nv_bfloat16* wb = nullptr;  // bf16 copies of the weight matrices (same offsets as w)
    float* g = nullptr;           // gradients
    float* m = nullptr;
    float* v = nullptr;           // Adam moments
    long long adam_t = 0;
    // activations for a batch
    int cap_B = 0;
    std::vector<float*> acts;     // acts[0] = input copy, acts[l] = output of layer l
    std::vector<float*> dacts;
    double* loss_dev = nullptr;
    float* Xb = nullptr;
    float* yb = nullptr;
    // partial sums of every layer's gradient (weights and biases) and of the loss
    std::vector<int> splits, chunk;
    std::vector<size_t> part_off;
    float* part = nullptr;
    double* loss_part = nullptr;
    int plan_B = 0;               // batch the partial sums are laid out for
    std::vector<void*> blocks;
    std::vector<size_t> block_bytes;
};

namespace {

void* mlp_alloc(Mlp& M, size_t bytes) {
    void* p = dev_alloc(bytes, nullptr);
    if (p) {
        M.blocks.push_back(p);
        M.block_bytes.push_back(bytes);
    }
    return p;
}

// rows per block of the head: groups of kHeadRows, at most kHeadBlocks blocks
int head_rows(int B) { return (B + kHeadRows * kHeadBlocks - 1) / (kHeadRows * kHeadBlocks) * kHeadRows; }
int head_blocks(int B) { return (B + head_rows(B) - 1) / head_rows(B); }

// most partial products of the weight gradient of layer l for batches up to B:
// enough for about 256 blocks
int max_splits(const Mlp& M, int l, int B) {
    if (l + 2 == (int)M.dims.size()) return std::min(kHeadBlocks, (B + kHeadRows - 1) / kHeadRows);
    const int tiles = ((M.dims[l + 1] + kBM - 1) / kBM) * ((M.dims[l] + kBN - 1) / kBN);
    return std::max(1, std::min((B + 63) / 64, 256 / tiles));
}

size_t layer_params(const Mlp& M, int l) { return (size_t)M.dims[l] * M.dims[l + 1] + M.dims[l + 1]; }

// Rows per partial product of each weight gradient, in whole k-steps.  A layer
// in one piece writes its gradient itself (splits 1).
void plan_splits(Mlp& M, int B) {
    const int L = (int)M.dims.size() - 1;
    for (int l = 0; l < L; ++l) {
        if (l + 1 == L) {
            M.splits[l] = head_blocks(B);   // the output layer's come from the head's blocks
            continue;
        }
        const int want = max_splits(M, l, B);
        M.chunk[l] = ((B + want - 1) / want + kBK - 1) / kBK * kBK;
        M.splits[l] = (B + M.chunk[l] - 1) / M.chunk[l];
    }
    M.plan_B = B;
}

// where the gradient of a layer, or its partial products, go
float* layer_part(Mlp& M, int l) { return M.splits[l] == 1 ? M.g + M.w_off[l] : M.part + M.part_off[l]; }

int ensure_batch(Mlp& M, int B) {
    if (B < 1) return NQS_ERR_ARG;
    if (B <= M.cap_B) return NQS_OK;
    M.cap_B = 0;   // until everything is there
    // activation buffers are re-allocated for the larger batch
    for (size_t i = 0; i < M.acts.size(); ++i) {
        dev_free(M.acts[i], 0, nullptr);
        dev_free(M.dacts[i], 0, nullptr);
    }
    dev_free(M.Xb, 0, nullptr);
    dev_free(M.yb, 0, nullptr);
    M.Xb = M.yb = nullptr;
    const int L = (int)M.dims.size();
    M.acts.assign(L, nullptr);
    M.dacts.assign(L, nullptr);
    for (int l = 0; l < L; ++l) {
        M.acts[l] = (float*)dev_alloc((size_t)B * M.dims[l] * sizeof(float), nullptr);
        M.dacts[l] = (float*)dev_alloc((size_t)B * M.dims[l] * sizeof(float), nullptr);
        if (!M.acts[l] || !M.dacts[l]) return NQS_ERR_NOMEM;
    }
    M.Xb = (float*)dev_alloc((size_t)B * M.dims[0] * sizeof(float), nullptr);
    M.yb = (float*)dev_alloc((size_t)B * sizeof(float), nullptr);
    if (!M.Xb || !M.yb) return NQS_ERR_NOMEM;
    dev_free(M.part, 0, nullptr);
    dev_free(M.loss_part, 0, nullptr);
    M.part = nullptr;
    M.loss_part = nullptr;
    // room for the partial products of any batch up to B
    M.splits.assign(L - 1, 1);
    M.chunk.assign(L - 1, 0);
    M.part_off.assign(L - 1, 0);
    M.plan_B = 0;
    size_t total = 0;
    for (int l = 0; l + 1 < L; ++l) {
        const int z = max_splits(M, l, B);
        M.part_off[l] = total;
        if (z > 1) total += z * layer_params(M, l);
    }
    M.part = (float*)dev_alloc(std::max<size_t>(total, 1) * sizeof(float), nullptr);
    M.loss_part = (double*)dev_alloc(kHeadBlocks * sizeof(double), nullptr);
    if (!M.part || !M.loss_part) return NQS_ERR_NOMEM;
    M.cap_B = B;
    return NQS_OK;
}

// whether the tiles of a layer may use vector loads: widths in whole float4s and
// every base aligned (weights lie at w_off; X is the caller's)
bool vector_loads(const Mlp& M, int l, const float* X) {
    return M.dims[l] % 4 == 0 && M.dims[l + 1] % 4 == 0 && M.w_off[l] % 4 == 0 && ((uintptr_t)X & 15) == 0;
}

void hidden_layers(Mlp& M, const float* X, int B, cudaStream_t st) {
    const int L = (int)M.dims.size() - 1;
    const float* in = X;
    for (int l = 0; l + 1 < L; ++l) {
        const int K = M.dims[l], N = M.dims[l + 1];
        const dim3 grid((N + kBN - 1) / kBN, (B + kBM - 1) / kBM);
        auto* const kernel = vector_loads(M, l, in) ? mlp_forward_kernel<true> : mlp_forward_kernel<false>;
        kernel<<<grid, kGemmThreads, 0, st>>>(B, N, K, in, M.wb + M.w_off[l], M.acts[l + 1], M.w + M.b_off[l], 1);
        in = M.acts[l + 1];
    }
}

// the head; with targets it starts the backward pass
void head(Mlp& M, const float* X, const float* y, int B, cudaStream_t st) {
    const int l = (int)M.dims.size() - 2;
    mlp_head_kernel<<<head_blocks(B), kHeadThreads, 0, st>>>(
        B, M.dims[l], head_rows(B), l == 0 ? X : M.acts[l], M.wb + M.w_off[l], M.w + M.b_off[l], M.acts[l + 1], y, M.dacts[l],
        M.loss_part, layer_part(M, l), l > 0);
}

int forward(Mlp& M, const float* X, int B, cudaStream_t st) {
    hidden_layers(M, X, B, st);
    head(M, X, nullptr, B, st);
    return cudaGetLastError() == cudaSuccess ? NQS_OK : NQS_ERR_CUDA;
}

// mean-squared error of the batch (X, y) and its gradients into M.g
int loss_and_gradient(Mlp& M, const float* X, const float* y, int B, cudaStream_t st) {
    const int L = (int)M.dims.size() - 1;
    if (B != M.plan_B) plan_splits(M, B);
    hidden_layers(M, X, B, st);
    head(M, X, y, B, st);
    for (int l = L - 2; l >= 0; --l) {
        LayerBack k{};
        k.B = B;
        k.out = M.dims[l + 1];
        k.in = M.dims[l];
        k.dx_tiles = l > 0 ? ((B + kBM - 1) / kBM) * ((k.in + kBN - 1) / kBN) : 0;
        k.splits = M.splits[l];
        k.chunk = M.chunk[l];
        k.dY = M.dacts[l + 1];
        k.X = l == 0 ? X : M.acts[l];
        k.W = M.wb + M.w_off[l];
        k.dX = M.dacts[l];
        k.part = layer_part(M, l);
        const int tiles = ((k.out + kBM - 1) / kBM) * ((k.in + kBN - 1) / kBN);
        auto* const kernel = vector_loads(M, l, k.X) ? mlp_backward_kernel<true> : mlp_backward_kernel<false>;
        kernel<<<k.dx_tiles + tiles * k.splits, kGemmThreads, 0, st>>>(k);
    }
    GradSums S{};
    S.layers = L;
    S.B = B;
    S.loss_parts = head_blocks(B);
    S.loss_part = M.loss_part;
    S.loss = M.loss_dev;
    for (int l = 0; l < L; ++l) {
        S.layer[l].part = layer_part(M, l);
        S.layer[l].splits = M.splits[l] == 1 ? 0 : M.splits[l];
        S.layer[l].count = (int)layer_params(M, l);
        S.layer[l].first = (int)M.w_off[l];
    }
    const int n = (int)M.n_params;
    mlp_gradient_kernel<<<std::min(1024, (n + 255) / 256), 256, 0, st>>>(S, M.g, n);
    return cudaGetLastError() == cudaSuccess ? NQS_OK : NQS_ERR_CUDA;
}

void refresh_bf16(Mlp& M, cudaStream_t st) {
    to_bf16_kernel<<<256, 256, 0, st>>>(M.w, M.wb, (int)M.n_params);
}

}  // namespace

void mlp_destroy(Mlp* M) {
    if (!M) return;
    cudaDeviceSynchronize();
    for (size_t i = 0; i < M->blocks.size(); ++i) dev_free(M->blocks[i], M->block_bytes[i], nullptr);
    for (size_t i = 0; i < M->acts.size(); ++i) {
        dev_free(M->acts[i], 0, nullptr);
        dev_free(M->dacts[i], 0, nullptr);
    }
    dev_free(M->Xb, 0, nullptr);
    dev_free(M->yb, 0, nullptr);
    dev_free(M->part, 0, nullptr);
    dev_free(M->loss_part, 0, nullptr);
    delete M;
}

int mlp_create(int n_in, int hidden, int layers, unsigned long long seed, Mlp** out) {
    if (n_in < 1 || n_in > 4096 || hidden < 1 || hidden > 4096 || layers < 1 || layers > 8) return NQS_ERR_ARG;
    Mlp* M = new Mlp();
    M->dims.push_back(n_in);
    for (int l = 0; l < layers; ++l) M->dims.push_back(hidden);
    M->dims.push_back(1);
    size_t off = 0;
    for (size_t l = 0; l + 1 < M->dims.size(); ++l) {
        M->w_off.push_back(off);
        off += (size_t)M->dims[l] * M->dims[l + 1];
        M->b_off.push_back(off);
        off += M->dims[l + 1];
    }
    M->n_params = off;
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights, zero biases, from SplitMix64
    std::vector<float> h(off, 0.f);
    unsigned long long state = seed;
    auto next = [&]() {
        state += 0x9E3779B97F4A7C15ull;
        unsigned long long z = state;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    for (size_t l = 0; l + 1 < M->dims.size(); ++l) {
        const double a = 1.0 / std::sqrt((double)M->dims[l]);
        for (size_t i = 0; i < (size_t)M->dims[l] * M->dims[l + 1]; ++i) {
            const double u = (next() >> 11) * (1.0 / 9007199254740992.0);
            h[M->w_off[l] + i] = (float)((2.0 * u - 1.0) * a);
        }
    }
    M->w = (float*)mlp_alloc(*M, off * sizeof(float));
    M->wb = (__nv_bfloat16*)mlp_alloc(*M, off * sizeof(__nv_bfloat16));
    M->g = (float*)mlp_alloc(*M, off * sizeof(float));
    M->m = (float*)mlp_alloc(*M, off * sizeof(float));
    M->v = (float*)mlp_alloc(*M, off * sizeof(float));
    M->loss_dev = (double*)mlp_alloc(*M, sizeof(double));
    if (!M->w || !M->wb || !M->g || !M->m || !M->v || !M->loss_dev) {
        mlp_destroy(M);
        return NQS_ERR_NOMEM;
    }
    if (cudaMemcpy(M->w, h.data(), off * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(M->m, 0, off * sizeof(float)) != cudaSuccess ||
        cudaMemset(M->v, 0, off * sizeof(float)) != cudaSuccess) {
        mlp_destroy(M);
        return NQS_ERR_CUDA;
    }
    refresh_bf16(*M, nullptr);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        mlp_destroy(M);
        return NQS_ERR_CUDA;
    }
    *out = M;
    return NQS_OK;
}

size_t mlp_n_params(const Mlp* M) { return M->n_params; }
int mlp_n_in(const Mlp* M) { return M->dims[0]; }

int mlp_get_params(Mlp* M, float* host, size_t cap) {
    if (cap < M->n_params) return NQS_ERR_ARG;
    return cudaMemcpy(host, M->w, M->n_params * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? NQS_OK
                                                                                                   : NQS_ERR_CUDA;
}

int mlp_set_params(Mlp* M, const float* host, size_t count) {
    if (count != M->n_params) return NQS_ERR_ARG;
    if (cudaMemcpy(M->w, host, count * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return NQS_ERR_CUDA;
    refresh_bf16(*M, nullptr);
    return cudaDeviceSynchronize() == cudaSuccess ? NQS_OK : NQS_ERR_CUDA;
}

int mlp_forward(Mlp* M, const float* X, int B, float* y, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    int rc = ensure_batch(*M, B);
    if (rc) return rc;
    rc = forward(*M, X, B, st);
    if (rc) return rc;
    return cudaMemcpyAsync(y, M->acts.back(), (size_t)B * sizeof(float), cudaMemcpyDefault, st) == cudaSuccess
               ? NQS_OK
               : NQS_ERR_CUDA;
}

int mlp_loss_grad(Mlp* M, const float* X, const float* y, int B, double* loss, float* grad_host, size_t cap,
                  void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    if (cap < M->n_params) return NQS_ERR_ARG;
    int rc = ensure_batch(*M, B);
    if (rc) return rc;
    rc = loss_and_gradient(*M, X, y, B, st);
    if (rc) return rc;
    if (cudaMemcpyAsync(loss, M->loss_dev, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess) return NQS_ERR_CUDA;
    if (cudaMemcpyAsync(grad_host, M->g, M->n_params * sizeof(float), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return NQS_ERR_CUDA;
    return cudaStreamSynchronize(st) == cudaSuccess ? NQS_OK : NQS_ERR_CUDA;
}

int mlp_train(Mlp* M, const float* X, const float* y, int n, int batch, int steps, float lr, unsigned long long seed,
              double* final_loss, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    if (n < 1 || batch < 1 || steps < 0) return NQS_ERR_ARG;
    int rc = ensure_batch(*M, batch);
    if (rc) return rc;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int s = 0; s < steps; ++s) {
        gather_batch_kernel<<<batch, 64, 0, st>>>(X, y, n, M->dims[0], M->Xb, M->yb, batch, seed, M->adam_t);
        rc = loss_and_gradient(*M, M->Xb, M->yb, batch, st);
        if (rc) return rc;
        ++M->adam_t;
        const float c1 = 1.f - std::pow(b1, (float)M->adam_t), c2 = 1.f - std::pow(b2, (float)M->adam_t);
        adam_kernel<<<256, 256, 0, st>>>(M->w, M->wb, M->g, M->m, M->v, (int)M->n_params, lr, b1, b2, eps, c1, c2);
    }
    if (final_loss) {
        if (cudaMemcpyAsync(final_loss, M->loss_dev, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess)
            return NQS_ERR_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return NQS_ERR_CUDA;
    }
    return cudaGetLastError() == cudaSuccess ? NQS_OK : NQS_ERR_CUDA;
}

}  // namespace nqs
