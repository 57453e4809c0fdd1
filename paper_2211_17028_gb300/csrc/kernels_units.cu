// Unit sweep kernel for sm_103a: many states ("units"), each swept through one
// pass of its schedule, in one launch.
//
// A tile is 12 qubits (4096 amplitudes) of one state; a block of 256 threads
// holds it in registers, 16 amplitudes per thread, and takes every
// unit_ctas-th tile of its unit.  The next tile comes into shared memory by
// TMA bulk copies (256-byte runs of the five low qubits) while the current one
// is processed; every wait on the copies' mbarrier is bounded.
//
// What bounds it: instructions wherever the launch fills the chip (24 qubits: an
// instruction issued in 51 to 54 % of the cycles of a scheduler with 5.6 warps, three
// in ten of them FMA-pipe instructions, the rest decoding, swapping halves and
// forming addresses; the largest stalls are fixed latencies, phi loads, barriers
// and instruction fetches; DRAM at 17 to 27 % of its peak), the latency of one
// tile where it does not.  Hence
// * one state per block and two or three blocks per SM, instead of the three
//   states of a branch group in one block of 512 threads: three times as many
//   blocks on a narrow circuit, and twice the amplitudes per decoded operation;
// * the program says what to do with pending diagonal factors (unit_program.h),
//   so an operation is a record, a jump and its arithmetic: no flags, no
//   loops over register bits;
// * the gates of a layer, up to one per register bit, share a record, and that
//   record is tested for first: decoding is a tree of compares (no jump table),
//   ten branches per operation;
// * thread bits and the bits of the tile's number sit in one word, so a
//   diagonal on any qubit outside the registers is one indexed table read;
// * the re-layout buffers are padded (index j at j + j/16 + j/256: additive, and
//   lanes on positions of distinct residue mod 4 meet distinct banks).
// The order of an amplitude's operations is the circuit's: the lowest level of
// a basis test state is one amplitude, whose error of about 1e-6 is the rounding
// of this order.  Gates as a phase and a real rotation (a third of the products)
// in an order of half as many phases ran 20 qubits level 2 in 5.4 ms, and rounded
// that amplitude up to three times worse on some inputs.
#include <algorithm>

#include "mbar.cuh"
#include "nqs_internal.h"
#include "unit_program.h"

namespace nqs {

namespace {

constexpr int kAmps = 1 << kMaxTileQ;
constexpr int kE = 1 << kUnitRB;
constexpr int kNT = kUnitThreads;
constexpr int kNW = kNT / 32;
constexpr int kChunk = 32;
constexpr int kChunks = kAmps / kChunk;
// padded index maps, additive over disjoint bits of j
__device__ __forceinline__ int relay_map(int j) { return j + (j >> 4) + (j >> 8); }
// staging: whole 32-amplitude runs stay contiguous and 16-byte aligned
__device__ __forceinline__ int stage_map(int j) { return j + 2 * (j >> 5) + 2 * (j >> 9); }
constexpr int kRelayAmps = kAmps + (kAmps >> 4) + (kAmps >> 8);
constexpr int kStageAmps = kAmps + 2 * (kAmps >> 5) + 2 * (kAmps >> 9);
// Two forms of the kernel.  Two blocks per SM: 128 registers, two alternating
// re-layout buffers.  Three blocks: 80 registers (30 words spilled) and one
// buffer with a second barrier per re-layout; half as many warps again hide more
// of the latency of decoding and of the sites' loads, so it is used where the
// launch has blocks for it and the program leaves room (5 % less time on 20
// qubits at level 2; 7 % more on 13 qubits, whose 66 tiles do not fill the chip).
constexpr int relay_bufs(int blocks) { return blocks == 2 ? 2 : 1; }
constexpr size_t fixed_smem(int blocks) { return ((size_t)kStageAmps + relay_bufs(blocks) * kRelayAmps) * sizeof(float2); }

// An amplitude is one 64-bit register pair (re in the low word) and every
// product on it a packed FP32x2 operation written as such: kept as two floats,
// every operation moved its sixteen amplitudes between register pairs (half of
// all instructions issued, 7470 per warp and tile of 27 gates).
typedef unsigned long long c64;

__device__ __forceinline__ c64 pk(float lo, float hi) {
    c64 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ float2 unpk(c64 v) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
__device__ __forceinline__ c64 swp(c64 v) {
    const float2 f = unpk(v);
    return pk(f.y, f.x);
}
__device__ __forceinline__ c64 mul2(c64 a, c64 b) {
    c64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ c64 fma2(c64 a, c64 b, c64 c) {
    c64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// A complex factor m as the two packed operands of a product:
//   m a = (m.x, m.x) * (a.x, a.y) + (-m.y, m.y) * (a.y, a.x)
struct Fac {
    c64 p, q;
};
__device__ __forceinline__ Fac fac(float2 m) { return Fac{pk(m.x, m.x), pk(-m.y, m.y)}; }
// (the products in the order of cmul and cfma)
__device__ __forceinline__ c64 mulc(Fac m, c64 a) { return fma2(m.p, a, mul2(m.q, swp(a))); }
__device__ __forceinline__ c64 fmac(Fac m, c64 a, c64 acc) { return fma2(m.p, a, fma2(m.q, swp(a), acc)); }
// m times f
__device__ __forceinline__ Fac times(Fac m, float2 f) {
    return fac(cmul(make_float2(unpk(m.p).x, unpk(m.q).y), f));
}
__device__ __forceinline__ Fac times_real(Fac m, float f) { return Fac{mul2(pk(f, f), m.p), mul2(pk(f, f), m.q)}; }
__device__ __forceinline__ Fac ld_fac(const float2* m) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(m);
    return Fac{v.x, v.y};
}

// y0 = m0 a + m1 b, y1 = m2 a + m3 b on register bit I.  A state swept alone
// adds the products as cfma(m0, a, cmul(m1, b)), the states of a branch group
// in the order (m0 a, m1 b): both orders are kept, so results do not depend on
// which kernel sweeps them.
template <int I, bool SINGLE>
__device__ __forceinline__ void u_dense(c64 (&x)[kE], const Fac (&k)[4]) {
#pragma unroll
    for (int r = 0; r < kE; ++r) {
        if (r & (1 << I)) continue;
        const c64 a = x[r], b = x[r | (1 << I)];
        const c64 as = swp(a), bs = swp(b);
        c64 y0, y1;
        if (SINGLE) {
            y1 = fma2(k[2].p, a, fma2(k[2].q, as, fma2(k[3].p, b, mul2(k[3].q, bs))));
            y0 = fma2(k[0].p, a, fma2(k[0].q, as, fma2(k[1].p, b, mul2(k[1].q, bs))));
        } else {
            y1 = fma2(k[3].q, bs, fma2(k[3].p, b, fma2(k[2].q, as, mul2(k[2].p, a))));
            y0 = fma2(k[1].q, bs, fma2(k[1].p, b, fma2(k[0].q, as, mul2(k[0].p, a))));
        }
        x[r] = y0;
        x[r | (1 << I)] = y1;
    }
}

// pending factors: a scalar and a pair or a ratio per register bit
template <bool PAIRS>
struct Pend {
    static constexpr int W = PAIRS ? 2 : 1;
    float2 d, h[kUnitRB][W];
    __device__ __forceinline__ void clear(int i) {
#pragma unroll
        for (int w = 0; w < W; ++w) h[i][w] = make_float2(1.f, 0.f);
    }
    __device__ __forceinline__ void clear() {
        d = make_float2(1.f, 0.f);
#pragma unroll
        for (int i = 0; i < kUnitRB; ++i) clear(i);
    }
};

// the dense gate of a record: its matrix with the pending factors it takes
template <int I, bool SINGLE, bool PAIRS>
__device__ __forceinline__ void u_gate(c64 (&x)[kE], const UnitRec& op, const float2* __restrict__ mats, Pend<PAIRS>& P,
                                       uint32_t bits) {
    const int fl = (int)(op.mask >> (8 * I));
    if (!(fl & UF_HERE)) return;
    const float2* const m = mats + op.off[I] + 2;
    Fac k[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) k[e] = ld_fac(m + 2 * e);
    if (fl & UF_SCALAR) {
        if (fl & UF_REAL) {
#pragma unroll
            for (int e = 0; e < 4; ++e) k[e] = times_real(k[e], P.d.x);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) k[e] = times(k[e], P.d);
        }
        P.d = make_float2(1.f, 0.f);
    }
    if (fl & UF_DIAG) {
        if (PAIRS) {
            k[0] = times(k[0], P.h[I][0]);
            k[2] = times(k[2], P.h[I][0]);
        }
        k[1] = times(k[1], P.h[I][PAIRS ? 1 : 0]);
        k[3] = times(k[3], P.h[I][PAIRS ? 1 : 0]);
        P.clear(I);
    }
    if (fl & UF_SIGN) {
        const float f = (__popc(bits & __float_as_uint(m[-2].x)) & 1) ? -1.f : 1.f;
        k[1] = times_real(k[1], f);
        k[3] = times_real(k[3], f);
    }
    u_dense<I, SINGLE>(x, k);
}

// A dense two-qubit gate reads its matrix anew for every quadruple: 32 held
// entries next to the amplitudes would spill (these gates are rare: the
// planner turns controlled gates into diagonals wherever it can).  The pending
// scalar, then the product of the pairs (first qubit's first), multiply each entry.
__device__ __forceinline__ float2 lds_again(const float2* p) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(smem_u32(p)));
    return v;
}

template <int I0, int I1, bool PAIRS>
__device__ __forceinline__ void u_g2(c64 (&x)[kE], const UnitRec& op, const float2* __restrict__ m, Pend<PAIRS>& P) {
    float2 f[4];
    const bool pair = PAIRS && (op.flags & UF_DIAG), scal = PAIRS && (op.flags & UF_SCALAR);
    if (PAIRS) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            f[c] = cmul(P.h[I0][(c >> 1) & (P.W - 1)], P.h[I1][c & (P.W - 1)]);
        }
    }
    auto entry = [&](int q, int c) {
        float2 e = lds_again(m + 4 * q + c);
        if (scal) e = cmul(e, P.d);
        if (pair) e = cmul(e, f[c]);
        return fac(e);
    };
#pragma unroll
    for (int r = 0; r < kE; ++r) {
        if (r & ((1 << I0) | (1 << I1))) continue;
        const int idx[4] = {r, r | (1 << I1), r | (1 << I0), r | (1 << I0) | (1 << I1)};
        c64 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = x[idx[q]];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            c64 y = mulc(entry(q, 0), v[0]);
            y = fmac(entry(q, 1), v[1], y);
            y = fmac(entry(q, 2), v[2], y);
            x[idx[q]] = fmac(entry(q, 3), v[3], y);
        }
    }
    if (PAIRS) {
        P.d = make_float2(1.f, 0.f);
        P.clear(I0);
        P.clear(I1);
    }
}

// amplitudes *= f0 or f1 by register bit I
template <int I>
__device__ __forceinline__ void u_by_bit(c64 (&x)[kE], float2 f0, float2 f1) {
    const Fac k0 = fac(f0), k1 = fac(f1);
#pragma unroll
    for (int r = 0; r < kE; ++r) x[r] = mulc((r >> I & 1) ? k1 : k0, x[r]);
}

template <int I>
__device__ __forceinline__ void u_flush_sign(c64 (&x)[kE], float h) {
    const c64 f = pk(h, h);
#pragma unroll
    for (int r = 0; r < kE; ++r)
        if (r & (1 << I)) x[r] = mul2(f, x[r]);
}

template <int I0, int I1>
__device__ __forceinline__ void u_negate(c64 (&x)[kE]) {
#pragma unroll
    for (int r = 0; r < kE; ++r)
        if ((r >> I0 & 1) && (r >> I1 & 1)) x[r] = mul2(pk(-1.f, -1.f), x[r]);
}

__device__ __forceinline__ void u_negate_pairs(c64 (&x)[kE], int pairs) {
    if (pairs & 1) u_negate<0, 1>(x);
    if (pairs & 2) u_negate<0, 2>(x);
    if (pairs & 4) u_negate<0, 3>(x);
    if (pairs & 8) u_negate<1, 2>(x);
    if (pairs & 16) u_negate<1, 3>(x);
    if (pairs & 32) u_negate<2, 3>(x);
}

template <int I0, int I1, bool PAIRS>
__device__ __forceinline__ void u_diag2(c64 (&x)[kE], const float2* __restrict__ m) {
#pragma unroll
    for (int c = PAIRS ? 0 : 3; c < 4; ++c) {
        const Fac f = fac(m[PAIRS ? c : 0]);
#pragma unroll
        for (int r = 0; r < kE; ++r)
            if (2 * (r >> I0 & 1) + (r >> I1 & 1) == c) x[r] = mulc(f, x[r]);
    }
}

// real factors of a diagonal K_0
template <int I>
__device__ __forceinline__ void u_by_bit_real(c64 (&x)[kE], float f0, float f1) {
    const c64 k0 = pk(f0, f0), k1 = pk(f1, f1);
#pragma unroll
    for (int r = 0; r < kE; ++r) x[r] = mul2((r >> I & 1) ? k1 : k0, x[r]);
}

template <int I>
__device__ __forceinline__ void u_ratio(c64 (&x)[kE], float2 h) {
    const Fac k = fac(h);
#pragma unroll
    for (int r = 0; r < kE; ++r)
        if (r & (1 << I)) x[r] = mulc(k, x[r]);
}

// tile index bits of the thread in a phase (those of the register bits are
// read again where they are used: held, they would spill)
__device__ __forceinline__ int thread_j(const UnitPhase& ph, int lane, int warp) {
    return ph.lane_j[lane] | ph.warp_j[warp];
}

// the tile's registers to or from a buffer under an additive index map
template <bool STORE, typename Map>
__device__ __forceinline__ void move_tile(c64 (&x)[kE], float2* buf, const UnitPhase& ph, int jT, Map map) {
    c64* const w = reinterpret_cast<c64*>(buf) + map(jT);
    int o[kUnitRB];
#pragma unroll
    for (int i = 0; i < kUnitRB; ++i) o[i] = map(ph.reg_j[i]);
#pragma unroll
    for (int r = 0; r < kE; ++r) {
        c64* const a =
            w + (((r & 1) ? o[0] : 0) + ((r & 2) ? o[1] : 0) + ((r & 4) ? o[2] : 0) + ((r & 8) ? o[3] : 0));
        if (STORE) *a = x[r];
        else x[r] = *a;
    }
}

__device__ __forceinline__ unsigned long long glob(const unsigned long long* hi_off, int j) {
    return hi_off[j >> 5] | (unsigned long long)(j & 31);
}

// Addresses of a thread's amplitudes in a state: sums over the register bits.
struct Addr {
    unsigned long long lo[4], hi[4];   // offsets of the bit pairs 0-1 and 2-3
    __device__ __forceinline__ Addr(const unsigned long long* hi_off, const UnitPhase& ph, unsigned long long at) {
        unsigned long long g[kUnitRB];
#pragma unroll
        for (int i = 0; i < kUnitRB; ++i) g[i] = glob(hi_off, ph.reg_j[i]);
        lo[0] = 0;
        lo[1] = g[0];
        lo[2] = g[1];
        lo[3] = g[0] + g[1];
        hi[0] = at;
        hi[1] = at + g[2];
        hi[2] = at + g[3];
        hi[3] = hi[1] + g[3];
    }
    __device__ __forceinline__ unsigned long long operator()(int r) const { return hi[r >> 2] + lo[r & 3]; }
};

template <int I, bool SINGLE>
__device__ __forceinline__ void u_site(const UnitRec& op, const float2* __restrict__ m, c64 (&x)[kE],
                                       const UnitPhase& ph, int jT, const SweepUnit& u, const unsigned long long* hi_off,
                                       float2* const* slot, unsigned long long base, double* acc, int lane, int warp) {
    const int fl = op.flags;
    // the addresses are the same for every site of a phase; opaque here, or the
    // compiler computes all of them ahead of the operation loop and spills
    asm volatile("" : "+r"(jT));
    const Addr off(hi_off, ph, base | glob(hi_off, jT));
    if (SINGLE && (fl & (FL_SAVE | FL_SAVE_FWD))) {   // branch groups save nothing
        c64* const save = reinterpret_cast<c64*>(slot[op.ev]);
#pragma unroll
        for (int r = 0; r < kE; ++r) __stcs(save + off(r), x[r]);
    }
    if (fl & FL_REDUCE) {
        // conj(f) a accumulated as A += (f.x a.x, f.y a.y), B += (f.x a.y, f.y a.x):
        // conj(f) a = (A.x + A.y, B.x - B.y).  The swapped amplitudes serve both
        // values of phi, and phi is used as it was loaded.
        const c64* const phi = reinterpret_cast<const c64*>(slot[op.ev]);
        c64 A[4], B[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) A[e] = B[e] = pk(0.f, 0.f);
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // phi in two halves of eight loads in flight
            c64 f[kE / 2];
            int k = 0;
#pragma unroll
            for (int r = 0; r < kE; ++r) {
                if (r & (1 << I)) continue;
                if (((r >> (I == 3 ? 2 : 3)) & 1) != h) continue;
                f[k++] = __ldg(phi + off(r));
                f[k++] = __ldg(phi + off(r | (1 << I)));
            }
            k = 0;
#pragma unroll
            for (int r = 0; r < kE; ++r) {
                if (r & (1 << I)) continue;
                if (((r >> (I == 3 ? 2 : 3)) & 1) != h) continue;
                const c64 f0 = f[k], f1 = f[k + 1];
                k += 2;
                const c64 a = x[r], b = x[r | (1 << I)], as = swp(a), bs = swp(b);
                A[0] = fma2(f0, a, A[0]);
                B[0] = fma2(f0, as, B[0]);
                A[1] = fma2(f0, b, A[1]);
                B[1] = fma2(f0, bs, B[1]);
                A[2] = fma2(f1, a, A[2]);
                B[2] = fma2(f1, as, B[2]);
                A[3] = fma2(f1, b, A[3]);
                B[3] = fma2(f1, bs, B[3]);
            }
        }
        float v[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 a = unpk(A[e]), b = unpk(B[e]);
            float2 R = make_float2(a.x + a.y, b.x - b.y);
            if (!SINGLE) R = cmul(m[0], R);   // the scale of the state
            v[2 * e] = R.x;
            v[2 * e + 1] = R.y;
        }
        // reduce-scatter over the warp: steps 16, 8, 4 halve the components a
        // lane keeps, steps 2, 1 complete the sum
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
        if ((lane & 3) == 0) {
            const int e = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
            acc[(op.ev * kNW + warp) * 8 + e] += (double)v[0];
        }
    }
    if (fl & FL_SPAWN) {
#pragma unroll 1
        for (int i = 0; i < op.nspawn; ++i) {
            Fac K[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) K[e] = fac(m[2 + 4 * i + e]);
            c64* const dst = reinterpret_cast<c64*>(u.spawn) + ((size_t)(3 * op.sp + i) << u.n);
#pragma unroll
            for (int r = 0; r < kE; ++r) {
                if (r & (1 << I)) continue;
                const c64 a = x[r], b = x[r | (1 << I)];
                __stcs(dst + off(r), fmac(K[0], a, mulc(K[1], b)));
                __stcs(dst + off(r | (1 << I)), fmac(K[2], a, mulc(K[3], b)));
            }
        }
    }
}

template <bool SINGLE, bool PAIRS, int BLOCKS>
__global__ void __launch_bounds__(kNT, BLOCKS) unit_sweep_kernel(const SweepUnit* __restrict__ units,
                                                                const int* __restrict__ blk, int ctas) {
    constexpr int kRelayBufs = relay_bufs(BLOCKS);
    constexpr size_t kFixedSmem = fixed_smem(BLOCKS);
    extern __shared__ __align__(128) unsigned char dyn[];
    float2* const stage = reinterpret_cast<float2*>(dyn);
    float2* const relay = stage + kStageAmps;                                  // one or two buffers
    __shared__ __align__(16) SweepUnit u;
    __shared__ __align__(8) uint64_t bar;
    __shared__ unsigned long long hi_off[kChunks];
    __shared__ float2* slot[kUnitSlots];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ui = blk ? blk[blockIdx.x] : (int)blockIdx.x / ctas;
    if (tid < (int)(sizeof(SweepUnit) / sizeof(uint2)))
        reinterpret_cast<uint2*>(&u)[tid] = reinterpret_cast<const uint2*>(units + ui)[tid];
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // program, acc slots and chunk offsets
    uint4* const prog = reinterpret_cast<uint4*>(dyn + kFixedSmem);
    const UnitHeader* const ghd = reinterpret_cast<const UnitHeader*>(u.prog);
    const int words = (int)ghd->words, n_events = (int)ghd->n_events;
    for (int i = tid; i < words; i += kNT) prog[i] = u.prog[i];
    double* const acc = reinterpret_cast<double*>(prog + words);
    for (int i = tid; i < n_events * kNW * 8; i += kNT) acc[i] = 0.0;
    for (int h = tid; h < kChunks; h += kNT) {
        unsigned long long o = 0;
#pragma unroll
        for (int j = 0; j < kMaxTileQ - 5; ++j)
            if ((h >> j) & 1) o |= 1ull << ghd->local[5 + j];
        hi_off[h] = o;
    }
    if (tid < (int)ghd->n_slots) {
        const unsigned s = ghd->slot_site[tid];
        slot[tid] = (s & 0x8000) ? u.ckpt_fwd[s & 0x7fff] : u.ckpt[s];
    }
    __syncthreads();
    const UnitHeader& hd = *reinterpret_cast<const UnitHeader*>(prog);
    const UnitPhase* const phases = reinterpret_cast<const UnitPhase*>(prog + 4);
    const UnitRec* const ops = reinterpret_cast<const UnitRec*>(prog + hd.ops_word);
    const float2* const mats = reinterpret_cast<const float2*>(prog + hd.mats_word);
    const int n_phases = (int)hd.n_phases, n_tiles = u.n_tiles, nctas = u.ctas;
    const int cta = blk ? (int)blockIdx.x - u.cta_begin : (int)blockIdx.x - ui * ctas;
    const unsigned long long nl = hd.nl_mask;

    // bits of the tile number on the qubits outside the tile
    auto tile_base = [&](int t) {
        unsigned long long b = 0, mk = nl;
        while (mk && t) {
            const unsigned long long low = mk & (~mk + 1ull);
            if (t & 1) b |= low;
            t >>= 1;
            mk ^= low;
        }
        return b;
    };
    // every thread issues its share of the copies; the mbarrier phase cannot
    // complete before thread 0's arrive.expect_tx, whatever lands first.  The
    // tile's phi values are brought to L2 meanwhile.
    auto prefetch = [&](unsigned long long b) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (tid == 0) mbar_arrive_expect_tx(&bar, (uint32_t)(kAmps * sizeof(float2)));
        if (tid < kChunks)
            bulk_copy_g2s(stage + stage_map(tid * kChunk), u.in + (b | hi_off[tid]), kChunk * sizeof(float2), &bar);
        for (int q = tid; q < n_events * kChunks; q += kNT)
            bulk_prefetch_l2(slot[q / kChunks] + (b | hi_off[q % kChunks]), kChunk * sizeof(float2));
    };

    // the next tile's base: the tile number's bits lie on the set bits of nl, so
    // with ones everywhere else a carry runs from one of them to the next
    const unsigned long long step = tile_base(nctas);
    unsigned long long base = tile_base(cta), next = base;
    if (cta < n_tiles) prefetch(base);
    uint32_t parity = 0;
    bool failed = false;
    c64 x[kE];
    int buf = 0;   // re-layout buffer to write next

    for (int t = cta; t < n_tiles; t += nctas) {
        const uint32_t bits = (uint32_t)tid | ((uint32_t)t << 8);
        const bool ok = mbar_wait_bounded(&bar, parity);
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        base = next;
        next = ((base | ~nl) + step) & nl;
        parity ^= 1u;
        int jT = thread_j(phases[0], lane, warp);
        move_tile<false>(x, stage, phases[0], jT, stage_map);
        __syncthreads();   // the staging buffer is free again
        if (t + nctas < n_tiles) prefetch(next);
        const float2 unit1 = make_float2(1.f, 0.f);
        Pend<PAIRS> P;
        P.clear();

#pragma unroll 1
        for (int p = 0; p < n_phases; ++p) {
            if (p > 0) {
                float2* const tb = relay + buf * kRelayAmps;
                if (kRelayBufs == 2) buf ^= 1;
                move_tile<true>(x, tb, phases[p - 1], jT, relay_map);
                __syncthreads();
                jT = thread_j(phases[p], lane, warp);
                move_tile<false>(x, tb, phases[p], jT, relay_map);
                if (kRelayBufs == 1) __syncthreads();
            }
            const int oe = phases[p].op_end;
#pragma unroll 1
            for (int o = phases[p].op_begin; o < oe; ++o) {
                const UnitRec op = ops[o];
                const float2* const m = mats + op.mat;
                const int c = (bits >> op.a) & 1;
#define U_COMMA ,
#define U_FOUR(F, BODY)                                  \
    case F + 0: { constexpr int I = 0; BODY; break; }    \
    case F + 1: { constexpr int I = 1; BODY; break; }    \
    case F + 2: { constexpr int I = 2; BODY; break; }    \
    case F + 3: { constexpr int I = 3; BODY; break; }
#define U_PAIRS(F, BODY)                                      \
    case F + 0: { constexpr int I = 0, J = 1; BODY; break; }  \
    case F + 1: { constexpr int I = 0, J = 2; BODY; break; }  \
    case F + 2: { constexpr int I = 0, J = 3; BODY; break; }  \
    case F + 3: { constexpr int I = 1, J = 2; BODY; break; }  \
    case F + 4: { constexpr int I = 1, J = 3; BODY; break; }  \
    case F + 5: { constexpr int I = 2, J = 3; BODY; break; }
                if (op.code == UO_G1) {   // the most frequent one, ahead of the tree of the others
                    if (op.a) u_negate_pairs(x, op.a);
                    u_gate<0, SINGLE, PAIRS>(x, op, mats, P, bits);
                    u_gate<1, SINGLE, PAIRS>(x, op, mats, P, bits);
                    u_gate<2, SINGLE, PAIRS>(x, op, mats, P, bits);
                    u_gate<3, SINGLE, PAIRS>(x, op, mats, P, bits);
                    continue;
                }
                switch (op.code) {
                    U_FOUR(UO_GK, const Fac k[4] = {ld_fac(m) U_COMMA ld_fac(m + 2) U_COMMA ld_fac(m + 4) U_COMMA ld_fac(m + 6)};
                           (u_dense<I, true>(x, k)))
                    U_FOUR(UO_KD, if (op.flags & UF_REAL) u_by_bit_real<I>(x, m[0].x, m[1].x);
                           else u_by_bit<I>(x, m[0], m[1]))
                    U_FOUR(UO_FLB, if (PAIRS) u_by_bit<I>(x, cmul(P.d, P.h[I][0]), cmul(P.d, P.h[I][P.W - 1]));
                           else u_ratio<I>(x, P.h[I][0]);
                           if (PAIRS) P.d = unit1;
                           P.clear(I))
                    U_FOUR(UO_FLR, u_flush_sign<I>(x, (__popc(bits & op.mask) & 1) ? -1.f : 1.f))
                    U_FOUR(UO_HP, const int at = c * P.W; P.h[I][0] = cmul(P.h[I][0], m[at]);
                           if (PAIRS) P.h[I][P.W - 1] = cmul(P.h[I][P.W - 1], m[at + 1]))
                    U_FOUR(UO_SITE, (u_site<I, SINGLE>(op, m, x, phases[p], jT, u, hi_off, slot, base, acc, lane, warp)))
                    case UO_DN: u_negate_pairs(x, op.a); break;
                    U_PAIRS(UO_DG, (u_diag2<I, J, PAIRS>(x, m)))
                    U_PAIRS(UO_G2, (u_g2<I, J, PAIRS>(x, op, m, P)))
                    U_PAIRS(UO_G2 + 6, (u_g2<J, I, PAIRS>(x, op, m, P)))
                    case UO_SC: P.d = cmul(P.d, m[c + 2 * ((bits >> op.b) & 1)]); break;
                    case UO_FLS:
                        if (op.flags & UF_REAL) {
#pragma unroll
                            for (int r = 0; r < kE; ++r) x[r] = mul2(pk(P.d.x, P.d.x), x[r]);
                        } else {
                            const Fac f = fac(P.d);
#pragma unroll
                            for (int r = 0; r < kE; ++r) x[r] = mulc(f, x[r]);
                        }
                        P.d = unit1;
                        break;
                    case UO_FLA:
                        if (PAIRS) {
#pragma unroll
                            for (int g = 0; g < 4; ++g) {
                                const float2 f2 = cmul(cmul(P.d, P.h[0][g & (P.W - 1)]), P.h[1][(g >> 1) & (P.W - 1)]);
#pragma unroll
                                for (int h = 0; h < 4; ++h)
                                    x[g + 4 * h] = mulc(fac(cmul(cmul(f2, P.h[2][h & (P.W - 1)]), P.h[3][(h >> 1) & (P.W - 1)])),
                                                        x[g + 4 * h]);
                            }
                        } else {
                            float2 f[8];
                            f[0] = P.d;
                            f[1] = cmul(f[0], P.h[0][0]);
                            f[2] = cmul(f[0], P.h[1][0]);
                            f[3] = cmul(f[1], P.h[1][0]);
#pragma unroll
                            for (int r = 0; r < 4; ++r) f[4 + r] = cmul(f[r], P.h[2][0]);
#pragma unroll
                            for (int r = 0; r < 8; ++r) {
                                x[r] = mulc(fac(f[r]), x[r]);
                                x[8 + r] = mulc(fac(cmul(f[r], P.h[3][0])), x[8 + r]);
                            }
                        }
                        P.clear();
                        break;
                    default: break;
                }
#undef U_FOUR
#undef U_PAIRS
#undef U_COMMA
            }
        }
        // store the tile, unless only its reductions or spawned states were wanted
        if (u.out) {
            c64* const dst = reinterpret_cast<c64*>(u.out);
            const Addr off(hi_off, phases[n_phases - 1], base | glob(hi_off, jT));
#pragma unroll
            for (int r = 0; r < kE; ++r) __stcs(dst + off(r), x[r]);
        }
    }

    if (failed) {
        if (tid == 0) atomicExch(u.err, NQS_ERR_DEVICE_TIMEOUT);
        mbar_wait_bounded(&bar, parity);   // let copies still in flight land
        return;
    }
    __syncthreads();
    for (int i = tid; i < n_events * 8; i += kNT) {
        const int ev = i >> 3, e = i & 7;
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < kNW; ++w) v += acc[(ev * kNW + w) * 8 + e];
        u.partials[((size_t)ev * nctas + cta) * 8 + e] = v;
    }
}

// Failure-detection self-test: the sweep kernels' bounded mbarrier wait on a
// barrier that nothing ever arrives at.  The wait must give up (after about
// two seconds) and report it through the status word, leaving the context usable.
__global__ void bounded_wait_probe_kernel(int* status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bool ok = mbar_wait_bounded(&bar, 0);
    if (threadIdx.x == 0) *status = ok ? NQS_OK : NQS_ERR_DEVICE_TIMEOUT;
}

}  // namespace

size_t unit_smem_bytes(int max_words, int max_events) {
    return fixed_smem(2) + (size_t)max_words * 16 + (size_t)max_events * kNW * 8 * sizeof(double);
}

namespace {

using UnitKernel = void (*)(const SweepUnit*, const int*, int);

// branch groups mostly keep ratios; a diagonal with zeros has none
UnitKernel unit_kernel(int kind, int blocks) {
    if (kind == unit_kind(true, UM_PAIRS)) return unit_sweep_kernel<true, true, 2>;
    if (kind == unit_kind(false, UM_PAIRS)) return unit_sweep_kernel<false, true, 2>;
    if (kind == unit_kind(true, UM_RATIOS)) return blocks == 3 ? unit_sweep_kernel<true, false, 3> : unit_sweep_kernel<true, false, 2>;
    return blocks == 3 ? unit_sweep_kernel<false, false, 3> : unit_sweep_kernel<false, false, 2>;
}

// shared memory of the three-block form for a program that needs `smem` in the other
size_t smem_of(int blocks, size_t smem) { return smem - fixed_smem(2) + fixed_smem(blocks); }

int attribute(cudaDeviceAttr a) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, a, dev);
    return v;
}

}  // namespace

// whether three blocks of such a program fit an SM (1 KB per block is the
// system's; pairs in 80 registers would spill 900 bytes)
bool unit_three_blocks(int kind, size_t smem) {
    if (kind == unit_kind(true, UM_PAIRS) || kind == unit_kind(false, UM_PAIRS)) return false;
    static const size_t fixed = [] {
        cudaFuncAttributes a{};
        return cudaFuncGetAttributes(&a, unit_sweep_kernel<true, false, 3>) == cudaSuccess ? a.sharedSizeBytes : (size_t)2048;
    }();
    return 3 * (smem_of(3, smem) + fixed + 1024) <= (size_t)attribute(cudaDevAttrMaxSharedMemoryPerMultiprocessor);
}

int unit_blocks_per_sm(int kind, size_t smem) {
    if (unit_three_blocks(kind, smem)) return 3;
    int nb = 0;
    const UnitKernel k = unit_kernel(kind, 2);
    allow_dynamic_smem((const void*)k);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, kNT, smem);
    return nb > 0 ? nb : 1;
}

cudaError_t launch_units(int kind, const SweepUnit* units, const int* blk, int ctas, int total_ctas, size_t smem,
                         cudaStream_t st) {
    const int blocks = total_ctas > 2 * attribute(cudaDevAttrMultiProcessorCount) && unit_three_blocks(kind, smem) ? 3 : 2;
    const UnitKernel kernel = unit_kernel(kind, blocks);
    smem = smem_of(blocks, smem);
    const cudaError_t e = allow_dynamic_smem((const void*)kernel);
    if (e != cudaSuccess) return e;
    kernel<<<total_ctas, kNT, smem, st>>>(units, blk, ctas);
    return cudaGetLastError();
}

int selftest_bounded_wait(int* status, void* stream) {
    bounded_wait_probe_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(status);
    return cudaGetLastError() == cudaSuccess ? NQS_OK : NQS_ERR_CUDA;
}

}  // namespace nqs
