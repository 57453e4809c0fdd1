// Unit sweep kernel for sm_103a: many states ("units"), each swept through one
// pass of its schedule, in one launch.
//
// A tile is 12 qubits (4096 amplitudes) of one state; a block of 256 threads
// holds it in registers, 16 amplitudes per thread, and takes every
// unit_ctas-th tile of its unit.  The next tile comes into shared memory by
// TMA bulk copies (256-byte runs of the five low qubits) while the current one
// is processed; every wait on the copies' mbarrier is bounded.
//
// What bounds it: issue slots (a dense one-qubit gate is 8 FP32 multiply-adds
// per amplitude) wherever the launch fills the chip, the latency of one tile
// where it does not.  Hence
// * one state per block and two blocks per SM, instead of the three states of
//   a branch group in one block of 512 threads: three times as many blocks on
//   a narrow circuit, and twice the amplitudes per decoded operation;
// * the program says what to do with pending diagonal factors (unit_program.h),
//   so an operation is a record, a jump and its arithmetic: no flags, no
//   loops over register bits;
// * thread bits and the bits of the tile's number sit in one word, so a
//   diagonal on any qubit outside the registers is one indexed table read;
// * the re-layout buffers alternate (one barrier per re-layout) and are padded
//   (index j at j + j/16 + j/256: additive, and lanes on positions of distinct
//   residue mod 4 meet distinct banks).
// One pass of 2^20 amplitudes x 60 states with 24 dense gates: see the figures
// at launch_units.
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
constexpr size_t kFixedSmem = ((size_t)kStageAmps + 2 * kRelayAmps) * sizeof(float2);

template <int I>
__device__ __forceinline__ void u_g1(float2 (&x)[kE], float2 m0, float2 m1, float2 m2, float2 m3) {
    const float2 p0 = make_float2(m0.x, m0.x), q0 = make_float2(-m0.y, m0.y);
    const float2 p1 = make_float2(m1.x, m1.x), q1 = make_float2(-m1.y, m1.y);
    const float2 p2 = make_float2(m2.x, m2.x), q2 = make_float2(-m2.y, m2.y);
    const float2 p3 = make_float2(m3.x, m3.x), q3 = make_float2(-m3.y, m3.y);
#pragma unroll
    for (int r = 0; r < kE; ++r) {
        if (r & (1 << I)) continue;
        const int r1 = r | (1 << I);
        const float2 a = x[r], b = x[r1];
        const float2 as = make_float2(a.y, a.x), bs = make_float2(b.y, b.x);
        float2 y0 = __fmul2_rn(p0, a);
        float2 y1 = __fmul2_rn(p2, a);
        y0 = __ffma2_rn(q0, as, y0);
        y1 = __ffma2_rn(q2, as, y1);
        y0 = __ffma2_rn(p1, b, y0);
        y1 = __ffma2_rn(p3, b, y1);
        y0 = __ffma2_rn(q1, bs, y0);
        y1 = __ffma2_rn(q3, bs, y1);
        x[r] = y0;
        x[r1] = y1;
    }
}

// A dense two-qubit gate reads its matrix anew for every quadruple: 32 held
// entries next to the amplitudes would spill (these gates are rare: the
// planner turns controlled gates into diagonals wherever it can).
__device__ __forceinline__ float2 lds_again(const float2* p) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(smem_u32(p)));
    return v;
}

template <int I0, int I1>
__device__ __forceinline__ void u_g2(float2 (&x)[kE], const float2* __restrict__ m) {
#pragma unroll
    for (int r = 0; r < kE; ++r) {
        if (r & ((1 << I0) | (1 << I1))) continue;
        const int idx[4] = {r, r | (1 << I1), r | (1 << I0), r | (1 << I0) | (1 << I1)};
        float2 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = x[idx[q]];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float2 y = cmul(lds_again(m + 4 * q), v[0]);
            y = cfma(lds_again(m + 4 * q + 1), v[1], y);
            y = cfma(lds_again(m + 4 * q + 2), v[2], y);
            y = cfma(lds_again(m + 4 * q + 3), v[3], y);
            x[idx[q]] = y;
        }
    }
}

template <int I>
__device__ __forceinline__ void u_flush_bit(float2 (&x)[kE], float2 f) {
#pragma unroll
    for (int r = 0; r < kE; ++r)
        if (r & (1 << I)) x[r] = cmul(f, x[r]);
}

template <int I0, int I1>
__device__ __forceinline__ void u_both(float2 (&x)[kE], float2 f) {
#pragma unroll
    for (int r = 0; r < kE; ++r)
        if ((r >> I0 & 1) && (r >> I1 & 1)) x[r] = cmul(f, x[r]);
}

// layout of a phase: tile index bits of the thread and of each register bit
struct Lay {
    int jT, jR[kUnitRB];
};

__device__ __forceinline__ void load_lay(Lay& L, const UnitPhase& ph, int lane, int warp) {
    L.jT = ph.lane_j[lane] | ph.warp_j[warp];
#pragma unroll
    for (int i = 0; i < kUnitRB; ++i) L.jR[i] = ph.reg_j[i];
}

__device__ __forceinline__ unsigned long long glob(const unsigned long long* hi_off, int j) {
    return hi_off[j >> 5] | (unsigned long long)(j & 31);
}

template <int I>
__device__ __forceinline__ void u_site(const UnitRec& op, const float2* __restrict__ m, float2 (&x)[kE],
                                       const Lay& L, const SweepUnit& u, const unsigned long long* hi_off,
                                       float2* const* slot, unsigned long long base, double* acc, int lane, int warp) {
    const int fl = op.flags;
    // the addresses are the same for every site of a phase; opaque here, or the
    // compiler computes all of them ahead of the operation loop and spills
    int jT = L.jT;
    asm volatile("" : "+r"(jT));
    const unsigned long long gT = base | glob(hi_off, jT);
    unsigned long long gR[kUnitRB];
#pragma unroll
    for (int i = 0; i < kUnitRB; ++i) gR[i] = glob(hi_off, L.jR[i]);
    auto off = [&](int r) {
        unsigned long long g = gT;
#pragma unroll
        for (int i = 0; i < kUnitRB; ++i)
            if (r & (1 << i)) g |= gR[i];
        return g;
    };
    const float2 sc = m[0];
    if (fl & (FL_SAVE | FL_SAVE_FWD)) {
        float2* const save = slot[op.ev];
#pragma unroll
        for (int r = 0; r < kE; ++r) __stcs(save + off(r), cmul(sc, x[r]));   // sc = 1 leaves them as they are
    }
    if (fl & FL_REDUCE) {
        // conj(f) a accumulated as A += f.x a, B += f.y a (no swapped operands):
        // conj(f) a = (A.x + B.y, A.y - B.x)
        const float2* const phi = slot[op.ev];
        float2 A[4], B[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) A[e] = B[e] = make_float2(0.f, 0.f);
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // phi in two halves of eight loads in flight
            float2 f[kE / 2];
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
                const float2 f0 = f[k++], f1 = f[k++];
                const float2 a = x[r], b = x[r | (1 << I)];
                const float2 f0x = make_float2(f0.x, f0.x), f0y = make_float2(f0.y, f0.y);
                const float2 f1x = make_float2(f1.x, f1.x), f1y = make_float2(f1.y, f1.y);
                A[0] = __ffma2_rn(f0x, a, A[0]);
                B[0] = __ffma2_rn(f0y, a, B[0]);
                A[1] = __ffma2_rn(f0x, b, A[1]);
                B[1] = __ffma2_rn(f0y, b, B[1]);
                A[2] = __ffma2_rn(f1x, a, A[2]);
                B[2] = __ffma2_rn(f1y, a, B[2]);
                A[3] = __ffma2_rn(f1x, b, A[3]);
                B[3] = __ffma2_rn(f1y, b, B[3]);
            }
        }
        float v[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 R = cmul(sc, make_float2(A[e].x + B[e].y, A[e].y - B[e].x));
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
            const float2* K = m + 2 + 4 * i;
            const float2 k0 = K[0], k1 = K[1], k2 = K[2], k3 = K[3];
            float2* const dst = u.spawn + ((size_t)(3 * op.sp + i) << u.n);
#pragma unroll
            for (int r = 0; r < kE; ++r) {
                if (r & (1 << I)) continue;
                const float2 a = x[r], b = x[r | (1 << I)];
                __stcs(dst + off(r), cfma(k0, a, cmul(k1, b)));
                __stcs(dst + off(r | (1 << I)), cfma(k2, a, cmul(k3, b)));
            }
        }
    }
}

__global__ void __launch_bounds__(kNT, 2) unit_sweep_kernel(const SweepUnit* __restrict__ units,
                                                            const int* __restrict__ blk, int ctas) {
    extern __shared__ __align__(128) unsigned char dyn[];
    float2* const stage = reinterpret_cast<float2*>(dyn);
    float2* const relay = stage + kStageAmps;                                  // two buffers
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

    int t = cta;
    unsigned long long base_next = tile_base(t);
    if (t < n_tiles) prefetch(base_next);
    uint32_t parity = 0;
    bool failed = false;
    float2 x[kE];
    int buf = 0;   // re-layout buffer to write next

    for (; t < n_tiles; t += nctas) {
        const unsigned long long base = base_next;
        const uint32_t bits = (uint32_t)tid | ((uint32_t)t << 8);
        const bool ok = mbar_wait_bounded(&bar, parity);
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        parity ^= 1u;
        Lay L;
        load_lay(L, phases[0], lane, warp);
        {
            const float2* const p = stage + stage_map(L.jT);
            int o[kUnitRB];
#pragma unroll
            for (int i = 0; i < kUnitRB; ++i) o[i] = stage_map(L.jR[i]);
#pragma unroll
            for (int r = 0; r < kE; ++r)
                x[r] = p[((r & 1) ? o[0] : 0) + ((r & 2) ? o[1] : 0) + ((r & 4) ? o[2] : 0) + ((r & 8) ? o[3] : 0)];
        }
        __syncthreads();   // the staging buffer is free again
        if (t + nctas < n_tiles) {
            base_next = tile_base(t + nctas);
            prefetch(base_next);
        }
        // pending diagonal: a scalar and a ratio per register bit
        const float2 unit1 = make_float2(1.f, 0.f);
        float2 dsc = unit1, h0 = unit1, h1 = unit1, h2 = unit1, h3 = unit1;

#pragma unroll 1
        for (int p = 0; p < n_phases; ++p) {
            if (p > 0) {
                float2* const tb = relay + buf * kRelayAmps;
                buf ^= 1;
                {
                    float2* const w = tb + relay_map(L.jT);
                    int o[kUnitRB];
#pragma unroll
                    for (int i = 0; i < kUnitRB; ++i) o[i] = relay_map(L.jR[i]);
#pragma unroll
                    for (int r = 0; r < kE; ++r)
                        w[((r & 1) ? o[0] : 0) + ((r & 2) ? o[1] : 0) + ((r & 4) ? o[2] : 0) + ((r & 8) ? o[3] : 0)] = x[r];
                }
                __syncthreads();
                load_lay(L, phases[p], lane, warp);
                {
                    const float2* const w = tb + relay_map(L.jT);
                    int o[kUnitRB];
#pragma unroll
                    for (int i = 0; i < kUnitRB; ++i) o[i] = relay_map(L.jR[i]);
#pragma unroll
                    for (int r = 0; r < kE; ++r)
                        x[r] = w[((r & 1) ? o[0] : 0) + ((r & 2) ? o[1] : 0) + ((r & 4) ? o[2] : 0) + ((r & 8) ? o[3] : 0)];
                }
            }
            const int oe = phases[p].op_end;
#pragma unroll 1
            for (int o = phases[p].op_begin; o < oe; ++o) {
                const UnitRec op = ops[o];
                const float2* const m = mats + op.mat;
                const int c = (bits >> op.a) & 1;
                // one branch per family, the common ones first
                const int code = op.code;
                if (code < UO_FLB) {
                    float2 m0 = m[0], m1 = m[1], m2 = m[2], m3 = m[3];
                    const int i = code & 3;
                    if (code >= UO_G1H) {
                        const float2 h = i == 0 ? h0 : i == 1 ? h1 : i == 2 ? h2 : h3;
                        m1 = cmul(m1, h);
                        m3 = cmul(m3, h);
                        if (i == 0) h0 = unit1;
                        else if (i == 1) h1 = unit1;
                        else if (i == 2) h2 = unit1;
                        else h3 = unit1;
                    }
                    if (i == 0) u_g1<0>(x, m0, m1, m2, m3);
                    else if (i == 1) u_g1<1>(x, m0, m1, m2, m3);
                    else if (i == 2) u_g1<2>(x, m0, m1, m2, m3);
                    else u_g1<3>(x, m0, m1, m2, m3);
                } else if (code < UO_HP) {
                    if (code == UO_FLB) {
                        u_flush_bit<0>(x, h0);
                        h0 = unit1;
                    } else if (code == UO_FLB + 1) {
                        u_flush_bit<1>(x, h1);
                        h1 = unit1;
                    } else if (code == UO_FLB + 2) {
                        u_flush_bit<2>(x, h2);
                        h2 = unit1;
                    } else {
                        u_flush_bit<3>(x, h3);
                        h3 = unit1;
                    }
                } else if (code < UO_SITE) {
                    float2 f;
                    if (code < UO_HR) {
                        const float4 q = *reinterpret_cast<const float4*>(m + 2 * c);
                        dsc = cmul(make_float2(q.x, q.y), dsc);
                        f = make_float2(q.z, q.w);
                    } else {
                        f = m[c];
                    }
                    const int i = code & 3;
                    if (i == 0) h0 = cmul(f, h0);
                    else if (i == 1) h1 = cmul(f, h1);
                    else if (i == 2) h2 = cmul(f, h2);
                    else h3 = cmul(f, h3);
                } else if (code < UO_SC) {
                    if (code == UO_SITE) u_site<0>(op, m, x, L, u, hi_off, slot, base, acc, lane, warp);
                    else if (code == UO_SITE + 1) u_site<1>(op, m, x, L, u, hi_off, slot, base, acc, lane, warp);
                    else if (code == UO_SITE + 2) u_site<2>(op, m, x, L, u, hi_off, slot, base, acc, lane, warp);
                    else u_site<3>(op, m, x, L, u, hi_off, slot, base, acc, lane, warp);
                } else if (code == UO_SC) {
                    dsc = cmul(m[c + 2 * ((bits >> op.b) & 1)], dsc);
                } else if (code == UO_FLS) {
#pragma unroll
                    for (int r = 0; r < kE; ++r) x[r] = cmul(dsc, x[r]);
                    dsc = unit1;
                } else if (code == UO_FLA) {
                    float2 f[8];
                    f[0] = dsc;
                    f[1] = cmul(f[0], h0);
                    f[2] = cmul(f[0], h1);
                    f[3] = cmul(f[1], h1);
#pragma unroll
                    for (int r = 0; r < 4; ++r) f[4 + r] = cmul(f[r], h2);
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        x[r] = cmul(f[r], x[r]);
                        f[r] = cmul(f[r], h3);
                        x[8 + r] = cmul(f[r], x[8 + r]);
                    }
                    dsc = h0 = h1 = h2 = h3 = unit1;
                } else if (code < UO_G2) {
                    const float2 f = m[0];
                    switch (code - UO_DD) {
                        case 0: u_both<0, 1>(x, f); break;
                        case 1: u_both<0, 2>(x, f); break;
                        case 2: u_both<0, 3>(x, f); break;
                        case 3: u_both<1, 2>(x, f); break;
                        case 4: u_both<1, 3>(x, f); break;
                        default: u_both<2, 3>(x, f); break;
                    }
                } else if (code < UO_DP) {
                    switch (code - UO_G2) {
                        case 0: u_g2<0, 1>(x, m); break;
                        case 1: u_g2<0, 2>(x, m); break;
                        case 2: u_g2<0, 3>(x, m); break;
                        case 3: u_g2<1, 2>(x, m); break;
                        case 4: u_g2<1, 3>(x, m); break;
                        default: u_g2<2, 3>(x, m); break;
                    }
                } else if (code == UO_DP) {
#pragma unroll
                    for (int r = 0; r < kE; ++r) x[r] = cmul(m[2 * c + ((r >> op.b) & 1)], x[r]);
                } else {
#pragma unroll
                    for (int r = 0; r < kE; ++r) x[r] = cmul(m[2 * ((r >> op.a) & 1) + ((r >> op.b) & 1)], x[r]);
                }
            }
        }
        // store the tile
        {
            float2* const dst = u.out + (base | glob(hi_off, L.jT));
            unsigned long long g[kUnitRB];
#pragma unroll
            for (int i = 0; i < kUnitRB; ++i) g[i] = glob(hi_off, L.jR[i]);
#pragma unroll
            for (int r = 0; r < kE; ++r)
                __stcs(dst + ((r & 1) ? g[0] : 0ull) + ((r & 2) ? g[1] : 0ull) + ((r & 4) ? g[2] : 0ull) +
                           ((r & 8) ? g[3] : 0ull),
                       x[r]);
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
    return kFixedSmem + (size_t)max_words * 16 + (size_t)max_events * kNW * 8 * sizeof(double);
}

int unit_blocks_per_sm(size_t smem) {
    int nb = 0;
    cudaFuncSetAttribute(unit_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, unit_sweep_kernel, kNT, smem);
    return nb > 0 ? nb : 1;
}

cudaError_t launch_units(const SweepUnit* units, const int* blk, int ctas, int total_ctas, size_t smem,
                         cudaStream_t st) {
    cudaError_t e =
        cudaFuncSetAttribute(unit_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    unit_sweep_kernel<<<total_ctas, kNT, smem, st>>>(units, blk, ctas);
    return cudaGetLastError();
}

int selftest_bounded_wait(int* status, void* stream) {
    bounded_wait_probe_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(status);
    return cudaGetLastError() == cudaSuccess ? NQS_OK : NQS_ERR_CUDA;
}

}  // namespace nqs
