// General-noise path: circuits with two-qubit noise channels or noises given
// by their matrix representation (Sec. IV's SVD in its general form, with
// d^2 factors per site and two factor sets when the tensor-permuted matrix
// is not positive semidefinite).
//
// Every kept assignment sigma is X = a_sigma * conj(b_sigma) with
// a = <v|C[KA_sigma]|psi>, b = <v|C[KB_sigma]|psi> (host_generic.cpp); b = a
// when every site has KA = KB.  Each network is evaluated for all kept
// assignments at once from checkpoints, on the device, one kernel per
// operation (complex64 states, FP64 reductions):
//   backward: phi_t = (events after site t with KX_0 at later sites)^dagger v,
//   forward:  depth-first from psi -- at site t the reduced matrix
//             R[a][b] = sum_rest conj(phi_t[rest, a]) w[rest, b] over the
//             site's qubits gives <phi_t| K_j |w> = sum_ab K_j[a][b] R[a][b]
//             for every factor j, and each non-dominant K_j w is swept on to
//             the later sites while the level allows.
// The amplitudes land at the canonical ranks of the kept-term list (level,
// site tuple, factor tuple, all lexicographic); a last kernel forms
// X = a conj(b), the per-level Neumaier sums of Re X and |sum Im X|.  This
// path has no gate fusion, tiling or pass specialisation; circuits of at most 14
// qubits go through generic_small.cu instead (whole states on chip), wider ones
// sweep all siblings of a prefix with one launch per gate and never wait for
// the host.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <vector>

#include "generic_gates.cuh"
#include "generic_small.h"
#include "level_sum.cuh"
#include "nqs_internal.h"

namespace nqs {

struct GEngine {
    void* buf = nullptr;
    size_t buf_bytes = 0;
    void* aux = nullptr;
    size_t aux_bytes = 0;
    bool one_sibling = false;      // the buffers hold one sibling per depth: more did not fit
    long long n_terms = 0;
    bool has_result = false;
    cudaStream_t last = nullptr;
    cudaEvent_t done = nullptr;    // end of the last call: a call on another stream waits for it
    double* vals = nullptr;
    // narrow circuits: what is prepared for one level (generic_small.cu)
    int small_level = -1;
    int sms = 0;
    double bound = 0;
    GSmallArgs side[2] = {};
    bool two_sided = false;
    long long* loff = nullptr;
    nqs_result* res = nullptr;
};

namespace {

constexpr int kT = 256;
// Siblings (the states of one prefix's last insertion) swept together by one
// launch per gate: up to this much of them.
constexpr size_t kSiblingBytes = (size_t)4 << 30;

struct GMat {
    float2 m[16];
};

// one gate on blockIdx.y states (dim apart)
__global__ void __launch_bounds__(kT) g_apply_kernel(float2* __restrict__ s, long long count, long long dim, int nq, int q0,
                                                     int q1, GMat g) {
    s += blockIdx.y * dim;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < count; p += stride) {
        if (nq == 1) {
            const long long bit = 1ll << q0;
            const long long lo = p & (bit - 1);
            const long long i0 = ((p - lo) << 1) | lo, i1 = i0 | bit;
            float2 a = s[i0], b = s[i1];
            gate2(g.m[0], g.m[1], g.m[2], g.m[3], a, b);
            s[i0] = a;
            s[i1] = b;
        } else {
            long long idx[4];
            quad_index(p, q0, q1, idx);
            float2 v[4] = {s[idx[0]], s[idx[1]], s[idx[2]], s[idx[3]]};
            gate4(g.m, v);
            for (int k = 0; k < 4; ++k) s[idx[k]] = v[k];
        }
    }
}

// K_1 .. K_{m-1} of a site on one state: states j - 1 of `out` (the children of a prefix)
__global__ void __launch_bounds__(kT) g_spawn_kernel(const float2* __restrict__ s, float2* __restrict__ out,
                                                     long long count, long long dim, int nq, int q0, int q1,
                                                     const float2* __restrict__ K) {
    out += blockIdx.y * dim;
    K += (size_t)(blockIdx.y + 1) * 16;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < count; p += stride) {
        if (nq == 1) {
            const long long bit = 1ll << q0;
            const long long lo = p & (bit - 1);
            const long long i0 = ((p - lo) << 1) | lo, i1 = i0 | bit;
            float2 a = s[i0], b = s[i1];
            gate2(K[0], K[1], K[2], K[3], a, b);
            out[i0] = a;
            out[i1] = b;
        } else {
            long long idx[4];
            quad_index(p, q0, q1, idx);
            float2 v[4] = {s[idx[0]], s[idx[1]], s[idx[2]], s[idx[3]]};
            gate4(K, v);
            for (int k = 0; k < 4; ++k) out[idx[k]] = v[k];
        }
    }
}

// per-block FP64 partials of R[a][b] (d^2 complex, d = 2 or 4) of phi against
// blockIdx.y states, in a fixed order
template <int NQ>
__global__ void __launch_bounds__(kT) g_reduce_kernel(const float2* __restrict__ phi, const float2* __restrict__ w,
                                                      long long count, long long dim, int q0, int q1,
                                                      double* __restrict__ part) {
    constexpr int D = 1 << NQ;
    w += blockIdx.y * dim;
    double acc[32];
#pragma unroll
    for (int e = 0; e < 32; ++e) acc[e] = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < count; p += stride) {
        long long idx[4];
        if (NQ == 1) {
            const long long bit = 1ll << q0;
            const long long lo = p & (bit - 1);
            idx[0] = ((p - lo) << 1) | lo;
            idx[1] = idx[0] | bit;
        } else {
            quad_index(p, q0, q1, idx);
        }
        float2 f[D], x[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            f[k] = phi[idx[k]];
            x[k] = w[idx[k]];
        }
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = 0; b < D; ++b) {
                acc[2 * (D * a + b)] += (double)f[a].x * x[b].x + (double)f[a].y * x[b].y;
                acc[2 * (D * a + b) + 1] += (double)f[a].x * x[b].y - (double)f[a].y * x[b].x;
            }
    }
    __shared__ double sm[kT / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    sm[warp][lane] = warp_scatter32(acc, lane);
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < kT / 32; ++k) v += sm[k][threadIdx.x];
        part[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 32 + threadIdx.x] = v;
    }
}

// R of state blockIdx.x from the partials (fixed order), then the amplitudes
// sum_ab K_j[a][b] R[a][b] of its factors: j = 1 .. m - 1 at rank + state *
// (m - 1) + j - 1 (consecutive: the last factor runs fastest in the canonical
// order), j = 0 at rank0; negative ranks: none
__global__ void __launch_bounds__(kT) g_finish_kernel(const double* __restrict__ part, int grid, int dd,
                                                      const double2* __restrict__ K, int m, long long rank,
                                                      long long rank0, double2* __restrict__ amps) {
    __shared__ double sm[kT / 32][32], R[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v = 0.0;
    for (int g = warp; g < grid; g += kT / 32) v += part[((size_t)blockIdx.x * grid + g) * 32 + lane];
    sm[warp][lane] = v;
    __syncthreads();
    if (warp == 0) {
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < kT / 32; ++k) t += sm[k][lane];
        R[lane] = t;
        __syncwarp();
        const long long at = lane == 0 ? rank0 : rank >= 0 ? rank + (long long)blockIdx.x * (m - 1) + lane - 1 : -1;
        if (lane < m && at >= 0) {
            const double2* const k = K + (size_t)lane * dd;
            double re = 0.0, im = 0.0;
            for (int e = 0; e < dd; ++e) {
                re += k[e].x * R[2 * e] - k[e].y * R[2 * e + 1];
                im += k[e].x * R[2 * e + 1] + k[e].y * R[2 * e];
            }
            amps[at] = make_double2(re, im);
        }
    }
}

__global__ void g_fill_kernel(float2* __restrict__ s, long long dim, unsigned long long bits) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < dim; i += stride)
        s[i] = make_float2((unsigned long long)i == bits ? 1.f : 0.f, 0.f);
}

// X = a conj(b) (b = a when b is null); per-level Neumaier sums of Re X in
// canonical order, |sum Im X|, the result record
__global__ void __launch_bounds__(kT) g_sum_kernel(const double2* __restrict__ a, const double2* __restrict__ b,
                                                   const long long* __restrict__ level_off, int level,
                                                   long long n_terms, double bound, double* __restrict__ vals,
                                                   nqs_result* __restrict__ res) {
    static_assert(kT == kSumThreads, "block size of level_sums");
    __shared__ double T[NQS_MAX_LEVEL + 1], im_part[kT / 32];
    double im_sum = 0.0;
    level_sums(level_off, level, [&](long long i) {
        const double2 x = a[i];
        const double2 y = b ? b[i] : x;
        const double re = x.x * y.x + x.y * y.y;
        vals[i] = re;
        im_sum += x.y * y.x - x.x * y.y;
        return re;
    }, T);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) im_sum += __shfl_xor_sync(0xffffffffu, im_sum, o);
    if ((threadIdx.x & 31) == 0) im_part[threadIdx.x >> 5] = im_sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double imag_tot = 0.0;
        for (int w = 0; w < kT / 32; ++w) imag_tot += im_part[w];
        store_levels(res, T, level);
        res->imag_residual = fabs(imag_tot);
        res->n_terms = (uint64_t)n_terms;
        res->bound = bound;
        res->level = level;
        res->status = NQS_OK;
    }
}

int cu(cudaError_t e) { return e == cudaSuccess ? NQS_OK : NQS_ERR_CUDA; }

// end of a call: results are there once `st` gets here
int finish_call(GEngine& G, cudaStream_t st, int rc) {
    if (!rc && !G.done) rc = cu(cudaEventCreateWithFlags(&G.done, cudaEventDisableTiming));
    if (!rc) rc = cu(cudaEventRecord(G.done, st));
    G.last = st;
    G.has_result = rc == NQS_OK;
    return rc;
}

struct Run {
    Handle& h;
    cudaStream_t st;
    int n, level, grid;
    long long dim;
    const TermIndex& ti;
    std::vector<float2*> phi;      // per site
    std::vector<float2*> work;     // per depth: `width` states (depth 0: one)
    int width;                     // siblings swept together
    double* part;                  // reduce partials (width x grid x 32)
    const float2* fdev;            // factors of this side in complex64: site s, factor j at (s * 16 + j) * 16
    double2* kdev;                 // factor tables of this side: site s at kofs[s]
    std::vector<size_t> kofs;
    double2* amps;                 // this side's amplitudes
    std::vector<int> site_ev;      // event index of each site
    std::vector<int> ev_gate;      // event -> gate index or -1
    std::vector<int> ev_site;      // event -> site index or -1
    int last_site_ev = -1;
    bool side_b;
    int rc = NQS_OK;

    GMat gate_mat(int g, bool adjoint) {
        const Gate& gt = h.circ.gates[g];
        GMat m{};
        if (gate_is_two_qubit(gt.kind)) {
            Mat4 a = gate_matrix_2q(gt);
            for (int r = 0; r < 4; ++r)
                for (int c = 0; c < 4; ++c) {
                    const cd v = adjoint ? std::conj(a[4 * c + r]) : a[4 * r + c];
                    m.m[4 * r + c] = make_float2((float)v.real(), (float)v.imag());
                }
        } else {
            Mat2 a = gate_matrix_1q(gt);
            for (int r = 0; r < 2; ++r)
                for (int c = 0; c < 2; ++c) {
                    const cd v = adjoint ? std::conj(a[2 * c + r]) : a[2 * r + c];
                    m.m[2 * r + c] = make_float2((float)v.real(), (float)v.imag());
                }
        }
        return m;
    }
    GMat factor_mat(int s, int j, bool adjoint) {
        const GFactors& f = h.gfac[s];
        const int d = f.nq == 1 ? 2 : 4;
        const std::vector<cd>& K = side_b ? f.KB : f.KA;
        GMat m{};
        for (int r = 0; r < d; ++r)
            for (int c = 0; c < d; ++c) {
                const cd v = adjoint ? std::conj(K[(size_t)j * d * d + d * c + r]) : K[(size_t)j * d * d + d * r + c];
                m.m[d * r + c] = make_float2((float)v.real(), (float)v.imag());
            }
        return m;
    }
    void apply(float2* s, int states, int nq, int q0, int q1, const GMat& m) {
        if (rc) return;
        g_apply_kernel<<<dim3(grid, states), kT, 0, st>>>(s, dim >> nq, dim, nq, q0, q1, m);
        rc = cu(cudaGetLastError());
    }
    void apply_event(float2* s, int states, int e, bool adjoint) {
        if (ev_gate[e] >= 0) {
            const Gate& g = h.circ.gates[ev_gate[e]];
            const bool two = gate_is_two_qubit(g.kind);
            apply(s, states, two ? 2 : 1, g.q0, g.q1, gate_mat(ev_gate[e], adjoint));
        } else {
            const GFactors& f = h.gfac[ev_site[e]];
            apply(s, states, f.nq, f.q0, f.q1, factor_mat(ev_site[e], 0, adjoint));
        }
    }
    // reduce (phi_t, w) of `states` siblings; the terms of the first one's
    // factors start at `rank`, the level-0 term lies at rank0
    void reduce_finish(int t, const float2* w, int states, long long rank, long long rank0) {
        if (rc || (rank < 0 && rank0 < 0)) return;
        const GFactors& f = h.gfac[t];
        const dim3 g(grid, states);
        if (f.nq == 1) g_reduce_kernel<1><<<g, kT, 0, st>>>(phi[t], w, dim >> 1, dim, f.q0, f.q1, part);
        else g_reduce_kernel<2><<<g, kT, 0, st>>>(phi[t], w, dim >> 2, dim, f.q0, f.q1, part);
        g_finish_kernel<<<states, kT, 0, st>>>(part, grid, f.nq == 1 ? 4 : 16, kdev + kofs[t], f.m, rank, rank0, amps);
        rc = cu(cudaGetLastError());
    }

    // `states` siblings (factor positions fp[depth - 1], + 1, ... of the last
    // insertion) from event e0 to the last site; every launch serves all of them
    void expand(float2* w, int states, int e0, int depth, std::vector<int>& c, std::vector<int>& fp) {
        for (int e = e0; e <= last_site_ev && !rc; ++e) {
            if (ev_gate[e] >= 0) {
                apply_event(w, states, e, false);
                continue;
            }
            const int t = ev_site[e];
            const GFactors& f = h.gfac[t];
            const bool last0 = depth == 0 && e == last_site_ev;
            if (depth < level || last0) {
                long long rank = -1;
                c[depth] = t;
                if (depth < level && f.m > 1) {
                    fp[depth] = 0;
                    rank = (long long)ti.rank(depth + 1, c.data(), fp.data());
                }
                reduce_finish(t, w, states, rank, last0 ? 0 : -1);
                if (depth + 1 < level) {
                    const int first = depth > 0 ? fp[depth - 1] : 0;
                    for (int s = 0; s < states && !rc; ++s) {
                        if (depth > 0) fp[depth - 1] = first + s;
                        for (int j = 1; j < f.m && !rc; j += width) {
                            const int k = std::min(width, f.m - j);
                            c[depth] = t;
                            fp[depth] = j - 1;
                            float2* const w2 = work[depth + 1];
                            g_spawn_kernel<<<dim3(grid, k), kT, 0, st>>>(w + s * dim, w2, dim >> f.nq, dim, f.nq, f.q0,
                                                                         f.q1, fdev + (size_t)(t * 16 + j - 1) * 16);
                            rc = cu(cudaGetLastError());
                            expand(w2, k, e + 1, depth + 1, c, fp);
                        }
                    }
                    if (depth > 0) fp[depth - 1] = first;
                }
            }
            apply_event(w, states, e, false);
        }
    }

    // the whole network for one factor set: backward checkpoints, forward expansion
    void network(const float2* psi0, const float2* v0) {
        const int n_ev = (int)ev_gate.size();
        float2* p = work[0];
        rc = cu(cudaMemcpyAsync(p, v0, dim * sizeof(float2), cudaMemcpyDeviceToDevice, st));
        for (int e = n_ev - 1; e >= 0 && !rc; --e) {
            if (ev_gate[e] >= 0) {
                apply_event(p, 1, e, true);
            } else {
                rc = cu(cudaMemcpyAsync(phi[ev_site[e]], p, dim * sizeof(float2), cudaMemcpyDeviceToDevice, st));
                apply_event(p, 1, e, true);
            }
        }
        if (rc) return;
        rc = cu(cudaMemcpyAsync(work[0], psi0, dim * sizeof(float2), cudaMemcpyDeviceToDevice, st));
        std::vector<int> c(level + 1), fp(level + 1);
        expand(work[0], 1, 0, 0, c, fp);
    }
};

void release(GEngine& G, void* stream) {
    if (G.buf) dev_free(G.buf, G.buf_bytes, stream);
    if (G.aux) dev_free(G.aux, G.aux_bytes, stream);
    G.buf = G.aux = nullptr;
    G.buf_bytes = G.aux_bytes = 0;
    G.one_sibling = false;
    G.small_level = -1;
    G.has_result = false;   // the term values went with it
}

double dropped_bound(const std::vector<GFactors>& fac, int level) {
    std::vector<double> poly(1, 1.0);
    for (const auto& f : fac) {
        std::vector<double> nx(poly.size() + 1, 0.0);
        for (size_t i = 0; i < poly.size(); ++i) {
            nx[i] += poly[i] * f.norm_dom;
            nx[i + 1] += poly[i] * f.norm_rest;
        }
        poly.swap(nx);
    }
    double bound = 0.0;
    for (size_t i = level + 1; i < poly.size(); ++i) bound += poly[i];
    return bound;
}

// a d x d matrix (or its adjoint) rounded to complex64
void put_matrix(const cd* k, int d, bool adjoint, float2* out) {
    for (int r = 0; r < d; ++r)
        for (int c = 0; c < d; ++c) {
            const cd v = adjoint ? std::conj(k[d * c + r]) : k[d * r + c];
            out[d * r + c] = make_float2((float)v.real(), (float)v.imag());
        }
}

// States of the prefixes held for the reductions of a narrow circuit, and the
// terms up to which it goes that way.
constexpr size_t kSmallStates = (size_t)1 << 30;
constexpr uint64_t kSmallTerms = 1ull << 22;

// Prepare the launches of a narrow circuit (generic_small.cu) for one level;
// NQS_ERR_UNSUPPORTED when it does not fit.
int prepare_small(Handle& h, GEngine& G, int level, const TermIndex& ti, void* stream) {
    if (G.small_level == level) return NQS_OK;
    const int n = h.circ.n, N = (int)h.gfac.size();
    if (n > kGSmallMaxQ || N > 4096 || ti.total > kSmallTerms) return NQS_ERR_UNSUPPORTED;
    // events in circuit order
    std::vector<GOp> fwd;
    std::vector<int> gate_of, site_op(N);
    {
        size_t ns = 0;
        auto sites_after = [&](int g) {
            for (; ns < h.circ.noises.size() && h.circ.noises[ns].after_gate == g; ++ns) {
                const GFactors& f = h.gfac[ns];
                GOp o{};
                o.type = GO_SITE;
                o.a = (unsigned char)f.q0;
                o.b = (unsigned char)std::max(f.q1, 0);
                o.nq = (unsigned char)f.nq;
                o.site = (int)ns;
                site_op[ns] = (int)fwd.size();
                fwd.push_back(o);
                gate_of.push_back(-1);
            }
        };
        sites_after(-1);
        for (size_t g = 0; g < h.circ.gates.size(); ++g) {
            const Gate& gt = h.circ.gates[g];
            GOp o{};
            o.type = gt.kind == G_CZ ? GO_CZ : gt.kind == G_CX ? GO_CX : GO_ONE;
            o.a = (unsigned char)gt.q0;
            o.b = (unsigned char)std::max(gt.q1, 0);
            o.site = -1;
            fwd.push_back(o);
            gate_of.push_back((int)g);
            sites_after((int)g);
        }
    }
    const int n_ops = (int)fwd.size();
    const size_t padded = ((size_t)n_ops + 31) / 32 * 32 + 32;
    // prefixes of up to level - 1 insertions, and all reductions
    std::vector<GUnit> units;
    std::vector<GPair> pairs;
    int slots = 0;
    const size_t state_bytes = sizeof(float2) << n;
    int sites[NQS_MAX_LEVEL + 1], fp[NQS_MAX_LEVEL + 1];
    auto first_rank = [&](int k) {
        if (h.gfac[sites[k - 1]].m < 2) return -1ll;
        fp[k - 1] = 0;
        return (long long)ti.rank(k, sites, fp);
    };
    for (int s = 0; s < N; ++s) {
        GPair pr{s, -1, -1, s == N - 1 ? 0 : -1};
        sites[0] = s;
        if (level >= 1) pr.rank = first_rank(1);
        if (pr.rank >= 0 || pr.rank0 >= 0) pairs.push_back(pr);
    }
    bool fits = true;
    std::function<void(int, int)> extend = [&](int depth, int from) {
        for (int s = from; s + 1 < N && fits; ++s) {
            sites[depth] = s;
            for (int j = 1; j < h.gfac[s].m && fits; ++j) {
                fp[depth] = j - 1;
                GUnit u{};
                u.depth = depth + 1;
                u.out = slots;
                for (int k = 0; k <= depth; ++k) {
                    u.site[k] = (unsigned short)sites[k];
                    u.factor[k] = (unsigned char)(fp[k] + 1);
                }
                for (int t = s + 1; t < N; ++t) {
                    sites[depth + 1] = t;
                    pairs.push_back(GPair{t, slots++, first_rank(depth + 2), -1});
                }
                units.push_back(u);
                fits = (size_t)slots * state_bytes <= kSmallStates;
                if (fits && depth + 2 < level) {
                    extend(depth + 1, s + 1);
                    sites[depth] = s;
                    fp[depth] = j - 1;
                }
            }
        }
    };
    if (level >= 2) extend(0, 0);
    if (!fits) return NQS_ERR_UNSUPPORTED;
    release(G, stream);
    if (!G.sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&G.sms, cudaDevAttrMultiProcessorCount, dev);
    }
    const int parts = generic_small_parts(n, (int)pairs.size(), G.sms);
    bool two = false;
    for (const auto& f : h.gfac) two = two || !f.same;
    // tables: the lists, then per side the matrices and factors
    std::vector<char> blob;
    auto put = [&](const void* src, size_t bytes) {
        const size_t at = (blob.size() + 255) & ~(size_t)255;
        blob.resize(at + bytes + 1);
        if (bytes) std::memcpy(blob.data() + at, src, bytes);
        return at;
    };
    std::vector<GOp> fo(padded), bo(padded);
    std::copy(fwd.begin(), fwd.end(), fo.begin());
    std::reverse_copy(fwd.begin(), fwd.end(), bo.begin());
    const size_t o_fo = put(fo.data(), padded * sizeof(GOp)), o_bo = put(bo.data(), padded * sizeof(GOp));
    std::vector<int> kofs(N), nf(N);
    size_t kc = 0;
    for (int s = 0; s < N; ++s) {
        kofs[s] = (int)kc;
        nf[s] = h.gfac[s].m;
        kc += h.gfac[s].KA.size();
    }
    const size_t o_so = put(site_op.data(), N * sizeof(int)), o_ko = put(kofs.data(), N * sizeof(int));
    const size_t o_nf = put(nf.data(), N * sizeof(int));
    const size_t o_un = put(units.data(), units.size() * sizeof(GUnit));
    const size_t o_pr = put(pairs.data(), pairs.size() * sizeof(GPair));
    std::vector<long long> lo(level + 2);
    for (int u = 0; u <= level + 1; ++u) lo[u] = (long long)ti.level_offset[u];
    const size_t o_lo = put(lo.data(), lo.size() * sizeof(long long));
    size_t o_fm[2], o_bm[2], o_fac[2], o_km[2];
    for (int b = 0; b < (two ? 2 : 1); ++b) {
        std::vector<float2> fm(padded * 16, make_float2(0.f, 0.f)), bm(fm), fac((size_t)N * 256, make_float2(0.f, 0.f));
        std::vector<double2> km(kc);
        for (int i = 0; i < n_ops; ++i) {
            float2* const f = fm.data() + (size_t)i * 16;
            float2* const g = bm.data() + (size_t)(n_ops - 1 - i) * 16;
            if (fwd[i].type == GO_SITE) {
                const GFactors& gf = h.gfac[fwd[i].site];
                const std::vector<cd>& K = b ? gf.KB : gf.KA;
                const int d = gf.nq == 1 ? 2 : 4;
                put_matrix(K.data(), d, false, f);
                put_matrix(K.data(), d, true, g);
                for (int j = 0; j < gf.m; ++j)
                    put_matrix(K.data() + (size_t)j * d * d, d, false, fac.data() + (size_t)(fwd[i].site * 16 + j) * 16);
                for (size_t e = 0; e < K.size(); ++e) km[kofs[fwd[i].site] + e] = make_double2(K[e].real(), K[e].imag());
            } else if (fwd[i].type == GO_ONE) {
                const Mat2 a = gate_matrix_1q(h.circ.gates[gate_of[i]]);
                put_matrix(a.data(), 2, false, f);
                put_matrix(a.data(), 2, true, g);
            }
        }
        o_fm[b] = put(fm.data(), fm.size() * sizeof(float2));
        o_bm[b] = put(bm.data(), bm.size() * sizeof(float2));
        o_fac[b] = put(fac.data(), fac.size() * sizeof(float2));
        o_km[b] = put(km.data(), km.size() * sizeof(double2));
    }
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t o_part = al(blob.size());
    const size_t o_amps = al(o_part + pairs.size() * parts * 32 * sizeof(double));
    const size_t o_vals = al(o_amps + (two ? 2 : 1) * (size_t)ti.total * sizeof(double2));
    const size_t o_res = al(o_vals + (size_t)ti.total * sizeof(double));
    G.buf_bytes = (2 * (size_t)N + slots) * state_bytes;
    G.aux_bytes = al(o_res + sizeof(nqs_result));
    G.buf = dev_alloc(G.buf_bytes, stream);
    G.aux = dev_alloc(G.aux_bytes, stream);
    if (!G.buf || !G.aux) {
        release(G, stream);
        return NQS_ERR_NOMEM;
    }
    cudaStream_t st = (cudaStream_t)stream;
    char* const ab = (char*)G.aux;
    int rc = cu(cudaMemcpyAsync(ab, blob.data(), blob.size(), cudaMemcpyHostToDevice, st));
    if (!rc) rc = cu(cudaMemsetAsync(ab + o_amps, 0, o_vals - o_amps, st));
    if (!rc) rc = cu(cudaStreamSynchronize(st));   // pageable source
    if (rc) {
        release(G, stream);
        return rc;
    }
    for (int b = 0; b < (two ? 2 : 1); ++b) {
        GSmallArgs& a = G.side[b];
        a = GSmallArgs{};
        a.n = n;
        a.n_units = (int)units.size();
        a.n_pairs = (int)pairs.size();
        a.parts = parts;
        a.fwd_ops = site_op[N - 1] + 1;
        a.bwd_ops = n_ops - site_op[0];
        a.all_ops = n_ops;
        a.fwd = (const GOp*)(ab + o_fo);
        a.fwd_mats = (const float2*)(ab + o_fm[b]);
        a.bwd = (const GOp*)(ab + o_bo);
        a.bwd_mats = (const float2*)(ab + o_bm[b]);
        a.site_op = (const int*)(ab + o_so);
        a.factors = (const float2*)(ab + o_fac[b]);
        a.kmats = (const double2*)(ab + o_km[b]);
        a.kofs = (const int*)(ab + o_ko);
        a.n_factors = (const int*)(ab + o_nf);
        a.phi = (float2*)G.buf;
        a.chi = a.phi + ((size_t)N << n);
        a.out = a.chi + ((size_t)N << n);
        a.units = (const GUnit*)(ab + o_un);
        a.pairs = (const GPair*)(ab + o_pr);
        a.part = (double*)(ab + o_part);
        a.amps = (double2*)(ab + o_amps) + (size_t)b * ti.total;
    }
    G.two_sided = two;
    G.loff = (long long*)(ab + o_lo);
    G.vals = (double*)(ab + o_vals);
    G.res = (nqs_result*)(ab + o_res);
    G.n_terms = (long long)ti.total;
    G.bound = dropped_bound(h.gfac, level);
    G.small_level = level;
    return NQS_OK;
}

int run_small(GEngine& G, const nqs_state* psi, const nqs_state* v, nqs_result* out, cudaStream_t st) {
    int rc = NQS_OK;
    for (int b = 0; b < (G.two_sided ? 2 : 1) && !rc; ++b) {
        GSmallArgs a = G.side[b];
        a.psi_kind = psi->kind;
        a.v_kind = v->kind;
        a.psi_bits = psi->bits;
        a.v_bits = v->bits;
        a.psi_dev = (const float2*)psi->dev;
        a.v_dev = (const float2*)v->dev;
        rc = cu(launch_generic_small(a, st));
    }
    if (rc) return rc;
    g_sum_kernel<<<1, kT, 0, st>>>(G.side[0].amps, G.two_sided ? G.side[1].amps : nullptr, G.loff, G.small_level,
                                   G.n_terms, G.bound, G.vals, G.res);
    rc = cu(cudaGetLastError());
    if (!rc) rc = cu(cudaMemcpyAsync(out, G.res, sizeof(nqs_result), cudaMemcpyDefault, st));
    return finish_call(G, st, rc);
}

}  // namespace

int general_fidelity(Handle& h, const nqs_state* psi, const nqs_state* v, int level, nqs_result* out, void* stream) {
    if (!h.geng) h.geng = new GEngine();
    GEngine& G = *h.geng;
    cudaStream_t st = (cudaStream_t)stream;
    const int n = h.circ.n, N = (int)h.gfac.size();
    const long long dim = 1ll << n;
    level = std::min(level, N);
    if (N == 0) return NQS_ERR_UNSUPPORTED;   // the general path needs at least one noise
    // the handle's buffers serve one call at a time
    if (G.done && G.last != st && cudaStreamWaitEvent(st, G.done, 0) != cudaSuccess) return NQS_ERR_CUDA;
    if (G.small_level == level) return run_small(G, psi, v, out, st);
    std::vector<int> m(N);
    bool two_sided = false;
    for (int s = 0; s < N; ++s) {
        m[s] = h.gfac[s].m - 1;
        two_sided = two_sided || !h.gfac[s].same;
    }
    TermIndex ti;
    ti.build(m, level);
    {
        const int rc = prepare_small(h, G, level, ti, stream);
        if (rc == NQS_OK) return run_small(G, psi, v, out, st);
        if (rc != NQS_ERR_UNSUPPORTED && rc != NQS_ERR_NOMEM) return rc;
    }
    // events in circuit order
    std::vector<int> ev_gate, ev_site, site_ev(N, -1);
    {
        size_t ns = 0;
        auto sites_after = [&](int g) {
            while (ns < h.circ.noises.size() && h.circ.noises[ns].after_gate == g) {
                site_ev[ns] = (int)ev_gate.size();
                ev_gate.push_back(-1);
                ev_site.push_back((int)ns);
                ++ns;
            }
        };
        sites_after(-1);
        for (size_t g = 0; g < h.circ.gates.size(); ++g) {
            ev_gate.push_back((int)g);
            ev_site.push_back(-1);
            sites_after((int)g);
        }
    }
    int last_site_ev = -1;
    for (int s = 0; s < N; ++s) last_site_ev = std::max(last_site_ev, site_ev[s]);
    // device memory: N phi, one state at depth 0 and `width` siblings at every
    // deeper one, psi, v; aux: factors, partials, amps, values, tables
    const size_t sb = (size_t)dim * sizeof(float2);
    const int depths = std::max(0, level - 1);
    const size_t kcount = [&] {
        size_t c = 0;
        for (const auto& f : h.gfac) c += (size_t)f.m * (f.nq == 1 ? 4 : 16);
        return c;
    }();
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = (int)std::max<long long>(1, std::min<long long>((long long)sms * 4, (dim / 2 + kT - 1) / kT));
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    int width = (int)std::max<size_t>(1, std::min<size_t>(15, kSiblingBytes / sb));
    size_t n_states, o_part, o_amps, o_vals, o_loff, o_res, o_fac, aux_bytes;
    const size_t o_k = 0;
    auto lay_out = [&] {
        n_states = (size_t)N + 1 + (size_t)depths * width + 2;
        o_part = al(o_k + 2 * kcount * sizeof(double2));
        o_amps = al(o_part + (size_t)width * grid * 32 * sizeof(double));
        o_vals = al(o_amps + (two_sided ? 2 : 1) * (size_t)ti.total * sizeof(double2));
        o_loff = al(o_vals + (size_t)ti.total * sizeof(double));
        o_res = al(o_loff + (size_t)(level + 2) * sizeof(long long));
        o_fac = al(o_res + sizeof(nqs_result));
        aux_bytes = al(o_fac + 2 * (size_t)N * 256 * sizeof(float2));
    };
    auto held = [&] { return G.buf_bytes >= n_states * sb && G.aux_bytes >= aux_bytes; };
    lay_out();
    G.small_level = -1;   // its tables are written over
    if (G.one_sibling && !held()) {
        const int all = width;
        width = 1;
        lay_out();
        if (!held()) width = all;
        lay_out();
    }
    if (!held()) {
        release(G, stream);
        // all siblings together where they fit, else one after another
        for (;; width = 1, lay_out()) {
            G.buf_bytes = n_states * sb;
            G.aux_bytes = aux_bytes;
            G.buf = dev_alloc(G.buf_bytes, stream);
            G.aux = dev_alloc(G.aux_bytes, stream);
            if (G.buf && G.aux) break;
            const bool last = width == 1;
            release(G, stream);
            if (last) return NQS_ERR_NOMEM;
            G.one_sibling = true;
        }
    }
    char* ab = (char*)G.aux;
    double2* kdevA = (double2*)(ab + o_k);
    double2* kdevB = kdevA + kcount;
    double* part = (double*)(ab + o_part);
    double2* ampsA = (double2*)(ab + o_amps);
    double2* ampsB = two_sided ? ampsA + ti.total : nullptr;
    double* vals = (double*)(ab + o_vals);
    long long* loff = (long long*)(ab + o_loff);
    nqs_result* res = (nqs_result*)(ab + o_res);
    float2* fac_dev = (float2*)(ab + o_fac);
    float2* base = (float2*)G.buf;
    float2* psi_buf = base + (size_t)(N + 1 + (size_t)depths * width) * dim;
    float2* v_buf = psi_buf + dim;
    // factor tables (complex128) of both sides
    std::vector<double2> kh(2 * kcount);
    std::vector<size_t> kofs(N);
    {
        size_t at = 0;
        for (int s = 0; s < N; ++s) {
            const GFactors& f = h.gfac[s];
            kofs[s] = at;
            for (size_t e = 0; e < f.KA.size(); ++e) {
                kh[at + e] = make_double2(f.KA[e].real(), f.KA[e].imag());
                kh[kcount + at + e] = make_double2(f.KB[e].real(), f.KB[e].imag());
            }
            at += f.KA.size();
        }
    }
    // the same in complex64, for the spawns
    std::vector<float2> fh(2 * (size_t)N * 256, make_float2(0.f, 0.f));
    for (int s = 0; s < N; ++s) {
        const GFactors& f = h.gfac[s];
        const int d = f.nq == 1 ? 2 : 4;
        for (int j = 0; j < f.m; ++j) {
            put_matrix(f.KA.data() + (size_t)j * d * d, d, false, fh.data() + (size_t)(s * 16 + j) * 16);
            put_matrix(f.KB.data() + (size_t)j * d * d, d, false, fh.data() + (size_t)((N + s) * 16 + j) * 16);
        }
    }
    std::vector<long long> lo(level + 2);
    for (int u = 0; u <= level + 1; ++u) lo[u] = (long long)ti.level_offset[u];
    int rc = cu(cudaMemcpyAsync(fac_dev, fh.data(), fh.size() * sizeof(float2), cudaMemcpyHostToDevice, st));
    if (!rc) rc = cu(cudaMemcpyAsync(kdevA, kh.data(), kh.size() * sizeof(double2), cudaMemcpyHostToDevice, st));
    if (!rc) rc = cu(cudaMemcpyAsync(loff, lo.data(), lo.size() * sizeof(long long), cudaMemcpyHostToDevice, st));
    if (!rc) rc = cu(cudaStreamSynchronize(st));   // pageable sources
    if (!rc) rc = cu(cudaMemsetAsync(ampsA, 0, (two_sided ? 2 : 1) * (size_t)ti.total * sizeof(double2), st));
    // psi, v
    const int fill_grid = (int)std::max<long long>(1, std::min<long long>((long long)sms * 8, dim / kT));
    if (!rc) {
        if (psi->kind == NQS_STATE_BASIS) g_fill_kernel<<<fill_grid, kT, 0, st>>>(psi_buf, dim, psi->bits);
        else rc = cu(cudaMemcpyAsync(psi_buf, psi->dev, sb, cudaMemcpyDeviceToDevice, st));
        if (!rc) rc = cu(cudaGetLastError());
    }
    Run R{h, st, n, level, grid, dim, ti, {}, {}, width, part, fac_dev, kdevA, kofs, ampsA, site_ev, ev_gate, ev_site,
          last_site_ev, false};
    for (int s = 0; s < N; ++s) R.phi.push_back(base + (size_t)s * dim);
    R.work.push_back(base + (size_t)N * dim);
    for (int d = 0; d < depths; ++d) R.work.push_back(base + (size_t)(N + 1 + (size_t)d * width) * dim);
    R.rc = rc;
    if (!R.rc) {
        if (v->kind == NQS_STATE_BASIS) {
            g_fill_kernel<<<fill_grid, kT, 0, st>>>(v_buf, dim, v->bits);
            R.rc = cu(cudaGetLastError());
        } else if (v->kind == NQS_STATE_DENSE) {
            R.rc = cu(cudaMemcpyAsync(v_buf, v->dev, sb, cudaMemcpyDeviceToDevice, st));
        } else {   // U |psi>
            R.rc = cu(cudaMemcpyAsync(v_buf, psi_buf, sb, cudaMemcpyDeviceToDevice, st));
            for (size_t e = 0; e < ev_gate.size() && !R.rc; ++e)
                if (ev_gate[e] >= 0) R.apply_event(v_buf, 1, (int)e, false);
        }
    }
    if (!R.rc) R.network(psi_buf, v_buf);
    if (!R.rc && two_sided) {
        R.side_b = true;
        R.kdev = kdevB;
        R.fdev = fac_dev + (size_t)N * 256;
        R.amps = ampsB;
        R.network(psi_buf, v_buf);
    }
    rc = R.rc;
    if (!rc) {
        const double bound = dropped_bound(h.gfac, level);
        g_sum_kernel<<<1, kT, 0, st>>>(ampsA, ampsB, loff, level, (long long)ti.total, bound, vals, res);
        rc = cu(cudaGetLastError());
    }
    if (!rc) rc = cu(cudaMemcpyAsync(out, res, sizeof(nqs_result), cudaMemcpyDefault, st));
    G.n_terms = (long long)ti.total;
    G.vals = vals;
    return finish_call(G, st, rc);
}

int general_term_values(Handle& h, double* out, size_t cap, size_t* count) {
    if (!h.geng || !h.geng->has_result) return NQS_ERR_ORDER;
    GEngine& G = *h.geng;
    *count = (size_t)G.n_terms;
    const size_t nb = std::min<size_t>(cap, (size_t)G.n_terms) * sizeof(double);
    if (cudaStreamSynchronize(G.last) != cudaSuccess) return NQS_ERR_CUDA;
    if (nb && cudaMemcpy(out, G.vals, nb, cudaMemcpyDeviceToHost) != cudaSuccess) return NQS_ERR_CUDA;
    return NQS_OK;
}

void general_destroy(Handle& h) {
    if (!h.geng) return;
    if (h.geng->last) cudaStreamSynchronize(h.geng->last);
    release(*h.geng, h.geng->last);
    if (h.geng->done) cudaEventDestroy(h.geng->done);
    delete h.geng;
    h.geng = nullptr;
}

}  // namespace nqs
