// Gate arithmetic of the general-noise path, shared by its kernels: every gate
// acts on its own, on complex64 amplitudes, with the same expressions wherever
// the state lies.
#pragma once

#include <cuda_runtime.h>

namespace nqs {

// a 2x2 matrix on the amplitude pair (a, b)
__device__ __forceinline__ void gate2(const float2 m0, const float2 m1, const float2 m2, const float2 m3, float2& a,
                                      float2& b) {
    const float2 x = a, y = b;
    a = make_float2(m0.x * x.x - m0.y * x.y + m1.x * y.x - m1.y * y.y, m0.x * x.y + m0.y * x.x + m1.x * y.y + m1.y * y.x);
    b = make_float2(m2.x * x.x - m2.y * x.y + m3.x * y.x - m3.y * y.y, m2.x * x.y + m2.y * x.x + m3.x * y.y + m3.y * y.x);
}

// a 4x4 matrix on four amplitudes
__device__ __forceinline__ void gate4(const float2* m, float2 (&v)[4]) {
    float2 in[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) in[k] = v[k];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float re = 0.f, im = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float2 w = m[4 * r + c];
            re += w.x * in[c].x - w.y * in[c].y;
            im += w.x * in[c].y + w.y * in[c].x;
        }
        v[r] = make_float2(re, im);
    }
}

// the four amplitudes of qubits (q0, q1), index 2 * b(q0) + b(q1), of group p
__device__ __forceinline__ void quad_index(long long p, int q0, int q1, long long (&idx)[4]) {
    const long long b0 = 1ll << q0, b1 = 1ll << q1;
    const long long lob = b0 < b1 ? b0 : b1, hib = b0 < b1 ? b1 : b0;
    long long x = p;
    long long lo = x & (lob - 1);
    x = ((x - lo) << 1) | lo;
    lo = x & (hib - 1);
    x = ((x - lo) << 1) | lo;
    idx[0] = x;
    idx[1] = x | b1;
    idx[2] = x | b0;
    idx[3] = x | b0 | b1;
}

// reduce-scatter of 32 doubles over a warp: lane l returns the warp's sum of
// component l (31 FP64 additions per lane; the chip has few FP64 units)
__device__ __forceinline__ double warp_scatter32(double (&v)[32], int lane) {
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const bool hi = lane & w;
#pragma unroll
        for (int e = 0; e < w; ++e) {
            const double send = hi ? v[e] : v[e + w];
            const double keep = hi ? v[e + w] : v[e];
            v[e] = keep + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
    return v[0];
}

}  // namespace nqs
