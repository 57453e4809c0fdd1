// General-noise expansions of circuits whose state fits in one block's shared
// memory (generic_small.cu).
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "nqs_internal.h"

namespace nqs {

constexpr int kGSmallMaxQ = 14;   // 128 KiB of complex64

enum GOpType : int { GO_ONE = 0, GO_CZ = 1, GO_CX = 2, GO_SITE = 3 };

struct GOp {                      // 16 bytes; its matrix (16 float2) at the same index of the table
    unsigned char type, a, b, nq; // qubits of the gate or site
    int site;
    int pad[2];
};

struct GUnit {                    // a prefix of insertions
    int depth;
    unsigned short site[NQS_MAX_LEVEL];
    unsigned char factor[NQS_MAX_LEVEL];   // 1 .. m - 1
    int out;                      // slot of its state at the first site after the last
};

struct GPair {                    // one reduction: phi of a site against a state
    int site, slot;               // slot -1: chi of the site
    long long rank;               // of factor 1's term; -1: none
    long long rank0;              // of factor 0's term; -1: none
};

// One network (KA or KB) of a prepared expansion, device pointers
struct GSmallArgs {
    int n, n_units, n_pairs, parts;
    int fwd_ops, bwd_ops, all_ops;
    const GOp* fwd;
    const float2* fwd_mats;       // K_0 at sites
    const GOp* bwd;
    const float2* bwd_mats;
    const int* site_op;
    const float2* factors;        // factor j of site s at factors[(s * 16 + j) * 16]
    const double2* kmats;         // complex128 factors, site s at kofs[s]
    const int* kofs;
    const int* n_factors;
    float2 *phi, *chi, *out;
    const GUnit* units;
    const GPair* pairs;
    double* part;                 // [pair][part][32]
    double2* amps;
    int psi_kind, v_kind;
    unsigned long long psi_bits, v_bits;
    const float2* psi_dev;
    const float2* v_dev;
};

cudaError_t launch_generic_small(const GSmallArgs& a, cudaStream_t st);
int generic_small_parts(int n, int n_pairs, int sms);

}  // namespace nqs
