// Whole expansions of circuits narrower than a sweep tile (small.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "nqs_internal.h"

namespace nqs {

constexpr int kSmallMaxQ = 11;
constexpr int kSmallDepth = NQS_MAX_LEVEL;      // insertions of a unit

// One operation (16 bytes); its matrix (16 float2) lies at the same index of
// the matrix table.
struct SmallOp {
    unsigned char type, a, b, diag;   // a, b: qubits; diag: a site's K_0 is diagonal
    int site;
    int pad[2];
};

// A state with fixed insertions: chi of the first site, K_f there, swept to the
// end with K_f at the other sites named and K_0 elsewhere, reduced against phi
// at every site after the last.
struct SmallUnit {
    long long rank;                   // index in the rank table of the term of the first site after the last
    int depth;
    int site[kSmallDepth];
    unsigned char factor[kSmallDepth];   // kept-factor positions
    int pad;
};

struct SmallArgs {
    int n, n_sites, n_units;
    int fwd_ops, bwd_ops;             // operations up to the last site; from the end back to the first
    int all_ops;                      // the whole circuit (U |psi>)
    const SmallOp* fwd;               // circuit order; K_0 and the kept factors at sites
    const float2* fwd_mats;
    const SmallOp* bwd;               // reversed, adjoint
    const float2* bwd_mats;
    const int* site_op;               // index of each site in fwd
    const int* n_factors;             // kept factors per site
    const double* kmats;              // complex128 factors, 32 doubles per site
    const int* keep;                  // factor index of each kept position, 3 per site
    float2* phi;                      // checkpoints, one state per site
    float2* chi;
    const SmallUnit* units;
    const long long* ranks;           // rank of the first factor's term of each (unit, site), -1 none
    const long long* pair_rank;       // the same for the sites on their own (level 1); -1 none
    long long level0;                 // rank of the level-0 term, -1 none
    double* term_vals;
    int psi_kind, v_kind;
    unsigned long long psi_bits, v_bits;
    const float2* psi_dev;
    const float2* v_dev;
};

cudaError_t launch_small(const SmallArgs& a, cudaStream_t st);

}  // namespace nqs
