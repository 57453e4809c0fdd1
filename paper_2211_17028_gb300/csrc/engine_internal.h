// Schedule and engine state shared by the single-circuit engine (engine.cu)
// and the batch executor (batch.cu).  Internal to libnqs.
#pragma once

#include <cuda_runtime.h>

#include <memory>
#include <vector>

#include "fp32_round.h"
#include "jit.h"
#include "nqs_internal.h"
#include "small.h"
#include "sweep_types.h"
#include "unit_program.h"

namespace nqs {


struct RunPass {
    int op_off = 0, n_ops = 0;       // in the device op buffer
    int k = 0, c = 0;
    int local[kTileSlots] = {};
    int nonlocal[kMaxQ] = {};
    std::vector<int> lin;            // linear op index of each device op
    std::vector<int> ev_site;        // site of reduction event e
    std::vector<int> spawn_sites;    // sites that spawn in this pass, in execution order
};

struct Run {
    std::vector<RunPass> passes;     // in execution order
};

enum LaunchKind { L_PASS, L_FINISH, L_FILL, L_COPY, L_REDUCE2, L_SUM, L_NORMALIZE, L_SMALL };

struct Launch {
    LaunchKind kind;
    int S = 1;                       // states of a branch group (1: single-state sweeps)
    // pass, generated or tile kernel: one group of S states
    PassArgs args{};
    int op_index = 0;                // offset of the first device op (rebased onto the device table)
    int prog_index = 0;              // offset (16-byte words) of the launch's program
    int rb = 4;                      // register qubits
    int grid = 0;
    size_t smem = 0;
    JitPass* jit = nullptr;          // pass-specialised kernel (owned by the engine)
    bool gen = false;                // runs a pass-specialised kernel
    bool seq = false;                // multi-state pass-specialised kernel sweeps its states one at a time
    // pass, unit kernel: n_units states of any number of groups, `grid` blocks in all
    int unit_off = 0, n_units = 0, ctas = 0;
    int unit_kind = 0;               // unit_kind of their programs
    int max_words = 0, max_events = 0, n_phases = 0;
    size_t part_off = 0;             // partial sums of the launch (doubles)
    // finisher
    int n_slots = 0;
    size_t slot_off = 0;
    int fin_grid = 0;                // blocks of the reduction a normalisation reads
    // fill / copy
    float2* dst = nullptr;
    const float2* src = nullptr;
    unsigned long long bits = 0;
    double bytes = 0;                // algorithmic bytes (pass kernels)
    bool bd_table = false;           // pass saves through the block-boundary checkpoint table
    int op_counts[8] = {};           // pass: G1, G2, D1, D2, sites, reductions, spawned states, saves
    bool units() const { return n_units > 0; }
};

struct Engine {
    int sm_count = 0;
    size_t smem_optin = 0;           // largest dynamic shared memory per block
    int device = -1;
    // persistent device buffers
    void* buf = nullptr;             // one allocation for states
    size_t buf_bytes = 0;
    void* aux = nullptr;             // ops, mats, tables, partials, term values, result
    size_t aux_bytes = 0;
    // schedule cache key
    int level = -1, psi_kind = -1, v_kind = -1;
    unsigned long long psi_bits = 0, v_bits = 0;
    const void* psi_dev = nullptr;
    const void* v_dev = nullptr;
    std::vector<Launch> launches;
    SmallArgs small{};               // narrow circuits: the whole expansion (L_SMALL)
    double bound = 0;
    long long n_terms = 0;
    int eff_level = 0;
    long long* level_off_dev = nullptr;
    double* term_vals = nullptr;
    nqs_result* res_dev = nullptr;
    FinishSlot* slots_dev = nullptr;
    SweepUnit* units_dev = nullptr;
    std::vector<SweepUnit> units;    // host copy of the unit table (the batch executor regroups it)
    double* partials = nullptr;
    double* kmats_dev = nullptr;
    int* err_dev = nullptr;
    // profiling
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_pool;
    struct EvUse {
        int kind, sub;   // stats slot; second slot for sweep passes (3: several states, 4: one), -1 none
        double bytes;
    };
    std::vector<EvUse> ev_used;
    size_t ev_next = 0;
    cudaStream_t last_stream = nullptr;
    bool has_result = false;
    uint64_t upload_bytes = 0;
    uint64_t gen = 0;                // bumped whenever the schedule is rebuilt
    int spacing = 0;                 // sites per checkpoint block of the current schedule (0: every site)
    size_t n_states = 0;             // state buffers of the current schedule
    std::vector<std::unique_ptr<JitPass>> jit;   // pass-specialised kernels of the current schedule
    int jit_launches = 0;
    int jit_state = 0;               // 0 not requested, 1 built, -1 failed (interpreter runs)
    Plan wide_plan;                  // the plan re-cut for 13-qubit tiles (generated kernels)
    bool wide = false;               // the current schedule runs on wide_plan
    bool wide_failed = false;        // a wide schedule's kernels could not be built: 12-qubit tiles
    bool jit_failed = false;         // this schedule's generated kernels could not be built: the precompiled one
};


// Matrix table builder (float2 for sweeps, complex128 for finishers).
struct Tables {
    std::vector<float2> mats;
    std::vector<double> kmats;     // per site: K_0..K_3, 8 doubles each
    // unitary matrices are rounded to stay as unitary as FP32 allows (fp32_round.h)
    int add(const cd* m, int cnt, bool adjoint, int dim) {
        int off = (int)mats.size();
        cd v[16];
        for (int r = 0; r < dim; ++r)
            for (int c = 0; c < dim; ++c) v[dim * r + c] = adjoint ? std::conj(m[dim * c + r]) : m[dim * r + c];
        float2 f[16];
        round_matrix_c64(v, dim, f);
        for (int e = 0; e < dim * dim; ++e) mats.push_back(f[e]);
        (void)cnt;
        return off;
    }
};

enum RunType { RT_IDEAL, RT_BWD, RT_FWD };

struct ProgInfo {
    int words_begin = 0, n_words = 0, ops_word = 0, mats_word = 0, n_phases = 0;
};

int cuda_err(cudaError_t e);
ProgInfo build_program(const std::vector<DevOp>& dops, int off, int n, int RB, const Tables& tab,
                       std::vector<uint4>& prog, int k = kMaxTileQ);
// Device ops of one sweep direction over the passes `segs`.  Backward runs
// save phi at every site, or only at the sites flagged in `save_only`.
Run make_run(const Plan& plan, const std::vector<PassSpec>& segs, RunType rt, bool reduce, bool spawn,
             bool level0_only, const std::vector<Factors>& fac, Tables& tab, std::vector<DevOp>& dops,
             const std::vector<char>* save_only = nullptr);

// schedule construction and execution (engine.cu)
int engine_init(Engine& E);
void engine_release(Engine& E, void* stream);
// allow_jit: the schedule may use pass-specialised kernels (the batch executor
// launches passes through its own multi-circuit kernel and passes false);
// make_do: where the states do not fit, a schedule with fewer of them, else
// NQS_ERR_NOMEM; close: one of many, which together fill the device
int build_schedule(Handle& h, Engine& E, const nqs_state* psi, const nqs_state* v, int level, void* stream,
                   bool allow_jit = true, bool make_do = true, bool close = false);
int run_schedule(Handle& h, Engine& E, cudaStream_t st);
int run_launch(Handle& h, Engine& E, const Launch& l, cudaStream_t st);
// whether E's schedule is the one for these states and this level
bool schedule_current(const Engine& E, const nqs_state* psi, const nqs_state* v, int level);
// most branch-group states a schedule holds beside its checkpoints and main state
size_t group_states(const Handle& h, int level, bool generated);

}  // namespace nqs
