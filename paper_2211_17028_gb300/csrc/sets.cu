// Evaluation of chosen noise-site sets: for a set S = {s_1 < ... < s_k}
// (k <= 3), W(S) = sum over the kept non-dominant factors at every site of S
// of the term values X (the dominant factor everywhere else) -- the
// quantity an importance-sampled estimate of the level-k sum T_k draws.
//
// nqs_prepare_sets stores phi_s (backward sweep from v) and chi_s (forward
// sweep from psi, saved before K_0 is applied) at every site.  A set is then
// evaluated between its sites' checkpoints.
//   k = 1: chi_{s_1} is reduced against phi_{s_1}.
//   k = 2: w_i = K_i chi_{s_1} is spawned (three states), swept to s_2 (K_0 at
//     the sites in between) and reduced against phi_{s_2}.
//   k = 3, meeting at s_2: u_j = K_j^dagger phi_{s_3} is spawned too and swept
//     backward to s_2, where each w_i is reduced against each u_j: six states
//     swept, and the nine 2x2 matrices give all 27 terms.
//   k = 3, forward: at s_2 the w_i spawn nine states, which are swept on and
//     reduced at s_3, at every third site of the sets that share s_1 and s_2.
// Sets are taken in lexicographic order so that sets with a common first site
// share the sweep of w_i.  A common pair meets while the third sites' backward
// sweeps (three states each) are together no longer than the nine forward
// states' sweep to the last of them, that is up to about three third sites.
//
// The sets of one first site are a chain of passes, each of which needs the
// one before; chains are independent.  They are dealt to lanes, each with its
// own states, and the r-th passes of all lanes are one launch: three states of
// a 20-qubit circuit are 768 tiles (2.5 rounds of the resident blocks), of a
// 14-qubit one twelve.  40 triples of a 20-qubit circuit with 200 noises:
// 110 ms with nine states swept by three launches of three each, one chain
// after another; 24.5 ms.
//
// When the 2N checkpoints do not fit in device memory (or the handle's
// checkpoint-spacing option asks for it), chi is kept only at the first site
// and phi only at the last site of each block of k sites: chi_{s_1} is
// recomputed by a forward sweep from its block's first site, and a block's
// phi by a backward sweep from its last site into a ring of k slots, once
// for every run of reductions that falls in the block.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <iterator>
#include <map>
#include <vector>

#include "engine_internal.h"

namespace nqs {

struct SetsState {
    int N = 0, n = 0;
    void* buf = nullptr;
    size_t buf_bytes = 0;
    void* aux = nullptr;
    size_t aux_bytes = 0;
    void* call = nullptr;
    size_t call_bytes = 0;
    std::vector<float2*> phi, chi;    // spaced: boundaries per block (phi at block-last, chi at block-first sites)
    std::vector<float2*> ring;        // spaced: recomputed phi of one block
    int spacing = 0;                  // sites per checkpoint block (0: every site)
    float2* main = nullptr;
    float2* scratch = nullptr;
    float2* work = nullptr;           // spaced: recomputed chi
    float2* work_mat = nullptr;       // spaced: backward recomputation state
    float2** phi_bd_tab = nullptr;    // spaced: site -> phi boundary of its block
    std::vector<PassSpec> segs;       // spaced: passes cut after every block-last site
    std::vector<PassSpec> fsegs;      // passes of the set sweeps: up to 16 sites each (K_0 only at most of them)
    std::vector<DevOp> mat_ops;       // spaced: backward ops saving phi at every site, per pass of segs
    std::vector<std::pair<int, int>> mat_pass;   // (first op in mat_ops, count) per pass, reversed order
    std::vector<int> mat_seg;         // segment index of each entry of mat_pass
    std::vector<int> mat_block;       // block of each entry of mat_pass
    float2* g1 = nullptr;             // lane 0: three states spawned at the first site
    float2* g2 = nullptr;             // and nine spawned at the second (or three at the third)
    int lanes = 1;                    // lane l: the same 12 states, 12 l states further on
    float2** lane_tab = nullptr;      // the first three states of g2 of every lane
    float2** phi_tab = nullptr;
    float2** chi_tab = nullptr;
    double* kmats = nullptr;
    double* partials = nullptr;
    size_t partial_doubles = 0;
    int* err = nullptr;
    Tables tab;
    std::vector<int> fwd_mat;        // forward matrix offset of every linear op
    std::vector<int> bwd_mat;        // adjoints
    std::vector<int> spawn_adj;      // per site: K_0 (unused), then the adjoints of the kept factors
    int sm_count = 0;
    bool ready = false;
};

namespace {

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// states of the lanes beyond the first, held from nqs_prepare_sets on
constexpr size_t kLaneBytes = (size_t)1 << 30;
constexpr int kMaxLanes = 96;         // three one-tile states each: the resident blocks
constexpr int kLaneStates = 12;

enum CkptTable : char { CT_PHI, CT_BOUNDARY, CT_LANE };   // what a unit's reductions and saves refer to

// One pass of a lane: its units, and the finisher slots of its reductions.
struct Step {
    int kind = 0, n_phases = 0, n_events = 0, lane = 0;
    size_t smem = 0, word = 0;
    int site_base = 0;
    CkptTable table = CT_PHI;
    std::vector<SweepUnit> units;
    struct Slot {
        int ev, state;
        FinishSlot f;
    };
    std::vector<Slot> slots;
};

struct Prog {
    int sm_count = 0;
    std::vector<DevOp> dops;          // shared-memory tile kernel
    std::vector<uint4> prog;          // unit kernel
    std::vector<SweepUnit> units;
    std::vector<size_t> unit_prog, unit_part;
    std::vector<char> unit_table, unit_lane;
    std::vector<int> unit_base;
    std::vector<std::vector<Step>> lanes = std::vector<std::vector<Step>>(1);   // passes not launched yet
    int lane = 0;                     // where passes are added
    std::vector<FinishSlot> slots;
    std::vector<Launch> L;
    size_t partial_doubles = 8, partial_top = 0, finished = 0;
    size_t take_partials(size_t need) {
        if (partial_top > 0 && partial_top + need > ((size_t)4 << 20)) flush_finish();
        const size_t at = partial_top;
        partial_top += need;
        partial_doubles = std::max(partial_doubles, partial_top);
        return at;
    }
    // finisher launch for the slots collected since the last one
    void flush_finish() {
        if (finished == slots.size()) return;
        Launch f;
        f.kind = L_FINISH;
        f.slot_off = finished;
        f.n_slots = (int)(slots.size() - finished);
        finished = slots.size();
        partial_top = 0;
        L.push_back(f);
    }
    // launches for the passes collected so far: round r takes the r-th pass of
    // every lane, one launch per kernel, the longest programs first
    void settle() {
        size_t rounds = 0;
        for (const auto& l : lanes) rounds = std::max(rounds, l.size());
        for (size_t r = 0; r < rounds; ++r)
            for (int kind = 0; kind < kUnitKinds; ++kind) {
                std::vector<const Step*> steps;
                for (const auto& l : lanes)
                    if (r < l.size() && l[r].kind == kind) steps.push_back(&l[r]);
                if (steps.empty()) continue;
                std::stable_sort(steps.begin(), steps.end(),
                                 [](const Step* x, const Step* y) { return x->n_phases > y->n_phases; });
                Launch l;
                l.kind = L_PASS;
                l.unit_kind = kind;
                l.unit_off = (int)units.size();
                for (const Step* s : steps) {
                    l.n_units += (int)s->units.size();
                    l.smem = std::max(l.smem, s->smem);
                    l.n_phases = std::max(l.n_phases, s->n_phases);
                }
                l.ctas = unit_ctas(l.n_units, steps[0]->units[0].n_tiles, unit_blocks_per_sm(kind, l.smem) * sm_count);
                l.grid = l.ctas * l.n_units;
                size_t need = 0;
                for (const Step* s : steps) need += s->units.size() * s->n_events * l.ctas * 8;
                size_t at = take_partials(need);
                int cta = 0;
                for (const Step* s : steps) {
                    const size_t event = (size_t)l.ctas * 8, state = event * s->n_events;
                    for (size_t u = 0; u < s->units.size(); ++u) {
                        units.push_back(s->units[u]);
                        units.back().ctas = l.ctas;
                        units.back().cta_begin = cta;
                        cta += l.ctas;
                        unit_prog.push_back(s->word);
                        unit_base.push_back(s->site_base);
                        unit_part.push_back(at + u * state);
                        unit_table.push_back(s->table);
                        unit_lane.push_back((char)s->lane);
                    }
                    for (const Step::Slot& x : s->slots) {
                        slots.push_back(x.f);
                        slots.back().part = at + x.state * state + x.ev * event;
                        slots.back().grid = l.ctas;
                    }
                    at += s->units.size() * state;
                }
                L.push_back(l);
            }
        for (auto& l : lanes) l.clear();
    }
    void push(const Launch& l) {   // a launch that is no unit pass
        settle();
        L.push_back(l);
    }
};

// DevOps for linear ops [a, b) of pass `ps`, with site flags chosen by
// `flag_of(site)`; back: the adjoints in reverse order.
template <typename F>
std::vector<DevOp> emit_range(const Plan& plan, const SetsState& S, const PassSpec& ps, int a, int b, F flag_of,
                              const std::vector<Factors>& fac, bool back = false) {
    std::vector<int> pos(plan.n, -1);
    for (int j = 0; j < plan.k; ++j) pos[ps.local[j]] = j;
    std::vector<DevOp> out;
    int events = 0;
    for (int e = a; e < b; ++e) {
        const int i = back ? a + b - 1 - e : e;
        const HostOp& o = plan.ops[i];
        DevOp d{};
        d.type = o.type;
        d.qa = o.q0;
        d.qb = o.q1;
        d.a = o.q0 >= 0 ? pos[o.q0] : -1;
        d.b = o.q1 >= 0 ? pos[o.q1] : -1;
        d.site = o.site;
        d.mat = back ? S.bwd_mat[i] : S.fwd_mat[i];
        if (o.type == OP_SITE) {
            int fl = flag_of(o.site);
            if (fl & FL_REDUCE) fl |= (events++) << 8;
            if (fl & FL_SPAWN) {
                fl |= fac[o.site].m << 16;
                if (back) d.mat = S.spawn_adj[o.site];
            }
            if (o.diag) fl |= FL_KDIAG;
            d.flags = fl;
        }
        out.push_back(d);
    }
    return out;
}

int pass_of(const std::vector<PassSpec>& segs, int lin) {
    for (size_t p = 0; p < segs.size(); ++p)
        if (segs[p].op_begin <= lin && lin < segs[p].op_end) return (int)p;
    return -1;
}

// One sweep pass over custom DevOps; the states and the buffers they spawn
// into are consecutive from in, out and spawn on.  out null: the swept states
// are not needed any more.  Returns what add_slot needs.
struct PassRef {
    int step = -1;                              // unit kernel: pass of the current lane
    size_t base = 0, state = 0, event = 0;      // tile kernel: layout of the partial sums
    int grid = 0;
};

PassRef add_launch(Prog& G, const Plan& plan, const SetsState& S, const PassSpec& ps, int nstates,
                   const std::vector<DevOp>& ops, const float2* in, float2* out, float2* spawn,
                   CkptTable table = CT_PHI) {
    const size_t dim = (size_t)1 << plan.n;
    PassRef pl;
    const long long n_tiles = 1ll << (plan.n - plan.k);
    if (plan.k == kMaxTileQ) {
        int local[kMaxTileQ];
        for (int j = 0; j < kMaxTileQ; ++j) local[j] = ps.local[j];
        const UnitProgram pi = assemble_unit(nstates == 1, ops, 0, (int)ops.size(), local, plan.n, S.tab.mats, G.prog);
        Step st;
        st.n_phases = pi.n_phases;
        st.n_events = pi.n_events;
        st.kind = unit_kind(nstates == 1, pi.mode);
        st.smem = unit_smem_bytes(pi.words, pi.n_events);
        st.word = (size_t)pi.word;
        st.site_base = pi.site_base;
        st.table = table;
        st.lane = G.lane;
        for (int s = 0; s < nstates; ++s) {
            SweepUnit u{};
            u.in = in + s * dim;
            u.out = out ? out + s * dim : nullptr;
            u.spawn = spawn ? spawn + 3 * s * dim : nullptr;
            u.n_tiles = (int)n_tiles;
            u.n = plan.n;
            st.units.push_back(u);
        }
        pl.step = (int)G.lanes[G.lane].size();
        G.lanes[G.lane].push_back(std::move(st));
        return pl;
    }
    Launch l;
    l.kind = L_PASS;
    l.S = nstates;
    if (!out) out = S.scratch;   // single states only
    PassArgs& a = l.args;
    a.n = plan.n;
    a.k = plan.k;
    a.c = plan.c;
    int n_ev = 0;
    for (const DevOp& d : ops)
        if (d.type == OP_SITE && (d.flags & FL_REDUCE)) ++n_ev;
    a.n_events = n_ev;
    std::vector<char> is_local(plan.n, 0);
    for (int j = 0; j < plan.k; ++j) {
        a.local[j] = ps.local[j];
        is_local[ps.local[j]] = 1;
    }
    int nl = 0;
    for (int q = 0; q < plan.n; ++q)
        if (!is_local[q]) a.nonlocal[nl++] = q;
    a.n_tiles = n_tiles;
    for (int s = 0; s < nstates; ++s) {
        a.in[s] = in + s * dim;
        a.out[s] = out + s * dim;
        if (spawn)
            for (int i = 0; i < 3; ++i) a.spawn[3 * s + i] = spawn + (3 * s + i) * dim;
    }
    l.bd_table = table == CT_BOUNDARY;
    l.op_index = (int)G.dops.size();
    G.dops.insert(G.dops.end(), ops.begin(), ops.end());
    a.n_ops = (int)ops.size();
    l.smem = (size_t)nstates * (1 << plan.k) * sizeof(float2);
    l.grid = (int)std::max<long long>(1, std::min<long long>((long long)tile_pass_blocks_per_sm(nstates, l.smem) * S.sm_count, n_tiles));
    pl.grid = l.grid;
    pl.state = (size_t)l.grid * 8;
    pl.event = pl.state * nstates;
    pl.base = l.part_off = G.take_partials(pl.event * n_ev);
    G.L.push_back(l);
    return pl;
}

// slot of one reduction (event ev of a pass, state st) at a site: factor
// position f -> value index rank_of(f)
template <typename R>
void add_slot(Prog& G, const PassRef& pl, int ev, int st, int site, const std::vector<Factors>& fac, R rank_of) {
    const Factors& ft = fac[site];
    FinishSlot f{};
    f.part = pl.base + ev * pl.event + st * pl.state;
    f.grid = pl.grid;
    for (int i = 0; i < 4; ++i) {
        f.d[i] = FinishDesc{-1, 0, 0};
        if (i >= 1 && i <= ft.m) f.d[i] = FinishDesc{(long long)rank_of(i - 1), site * 32 + ft.keep[i - 1] * 8, 0};
    }
    if (pl.step >= 0) G.lanes[G.lane][pl.step].slots.push_back({ev, st, f});
    else G.slots.push_back(f);
}

// sweep `nstates` states over the linear ops (a, b]; site t gets flag_of(t)
// (which may spawn only at b); last: the states are not needed afterwards
template <typename FlagFn, typename RankFn>
void sweep_range(Prog& G, const Handle& h, const SetsState& S, int a, int b, FlagFn flag_of, int nstates,
                 float2* states, float2* spawn, bool last, RankFn rank_of) {
    const Plan& plan = h.plan;
    for (int p = pass_of(S.fsegs, a + 1); p >= 0 && p < (int)S.fsegs.size(); ++p) {
        const PassSpec& ps = S.fsegs[p];
        const int lo = std::max(ps.op_begin, a + 1), hi = std::min(ps.op_end, b + 1);
        if (lo >= hi) break;
        const bool has_last = hi == b + 1;
        // one launch per run of at most four reductions (the kernels' reduction slots)
        for (int c0 = lo; c0 < hi;) {
            int c1 = c0, red = 0;
            while (c1 < hi) {
                const HostOp& o = plan.ops[c1];
                const bool r = o.type == OP_SITE && (flag_of(o.site) & FL_REDUCE);
                if (r && red == 4) break;
                red += r;
                ++c1;
            }
            auto ops = emit_range(plan, S, ps, c0, c1, flag_of, h.factors);
            const bool last_chunk = has_last && c1 == hi;
            const bool drop = last && last_chunk && plan.k == kMaxTileQ;
            const PassRef pl = add_launch(G, plan, S, ps, nstates, ops, states, drop ? nullptr : states,
                                          last_chunk ? spawn : nullptr);
            int ev = 0;
            for (const DevOp& d : ops) {
                if (d.type != OP_SITE || !(d.flags & FL_REDUCE)) continue;
                for (int st = 0; st < nstates; ++st)
                    add_slot(G, pl, ev, st, d.site, h.factors, [&](int f) { return rank_of(d.site, st, f); });
                ++ev;
            }
            c0 = c1;
        }
        if (has_last) break;
    }
}

// sweep `nstates` states backward over the linear ops (a, b), K_0^dagger at sites
void sweep_back(Prog& G, const Handle& h, const SetsState& S, int a, int b, int nstates, float2* states) {
    for (int p = pass_of(S.fsegs, b - 1); p >= 0; --p) {
        const PassSpec& ps = S.fsegs[p];
        const int lo = std::max(ps.op_begin, a + 1), hi = std::min(ps.op_end, b);
        if (lo >= hi) break;
        add_launch(G, h.plan, S, ps, nstates, emit_range(h.plan, S, ps, lo, hi, [](int) { return FL_APPLY; }, h.factors, true),
                   states, states, nullptr);
    }
}

// sweep `nstates` states forward over the linear ops [a, b), b a site, and
// reduce each against the lane's n_back backward states on the site's qubit
template <typename RankFn>
void sweep_and_meet(Prog& G, const Handle& h, const SetsState& S, int a, int b, int nstates, float2* states,
                    int n_back, bool last, RankFn rank_of) {
    const Plan& plan = h.plan;
    const int end = pass_of(S.fsegs, b);
    const auto apply = [](int) { return FL_APPLY; };
    for (int p = pass_of(S.fsegs, a); p < end; ++p) {
        const PassSpec& ps = S.fsegs[p];
        const int lo = std::max(ps.op_begin, a);
        if (lo < ps.op_end)
            add_launch(G, plan, S, ps, nstates, emit_range(plan, S, ps, lo, ps.op_end, apply, h.factors), states, states,
                       nullptr);
    }
    const PassSpec& ps = S.fsegs[end];
    auto ops = emit_range(plan, S, ps, std::max(ps.op_begin, a), b, apply, h.factors);
    const auto at = emit_range(plan, S, ps, b, b + 1, [](int) { return FL_REDUCE; }, h.factors);
    for (int j = 0; j < n_back; ++j) {
        ops.push_back(at[0]);
        ops.back().site = j;                              // of the lane's table
        ops.back().flags = FL_REDUCE | (j << 8);
    }
    const PassRef pl = add_launch(G, plan, S, ps, nstates, ops, states, last ? nullptr : states, nullptr, CT_LANE);
    for (int j = 0; j < n_back; ++j)
        for (int st = 0; st < nstates; ++st)
            add_slot(G, pl, j, st, plan.ops[b].site, h.factors, [&](int f) { return rank_of(j, st, f); });
}

int upload_and_run(Handle& h, SetsState& S, Prog& G, size_t extra_bytes, void** extra, cudaStream_t st) {
    G.settle();
    G.flush_finish();
    // per-call buffer: device ops, programs, units, finisher slots, partials, extra
    const size_t o_prog = align256(G.dops.size() * sizeof(DevOp) + 1);
    const size_t o_unit = align256(o_prog + G.prog.size() * sizeof(uint4) + 1);
    const size_t o_slot = align256(o_unit + G.units.size() * sizeof(SweepUnit) + 1);
    const size_t o_part = align256(o_slot + G.slots.size() * sizeof(FinishSlot) + 1);
    const size_t o_extra = align256(o_part + G.partial_doubles * sizeof(double));
    const size_t need = align256(o_extra + extra_bytes + 1);
    if (need > S.call_bytes) {
        if (S.call) {
            cudaStreamSynchronize(st);
            dev_free(S.call, S.call_bytes, st);
        }
        S.call = dev_alloc(need, st);
        S.call_bytes = S.call ? need : 0;
        if (!S.call) return NQS_ERR_NOMEM;
    }
    char* base = (char*)S.call;
    Engine E;   // a throwaway engine view carrying the pointers run_launch reads
    E.sm_count = S.sm_count;
    E.partials = (double*)(base + o_part);
    E.slots_dev = (FinishSlot*)(base + o_slot);
    E.units_dev = (SweepUnit*)(base + o_unit);
    E.kmats_dev = S.kmats;
    E.err_dev = S.err;
    for (size_t u = 0; u < G.units.size(); ++u) {
        SweepUnit& x = G.units[u];
        x.prog = (const uint4*)(base + o_prog) + G.unit_prog[u];
        x.ckpt = G.unit_table[u] == CT_LANE       ? S.lane_tab + 3 * G.unit_lane[u]
                 : G.unit_table[u] == CT_BOUNDARY ? S.phi_bd_tab
                                                  : S.phi_tab;
        x.ckpt += G.unit_base[u];
        x.ckpt_fwd = S.chi_tab + G.unit_base[u];
        x.partials = E.partials + G.unit_part[u];
        x.err = S.err;
    }
    int rc = NQS_OK;
    auto up = [&](size_t off, const void* src, size_t bytes) {
        if (bytes && rc == NQS_OK) rc = cuda_err(cudaMemcpyAsync(base + off, src, bytes, cudaMemcpyHostToDevice, st));
    };
    up(0, G.dops.data(), G.dops.size() * sizeof(DevOp));
    up(o_prog, G.prog.data(), G.prog.size() * sizeof(uint4));
    up(o_unit, G.units.data(), G.units.size() * sizeof(SweepUnit));
    up(o_slot, G.slots.data(), G.slots.size() * sizeof(FinishSlot));
    if (rc == NQS_OK && extra_bytes) rc = cuda_err(cudaMemsetAsync(base + o_extra, 0, extra_bytes, st));
    if (rc == NQS_OK) rc = cuda_err(cudaStreamSynchronize(st));   // pageable sources
    if (rc != NQS_OK) return rc;
    if (extra) *extra = base + o_extra;
    for (Launch& l : G.L) {
        if (l.kind == L_PASS && !l.units()) {
            l.args.ops = (const DevOp*)base + l.op_index;
            l.args.ckpt = l.bd_table ? S.phi_bd_tab : S.phi_tab;
            l.args.ckpt_fwd = S.chi_tab;
            l.args.partials = E.partials + l.part_off;
            l.args.err = S.err;
        }
    }
    E.term_vals = extra ? (double*)*extra : nullptr;
    for (const Launch& l : G.L) {
        rc = run_launch(h, E, l, st);
        if (rc != NQS_OK) break;
    }
    E.launches.clear();
    return rc;
}

}  // namespace

void sets_destroy(Handle& h) {
    if (!h.sets) return;
    SetsState& S = *h.sets;
    cudaDeviceSynchronize();
    if (S.buf) dev_free(S.buf, S.buf_bytes, nullptr);
    if (S.aux) dev_free(S.aux, S.aux_bytes, nullptr);
    if (S.call) dev_free(S.call, S.call_bytes, nullptr);
    delete h.sets;
    h.sets = nullptr;
}

int engine_prepare_sets(Handle& h, const nqs_state* psi, const nqs_state* v, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const Plan& plan = h.plan;
    const int N = (int)h.factors.size();
    if (N < 1) return NQS_ERR_ARG;
    sets_destroy(h);
    h.sets = new SetsState();
    SetsState& S = *h.sets;
    S.N = N;
    S.n = plan.n;
    int dev;
    if (cudaGetDevice(&dev) != cudaSuccess) return NQS_ERR_CUDA;
    cudaDeviceGetAttribute(&S.sm_count, cudaDevAttrMultiProcessorCount, dev);
    const size_t dim = (size_t)1 << plan.n;
    const size_t sbytes = dim * sizeof(float2);
    // every site, else blocks of k sites: boundaries 2 ceil(N/k), ring k, five work states, 12 group states
    auto spaced_states = [&](int k) { return 2 * (size_t)((N + k - 1) / k) + (size_t)k + 5 + 12; };
    int k = (h.opt_spacing > 0 && h.opt_spacing < N) ? h.opt_spacing : 0;
    if (k == 0) {
        const size_t own = 2 * (size_t)N + 2 + kLaneStates;
        // further lanes where they fit; narrow circuits' tile kernel and spaced
        // checkpoints have one
        S.lanes = plan.k == kMaxTileQ ? 1 + (int)std::min<size_t>(std::min(kMaxLanes, N) - 1, kLaneBytes / (kLaneStates * sbytes)) : 1;
        S.buf_bytes = (own + (size_t)(S.lanes - 1) * kLaneStates) * sbytes;
        S.buf = dev_alloc(S.buf_bytes, stream);
        if (!S.buf && S.lanes > 1) {
            S.lanes = 1;
            S.buf_bytes = own * sbytes;
            S.buf = dev_alloc(S.buf_bytes, stream);
        }
        if (!S.buf && h.opt_spacing == 0 && N > 1) {
            k = 1;
            for (int c = 2; c < N; ++c)
                if (spaced_states(c) < spaced_states(k)) k = c;
        }
    }
    if (k > 0) {
        S.lanes = 1;
        S.buf_bytes = spaced_states(k) * sbytes;
        S.buf = dev_alloc(S.buf_bytes, stream);
    }
    if (!S.buf) {
        S.buf_bytes = 0;
        sets_destroy(h);
        return NQS_ERR_NOMEM;
    }
    S.spacing = k;
    float2* b = (float2*)S.buf;
    size_t next = 0;
    const int nslots = k ? (N + k - 1) / k : N;
    for (int s = 0; s < nslots; ++s) S.phi.push_back(b + (next++) * dim);
    for (int s = 0; s < nslots; ++s) S.chi.push_back(b + (next++) * dim);
    for (int j = 0; j < k; ++j) S.ring.push_back(b + (next++) * dim);
    S.main = b + (next++) * dim;
    S.scratch = b + (next++) * dim;
    if (k) {
        S.work = b + (next++) * dim;
        S.work_mat = b + (next++) * dim;
        next++;   // spare (keeps the count of spaced_states)
    }
    S.g1 = b + next * dim;
    S.g2 = S.g1 + 3 * dim;

    // matrices: forward factors for every op (and adjoints for the backward runs)
    std::vector<char> block_last, block_first;
    if (k) {
        block_last.assign(N, 0);
        block_first.assign(N, 0);
        for (int s = 0; s < N; ++s) {
            block_last[s] = ((s + 1) % k == 0) || s == N - 1;
            block_first[s] = s % k == 0;
        }
        S.segs = segment(plan, false, h.opt_max_sites > 0 ? h.opt_max_sites : 4,
                         h.opt_max_ops > 0 ? h.opt_max_ops : 96, &block_last);
    }
    S.fsegs = segment(plan, false, 16, h.opt_max_ops > 0 ? h.opt_max_ops : 96);
    const std::vector<PassSpec>& bsegs = k ? S.segs : plan.free_passes;
    std::vector<DevOp> run_ops;
    Run run_bwd = make_run(plan, bsegs, RT_BWD, false, false, false, h.factors, S.tab, run_ops,
                           k ? &block_last : nullptr);
    Run run_fwd = make_run(plan, plan.free_passes, RT_FWD, false, false, false, h.factors, S.tab, run_ops);
    S.fwd_mat.assign(plan.ops.size(), -1);
    for (const RunPass& rp : run_fwd.passes)
        for (int o = 0; o < rp.n_ops; ++o) S.fwd_mat[rp.lin[o]] = run_ops[rp.op_off + o].mat;
    S.bwd_mat.assign(plan.ops.size(), -1);
    for (const RunPass& rp : run_bwd.passes)
        for (int o = 0; o < rp.n_ops; ++o) S.bwd_mat[rp.lin[o]] = run_ops[rp.op_off + o].mat;
    for (int s = 0; s < N; ++s) {
        const Factors& f = h.factors[s];
        S.spawn_adj.push_back(S.tab.add(f.K[0].data(), 4, true, 2));
        for (int j = 0; j < 3; ++j) {
            const Mat2 z{};
            S.tab.add((j < f.m ? f.K[f.keep[j]] : z).data(), 4, true, 2);
        }
    }
    Run run_ideal;
    if (v->kind == NQS_STATE_IDEAL) run_ideal = make_run(plan, plan.free_passes, RT_IDEAL, false, false, false, h.factors,
                                                         S.tab, run_ops);
    if (k) {
        // per-block recomputation of phi (saves at every site), kept for evaluation calls
        Run run_mat = make_run(plan, S.segs, RT_BWD, false, false, false, h.factors, S.tab, S.mat_ops);
        const int nb = (N + k - 1) / k;
        for (size_t p = 0; p < run_mat.passes.size(); ++p) {
            const RunPass& rp = run_mat.passes[p];
            int blk = nb;
            if (!rp.lin.empty())
                for (int c = 0; c < nb; ++c)
                    if (rp.lin[0] <= plan.site_pos[std::min(N, (c + 1) * k) - 1]) {
                        blk = c;
                        break;
                    }
            S.mat_pass.push_back({rp.op_off, rp.n_ops});
            S.mat_seg.push_back((int)(run_mat.passes.size() - 1 - p));
            S.mat_block.push_back(blk);
        }
    }

    // aux: checkpoint tables, factor table (complex128), status word, matrix table
    const size_t o_phi = 0, o_chi = align256(N * sizeof(float2*));
    const size_t o_kmat = align256(o_chi + N * sizeof(float2*));
    const size_t o_err = align256(o_kmat + (size_t)N * 32 * sizeof(double));
    const size_t o_mats = align256(o_err + sizeof(int));
    const size_t o_bd = align256(o_mats + S.tab.mats.size() * sizeof(float2) + 1);
    const size_t o_lane = align256(o_bd + N * sizeof(float2*));
    S.aux_bytes = align256(o_lane + 3 * (size_t)S.lanes * sizeof(float2*));
    S.aux = dev_alloc(S.aux_bytes, stream);
    if (!S.aux) {
        S.aux_bytes = 0;
        sets_destroy(h);
        return NQS_ERR_NOMEM;
    }
    char* ab = (char*)S.aux;
    S.phi_tab = (float2**)(ab + o_phi);
    S.chi_tab = (float2**)(ab + o_chi);
    S.kmats = (double*)(ab + o_kmat);
    S.err = (int*)(ab + o_err);
    S.phi_bd_tab = (float2**)(ab + o_bd);
    S.lane_tab = (float2**)(ab + o_lane);
    float2* mats_dev = (float2*)(ab + o_mats);
    std::vector<double> kh((size_t)N * 32);
    for (int s = 0; s < N; ++s)
        for (int i = 0; i < 4; ++i)
            for (int e = 0; e < 4; ++e) {
                kh[s * 32 + i * 8 + 2 * e] = h.factors[s].K[i][e].real();
                kh[s * 32 + i * 8 + 2 * e + 1] = h.factors[s].K[i][e].imag();
            }
    std::vector<float2*> phi_t(N), chi_t(N), bd_t(N);
    for (int s = 0; s < N; ++s) {
        phi_t[s] = k ? S.ring[s % k] : S.phi[s];
        chi_t[s] = k ? S.chi[s / k] : S.chi[s];
        bd_t[s] = k ? S.phi[s / k] : S.phi[s];
    }
    std::vector<float2*> lane_t;
    for (int l = 0; l < S.lanes; ++l)
        for (int j = 0; j < 3; ++j) lane_t.push_back(S.g2 + ((size_t)l * kLaneStates + j) * dim);
    int rc = NQS_OK;
    auto up = [&](void* dst, const void* src, size_t bytes) {
        if (bytes && rc == NQS_OK) rc = cuda_err(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st));
    };
    up(S.lane_tab, lane_t.data(), lane_t.size() * sizeof(float2*));
    up(S.phi_tab, phi_t.data(), N * sizeof(float2*));
    up(S.chi_tab, chi_t.data(), N * sizeof(float2*));
    up(S.phi_bd_tab, bd_t.data(), N * sizeof(float2*));
    up(S.kmats, kh.data(), kh.size() * sizeof(double));
    up(mats_dev, S.tab.mats.data(), S.tab.mats.size() * sizeof(float2));
    if (rc == NQS_OK) rc = cuda_err(cudaMemsetAsync(S.err, 0, sizeof(int), st));
    if (rc == NQS_OK) rc = cuda_err(cudaStreamSynchronize(st));
    if (rc != NQS_OK) {
        sets_destroy(h);
        return rc;
    }

    // checkpoint sweeps: (ideal v) -> backward saving phi -> forward saving chi
    Prog G;
    G.sm_count = S.sm_count;
    auto run_passes = [&](const Run& run, const std::vector<PassSpec>& segs, const float2* first_in, bool bwd,
                          bool save_fwd) {
        for (size_t p = 0; p < run.passes.size(); ++p) {
            const RunPass& rp = run.passes[p];
            // the backward sweep is done once phi of the first site is saved, the
            // forward one once chi of the last site is
            if (p > 0 && !rp.lin.empty()) {
                if (bwd && *std::max_element(rp.lin.begin(), rp.lin.end()) < plan.site_pos[0]) break;
                if (save_fwd && *std::min_element(rp.lin.begin(), rp.lin.end()) > plan.site_pos[N - 1]) break;
            }
            std::vector<DevOp> ops(run_ops.begin() + rp.op_off, run_ops.begin() + rp.op_off + rp.n_ops);
            for (DevOp& d : ops)
                if (d.type == OP_SITE && save_fwd)
                    d.flags = FL_APPLY | ((!k || block_first[d.site]) ? FL_SAVE_FWD : 0) | (d.flags & FL_KDIAG);
            const PassSpec& ps = segs[bwd ? run.passes.size() - 1 - p : p];
            add_launch(G, plan, S, ps, 1, ops, (p == 0 && first_in) ? first_in : S.main, S.main, nullptr,
                       bwd ? CT_BOUNDARY : CT_PHI);
        }
    };
    auto fill = [&](const nqs_state* st8, const float2*& ext) {
        ext = nullptr;
        if (st8->kind == NQS_STATE_BASIS) {
            Launch l;
            l.kind = L_FILL;
            l.dst = S.main;
            l.bits = st8->bits;
            G.push(l);
        } else {
            ext = (const float2*)st8->dev;
        }
    };
    const float2* ext = nullptr;
    if (v->kind == NQS_STATE_IDEAL) {
        fill(psi, ext);
        run_passes(run_ideal, plan.free_passes, ext, false, false);
        ext = nullptr;
    } else {
        fill(v, ext);
    }
    run_passes(run_bwd, bsegs, ext, true, false);
    fill(psi, ext);
    run_passes(run_fwd, plan.free_passes, ext, false, true);
    G.settle();
    // the matrices of the device table: programs index their own copies, the
    // shared-memory tile kernel reads the table
    for (Launch& l : G.L)
        if (l.kind == L_PASS && !l.units()) l.args.mats = mats_dev;
    rc = upload_and_run(h, S, G, 0, nullptr, st);
    if (rc == NQS_OK) rc = cuda_err(cudaStreamSynchronize(st));
    if (rc != NQS_OK) {
        sets_destroy(h);
        return rc;
    }
    S.ready = true;
    return NQS_OK;
}

int engine_eval_sets(Handle& h, int k, const int* sets, size_t m, double* W_out, void* stream) {
    if (!h.sets || !h.sets->ready) return NQS_ERR_ORDER;
    SetsState& S = *h.sets;
    const Plan& plan = h.plan;
    cudaStream_t st = (cudaStream_t)stream;
    if (k < 1 || k > 3 || m == 0) return NQS_ERR_ARG;
    for (size_t j = 0; j < m; ++j)
        for (int r = 0; r < k; ++r) {
            const int s = sets[j * k + r];
            if (s < 0 || s >= S.N || (r > 0 && s <= sets[j * k + r - 1])) return NQS_ERR_ARG;
        }
    Prog G;
    G.sm_count = S.sm_count;
    const float2* mats_dev = nullptr;
    {
        // the matrix table sits at the end of aux (see engine_prepare_sets)
        const size_t o_chi = align256(S.N * sizeof(float2*));
        const size_t o_kmat = align256(o_chi + S.N * sizeof(float2*));
        const size_t o_err = align256(o_kmat + (size_t)S.N * 32 * sizeof(double));
        mats_dev = (const float2*)((char*)S.aux + align256(o_err + sizeof(int)));
    }
    std::vector<size_t> order(m);
    for (size_t j = 0; j < m; ++j) order[j] = j;
    std::sort(order.begin(), order.end(), [&](size_t x, size_t y) {
        return std::lexicographical_compare(sets + x * k, sets + x * k + k, sets + y * k, sets + y * k + k);
    });
    auto at = [&](size_t r, int c) { return sets[order[r] * k + c]; };
    const int K = S.spacing;
    // spaced checkpoints: phi of block c into the ring (once per run of reductions in it)
    int ring_block = -1;
    auto materialize = [&](int c) {
        if (!K || ring_block == c) return;
        bool first_in = true;
        for (size_t p = 0; p < S.mat_pass.size(); ++p) {
            if (S.mat_block[p] != c) continue;
            std::vector<DevOp> ops(S.mat_ops.begin() + S.mat_pass[p].first,
                                   S.mat_ops.begin() + S.mat_pass[p].first + S.mat_pass[p].second);
            add_launch(G, plan, S, S.segs[S.mat_seg[p]], 1, ops, first_in ? S.phi[c] : S.work_mat, S.work_mat, nullptr);
            first_in = false;
        }
        ring_block = c;
    };
    auto phi_of = [&](int t) { return K ? S.ring[t % K] : S.phi[t]; };
    // chi_{s1}: stored, or swept forward from the first site of its block
    auto chi_of = [&](int s1) -> const float2* {
        if (!K) return S.chi[s1];
        const int first = (s1 / K) * K;
        if (s1 == first) return S.chi[s1 / K];
        Launch c;
        c.kind = L_COPY;
        c.dst = S.work;
        c.src = S.chi[s1 / K];
        G.push(c);
        sweep_range(G, h, S, plan.site_pos[first] - 1, plan.site_pos[s1] - 1, [](int) { return FL_APPLY; }, 1, S.work,
                    nullptr, false, [](int, int, int) { return -1ll; });
        return S.work;
    };
    // sweep `states` from linear op `from` through the reduction sites of
    // `slots` (site -> value slot base), one checkpoint block at a time
    auto reduce_through = [&](int from, const std::map<int, long long>& slots, int nst, float2* states,
                              bool drop) {
        int pos = from;
        for (auto it = slots.begin(); it != slots.end();) {
            const int blk = K ? it->first / K : 0;
            auto end = it;
            while (end != slots.end() && (!K || end->first / K == blk)) ++end;
            materialize(blk);
            const int last = std::prev(end)->first;
            sweep_range(G, h, S, pos, plan.site_pos[last],
                        [&](int t) { return FL_APPLY | (slots.count(t) ? FL_REDUCE : 0); }, nst, states, nullptr,
                        drop && end == slots.end(),
                        [&](int t, int st, int f) { return slots.at(t) + 3 * st + f; });
            pos = plan.site_pos[last];
            it = end;
        }
    };
    if (k == 1) {
        for (size_t r = 0; r < m; ++r) {
            const int s1 = at(r, 0);
            const float2* chi = chi_of(s1);
            materialize(K ? s1 / K : 0);
            const long long base = (long long)order[r] * 27;
            Launch l;
            l.kind = L_REDUCE2;
            l.src = phi_of(s1);
            l.dst = const_cast<float2*>(chi);   // read only
            l.bits = (unsigned long long)h.circ.noises[s1].qubit;
            const long long npairs = 1ll << (plan.n - 1);
            PassRef pl;
            G.settle();
            pl.grid = l.grid = (int)std::max<long long>(
                1, std::min<long long>((long long)S.sm_count * 4, (npairs + 16ll * kThreads - 1) / (16ll * kThreads)));
            pl.base = l.part_off = G.take_partials((size_t)l.grid * 8);
            G.push(l);
            add_slot(G, pl, 0, 0, s1, h.factors, [&](int f) { return base + f; });
        }
    }
    // sets [i, i1) of the first site at(i, 0), as passes of the current lane
    auto chain = [&](size_t i, size_t i1) {
        float2* const g1 = S.g1 + (size_t)G.lane * kLaneStates * ((size_t)1 << plan.n);
        float2* const g2 = g1 + (S.g2 - S.g1);
        const size_t dim = (size_t)1 << plan.n;
        const int s1 = at(i, 0), p1 = plan.site_pos[s1], m1 = h.factors[s1].m;
        if (m1 == 0) return;   // every term is zero
        // spawn K_i chi_{s1} into the first group (shared by every set starting at s1)
        const PassSpec& ps1 = S.fsegs[pass_of(S.fsegs, p1)];
        const float2* chi = chi_of(s1);
        add_launch(G, plan, S, ps1, 1, emit_range(plan, S, ps1, p1, p1 + 1, [](int) { return FL_SPAWN; }, h.factors), chi,
                   nullptr, g1);
        if (k == 2) {
            std::map<int, long long> base2;   // second site -> value slots of its set
            for (size_t r = i; r < i1; ++r) base2[at(r, 1)] = (long long)order[r] * 27;
            reduce_through(p1, base2, m1, g1, true);
            return;
        }
        int pos = p1;   // operations up to here are applied to the first group
        for (size_t r = i; r < i1;) {
            const int s2 = at(r, 1), p2 = plan.site_pos[s2], m2 = h.factors[s2].m;
            size_t r2 = r;
            while (r2 < i1 && at(r2, 1) == s2) ++r2;
            std::map<int, long long> base3;   // third site -> value slots of its set
            long long back = 0;
            for (size_t q = r; q < r2; ++q) {
                base3[at(q, 2)] = (long long)order[q] * 27;
                back += (long long)h.factors[at(q, 2)].m * (plan.site_pos[at(q, 2)] - p2);
            }
            const long long fwd = (long long)m1 * m2 * (plan.site_pos[base3.rbegin()->first] - p2);
            if (m2 == 0) {
                r = r2;
                continue;
            }
            if (!K && plan.k == kMaxTileQ && back <= fwd) {
                for (auto it = base3.begin(); it != base3.end(); ++it) {
                    const int s3 = it->first, p3 = plan.site_pos[s3], m3 = h.factors[s3].m;
                    if (m3 == 0) continue;
                    const PassSpec& ps3 = S.fsegs[pass_of(S.fsegs, p3)];
                    add_launch(G, plan, S, ps3, 1,
                               emit_range(plan, S, ps3, p3, p3 + 1, [](int) { return FL_SPAWN; }, h.factors, true), S.phi[s3],
                               nullptr, g2);
                    sweep_back(G, h, S, p2, p3, m3, g2);
                    sweep_and_meet(G, h, S, pos + 1, p2, m1, g1, m3, r2 == i1 && std::next(it) == base3.end(),
                                   [&](int j, int st, int f) { return it->second + 9 * st + 3 * f + j; });
                    pos = p2 - 1;
                }
                r = r2;
                continue;
            }
            // carry the first group to s2 (K_0 there), spawning the nine states
            sweep_range(G, h, S, pos, p2, [&](int t) { return FL_APPLY | (t == s2 ? FL_SPAWN : 0); }, m1, g1, g2, false,
                        [](int, int, int) { return -1ll; });
            pos = p2;
            if (m2 == 3 && plan.k == kMaxTileQ) {
                reduce_through(p2, base3, 3 * m1, g2, true);
            } else {
                // one checkpoint block at a time for all groups, so each block's phi is recomputed once
                int gpos[3] = {p2, p2, p2};
                for (auto it = base3.begin(); it != base3.end();) {
                    const int blk = K ? it->first / K : 0;
                    auto end = it;
                    while (end != base3.end() && (!K || end->first / K == blk)) ++end;
                    std::map<int, long long> part(it, end);
                    for (int g = 0; g < m1; ++g) {
                        std::map<int, long long> bg = part;
                        for (auto& e : bg) e.second += g * 9;
                        reduce_through(gpos[g], bg, m2, g2 + (size_t)3 * g * dim, false);
                        gpos[g] = plan.site_pos[std::prev(end)->first];
                    }
                    it = end;
                }
            }
            r = r2;
        }
    };
    if (k > 1) {
        // chains, the longest first, each to the lane with the least work
        struct Chain {
            size_t begin, end;
            long long ops;
        };
        std::vector<Chain> chains;
        for (size_t i = 0; i < m;) {
            Chain c{i, i, 0};
            while (c.end < m && at(c.end, 0) == at(i, 0)) {
                const size_t r = c.end++;
                c.ops += plan.site_pos[at(r, k - 1)] - plan.site_pos[at(r, 0)];
            }
            chains.push_back(c);
            i = c.end;
        }
        const int lanes = std::min<int>(S.lanes, (int)chains.size());
        if (lanes > 1)
            std::stable_sort(chains.begin(), chains.end(), [](const Chain& x, const Chain& y) { return x.ops > y.ops; });
        G.lanes.resize(lanes);
        for (const Chain& c : chains) {
            G.lane = 0;
            for (int l = 1; l < lanes; ++l)
                if (G.lanes[l].size() < G.lanes[G.lane].size()) G.lane = l;
            chain(c.begin, c.end);
        }
        G.lane = 0;
    }
    G.settle();
    for (Launch& l : G.L)
        if (l.kind == L_PASS && !l.units()) l.args.mats = mats_dev;
    void* vals = nullptr;
    int rc = upload_and_run(h, S, G, m * 27 * sizeof(double), &vals, st);   // value slots start at zero
    if (rc != NQS_OK) return rc;
    std::vector<double> hv(m * 27);
    rc = cuda_err(cudaMemcpyAsync(hv.data(), vals, m * 27 * sizeof(double), cudaMemcpyDeviceToHost, st));
    if (rc == NQS_OK) rc = cuda_err(cudaStreamSynchronize(st));
    if (rc != NQS_OK) return rc;
    int err = 0;
    cudaMemcpy(&err, S.err, sizeof(int), cudaMemcpyDeviceToHost);
    if (err) return NQS_ERR_DEVICE_TIMEOUT;
    for (size_t j = 0; j < m; ++j) {
        double w = 0.0;
        for (int t = 0; t < 27; ++t) w += hv[j * 27 + t];
        W_out[j] = w;
    }
    return NQS_OK;
}

}  // namespace nqs
