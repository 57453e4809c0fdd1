// Assembler of the unit sweep kernel's programs (unit_program.h).
#include "unit_program.h"

#include <algorithm>
#include <climits>
#include <cmath>
#include <complex>
#include <cstring>

#include "fp32_round.h"
#include "nqs_internal.h"

namespace nqs {

namespace {

bool is(float2 f, float re) { return f.x == re && f.y == 0.f; }

// a diagonal factor pair that is a sign: 1 or (1, -1) by another bit
bool is_sign(float2 v0, float2 v1, float2 w0, float2 w1) {
    return is(v0, 1.f) && is(v1, 1.f) && is(w0, 1.f) && is(w1, -1.f);
}

struct Records {
    std::vector<UnitRec> recs;
    std::vector<float2> mats;
    int put(const float2* v, int n) {   // matrices start on 16 bytes
        if (mats.size() & 1) mats.push_back(make_float2(0.f, 0.f));
        const int at = (int)mats.size();
        mats.insert(mats.end(), v, v + n);
        return at;
    }
    // a 2x2 matrix as the packed operands of the kernel: (re, re), (-im, im) per entry
    static void packed(const float2* f, float2* v) {
        for (int e = 0; e < 4; ++e) {
            v[2 * e] = make_float2(f[e].x, f[e].x);
            v[2 * e + 1] = make_float2(-f[e].y, f[e].y);
        }
    }
    int put_matrix(const float2* f) {
        float2 v[8];
        packed(f, v);
        return put(v, 8);
    }
    UnitRec& emit(int code, int a = kNoLoc, int b = kNoLoc) {
        UnitRec r{};
        r.code = (unsigned char)code;
        r.a = (unsigned char)a;
        r.b = (unsigned char)b;
        recs.push_back(r);
        return recs.back();
    }
    // Dense gates that nothing on their bit separates share a record, in the
    // order of their bits (so every amplitude sees the same arithmetic as with a
    // record each): decoding a record costs about as much as a third of a gate.
    size_t joint = 0;        // 1 + record that more gates may join
    size_t first = 0;        // first record of the phase
    int last_bit = 0;        // bit of the last gate
    static int pairs_of(int i) {
        int m = 0;
        for (int j = 0; j < 4; ++j)
            if (j != i) m |= 1 << unit_pair(std::min(i, j), std::max(i, j));
        return m;
    }
    bool joins(int i, int flags) const {
        if (joint == 0 || (recs[joint - 1].mask >> (8 * i)) != 0) return false;   // a bit below the ones there
        for (size_t k = joint; k < recs.size(); ++k) {
            const int code = recs[k].code;
            if (!((code >= UO_HP && code < UO_HP + 4 && code != UO_HP + i) || (code == UO_SC && !(flags & UF_SCALAR)) ||
                  (code == UO_DN && !(recs[k].a & pairs_of(i)))))
                return false;
        }
        return true;
    }
    void gate_record(int i, const float2* f, int flags, uint32_t sign) {
        float2 v[10] = {};
        std::memcpy(&v[0].x, &sign, sizeof(sign));
        packed(f, v + 2);
        const int at = put(v, 10);
        if (!joins(i, flags)) {
            unsigned char before = 0;
            if (recs.size() > first && recs.back().code == UO_DN) {
                before = recs.back().a;
                recs.pop_back();
            }
            emit(UO_G1, before);
            joint = recs.size();
        }
        UnitRec& r = recs[joint - 1];
        r.off[i] = (unsigned short)at;
        r.mask |= (unsigned)(flags | UF_HERE) << (8 * i);
        last_bit = i;
    }
    // negate where both bits of a pair are set
    void negate(int pair) {
        if (recs.size() <= first || recs.back().code != UO_DN) emit(UO_DN, 0);
        recs.back().a ^= (unsigned char)(1 << pair);
    }
    void start_phase() {
        joint = 0;
        first = recs.size();
    }
    // K_0 of a site on register bit i, and the record of its other actions
    void apply_site(int i, const float2* m, bool diag) {
        if (diag) {
            const float2 kd[2] = {m[0], m[3]};
            const int mt = put(kd, 2);
            UnitRec& r = emit(UO_KD + i);
            r.mat = (unsigned short)mt;
            if (m[0].y == 0.f && m[3].y == 0.f) r.flags = UF_REAL;
        } else {
            const int mt = put_matrix(m);
            emit(UO_GK + i).mat = (unsigned short)mt;
        }
    }
    UnitRec& site(int i, const float2* m, int n_spawn, cd scale) {
        float2 k[16];
        const float2 sc = round_c64(scale);
        k[0] = k[1] = sc;
        for (int e = 0; e < 4 * n_spawn; ++e)
            k[2 + e] = is(sc, 1.f) ? m[4 + e] : round_c64(cd(m[4 + e].x, m[4 + e].y) * scale);
        const int mt = put(k, 2 + 4 * n_spawn);
        UnitRec& r = emit(UO_SITE + i);
        r.mat = (unsigned short)mt;
        r.nspawn = (unsigned char)n_spawn;
        return r;
    }
};

// The arithmetic of every amplitude is fixed by the operation order alone: a
// pending diagonal is a scalar and one pair of factors per register bit, a
// gate takes the scalar and the pair of its bit into its matrix (scalar first),
// sites and phase ends multiply what is left into the amplitudes.  Signs (CZ)
// are exact whatever way they go, so they are kept as parities of thread and
// tile bits and cost nothing until a gate or the end of the phase takes them.
struct PairAssembler : Records {
    // what the kernel holds: scalar (and whether it is real), pairs; and signs
    bool scal = false, scal_real = true;
    bool pair[4] = {false, false, false, false};
    uint32_t sign[4] = {0, 0, 0, 0};

    void scalar(const float2* v, int n, int la, int lb) {   // by bit a + 2 * bit b
        float2 w[4] = {v[0], v[1], n > 2 ? v[2] : v[0], n > 2 ? v[3] : v[1]};
        const int at = put(w, 4);
        emit(UO_SC, la, lb).mat = (unsigned short)at;
        scal = true;
        for (const float2& f : w) scal_real = scal_real && f.y == 0.f;
    }
    // pair of bit i *= (v0, v1) or (w0, w1) by the bit at loc
    void pair_op(int i, int loc, float2 v0, float2 v1, float2 w0, float2 w1) {
        if (!pair[i] && loc != kNoLoc && is_sign(v0, v1, w0, w1)) {
            sign[i] ^= 1u << loc;
            return;
        }
        to_pair(i);
        const float2 v[4] = {v0, v1, w0, w1};
        const int at = put(v, 4);
        emit(UO_HP + i, loc).mat = (unsigned short)at;
        pair[i] = true;
    }
    // the sign of bit i joins its pair
    void to_pair(int i) {
        const float2 one = make_float2(1.f, 0.f), neg = make_float2(-1.f, 0.f);
        for (int l = 0; l < 31; ++l) {
            if (!(sign[i] >> l & 1)) continue;
            const float2 v[4] = {one, one, one, neg};
            const int at = put(v, 4);
            emit(UO_HP + i, l).mat = (unsigned short)at;
            pair[i] = true;
        }
        sign[i] = 0;
    }
    cd scale() const { return 1.0; }   // of what a site sees
    void at_site() { flush(); }
    void at_end(bool) { flush(); }
    void begin_phase(const std::vector<int>&) { start_phase(); }
    void outside(int, int) {}
    // multiply everything pending into the amplitudes
    void flush() {
        int pairs = 0, which = 0;
        for (int i = 0; i < 4; ++i)
            if (pair[i]) {
                ++pairs;
                which = i;
            }
        if (pairs > 1) {
            for (int i = 0; i < 4; ++i) to_pair(i);
            emit(UO_FLA);
        } else if (pairs == 1) {
            to_pair(which);
            emit(UO_FLB + which);
        } else if (scal) {
            emit(UO_FLS).flags = scal_real ? UF_REAL : 0;
        }
        for (int i = 0; i < 4; ++i) {
            if (sign[i]) emit(UO_FLR + i).mask = sign[i];
            pair[i] = false;
            sign[i] = 0;
        }
        scal = false;
        scal_real = true;
        joint = 0;
    }
    void g1(int i, const float2* m) {
        gate_record(i, m,
                    (pair[i] ? UF_DIAG : 0) | (sign[i] ? UF_SIGN : 0) | (scal ? UF_SCALAR : 0) | (scal_real ? UF_REAL : 0),
                    sign[i]);
        pair[i] = scal = false;
        scal_real = true;
        sign[i] = 0;
    }
    void g2(int i, int j, const float2* m) {   // first qubit on register bit i, second on j
        // the scalar and the pairs of both bits go into the matrix on the device
        to_pair(i);
        to_pair(j);
        const int at = put(m, 16);
        UnitRec& r = emit(UO_G2 + unit_pair(std::min(i, j), std::max(i, j)) + (i > j ? 6 : 0));
        r.mat = (unsigned short)at;
        r.flags = (unsigned char)((pair[i] || pair[j] ? UF_DIAG : 0) | (scal ? UF_SCALAR : 0));
        pair[i] = pair[j] = scal = false;
        scal_real = true;
    }
    void d1(int la, const float2* m) {   // m[0], m[3]
        if (la < kUnitRB) {
            pair_op(la, kNoLoc, m[0], m[3], m[0], m[3]);
        } else {
            const float2 v[2] = {m[0], m[3]};
            scalar(v, 2, la - LOC_THREAD, kNoLoc);
        }
    }
    void d2(int la, int lb, const float2* m) {   // m[5 * (2 * bit a + bit b)]
        const float2 d[4] = {m[0], m[5], m[10], m[15]};
        const bool ra = la < kUnitRB, rb = lb < kUnitRB;
        if (ra && rb) {
            if (is_sign(d[0], d[1], d[2], d[3])) {
                negate(unit_pair(std::min(la, lb), std::max(la, lb)));
                return;
            }
            const float2 v[4] = {d[0], la < lb ? d[1] : d[2], la < lb ? d[2] : d[1], d[3]};
            const int at = put(v, 4);
            emit(UO_DG + unit_pair(std::min(la, lb), std::max(la, lb))).mat = (unsigned short)at;
        } else if (ra) {
            pair_op(la, lb - LOC_THREAD, d[0], d[2], d[1], d[3]);
        } else if (rb) {
            pair_op(lb, la - LOC_THREAD, d[0], d[1], d[2], d[3]);
        } else {
            const float2 v[4] = {d[0], d[2], d[1], d[3]};
            scalar(v, 4, la - LOC_THREAD, lb - LOC_THREAD);
        }
    }
};

// Ratios: a diagonal on a register bit is its value at 0, a scalar, times a
// ratio where the bit is set.  Constants fold into matrices on the host; the
// scalar commutes with every gate, so the last gate of a phase takes it into
// its matrix (a few products per thread instead of one per amplitude).
struct RatioAssembler : Records {
    cd cs = 1.0, cp[4] = {1.0, 1.0, 1.0, 1.0};   // constants: scalar, ratios
    bool scal = false, scal_real = true;         // held by the kernel
    bool rat[4] = {false, false, false, false};
    uint32_t sign[4] = {0, 0, 0, 0};
    size_t last_gate = 0;    // 1 + record of the last one-qubit gate since the pending factors were last applied
    float2 gate[4] = {};     // its matrix
    std::vector<cd> carry;   // constant ratio pending on each tile position across phases
    std::vector<int> regs;

    static bool one(cd c) {
        if (c == cd(1.0)) return true;
        return std::fabs(c.real() - 1.0) < 1e-7 && std::fabs(c.imag()) < 1e-7 && is(round_c64(c), 1.f);
    }
    int put_c(std::initializer_list<cd> v) {
        float2 f[4];
        int n = 0;
        for (cd c : v) f[n++] = round_c64(c);
        return put(f, n);
    }
    // Rounded phases are off modulus 1 by up to 1e-8, and a circuit repeats its
    // phases (every edge of a QAOA layer has the same one), so the errors add up:
    // what the entries f of v have in common is taken out of the constants, in
    // full for a factor of all amplitudes, by half for one of those with a set
    // bit.  Signs are exact and change nothing.
    void keep_norm(int at, std::initializer_list<cd> v, double weight) {
        double s = 0.0;   // sum of the relative errors of the moduli
        const float2* f = mats.data() + at;
        for (const cd& c : v) {
            s += 0.5 * (std::norm(cd(f->x, f->y)) / std::norm(c) - 1.0);
            ++f;
        }
        if (std::fabs(s) < 1e-6) cs *= 1.0 - weight * s / (double)v.size();
    }
    void ratio(int i, cd v0, cd v1, int loc = kNoLoc) {
        const float2 f0 = round_c64(v0), f1 = round_c64(v1);
        if (loc != kNoLoc && is(f0, 1.f) && is(f1, -1.f)) {
            sign[i] ^= 1u << loc;
            return;
        }
        const int at = put_c({v0, v1});
        emit(UO_HP + i, loc).mat = (unsigned short)at;
        rat[i] = true;
        keep_norm(at, {v0, v1}, 0.5);
    }
    void scalar(cd v0, cd va, cd vb, cd vab, int la = kNoLoc, int lb = kNoLoc) {
        const int at = put_c({v0, va, vb, vab});
        emit(UO_SC, la, lb).mat = (unsigned short)at;
        scal = true;
        keep_norm(at, {v0, va, vb, vab}, 1.0);
        for (cd c : {v0, va, vb, vab}) scal_real = scal_real && round_c64(c).y == 0.f;
    }
    // keep_scalar leaves the constant scalar pending (the caller scales what it writes)
    void flush(bool keep_scalar) {
        for (int i = 0; i < 4; ++i)
            if (!one(cp[i])) {
                ratio(i, cp[i], cp[i]);
                cp[i] = 1.0;
            }
        if (!keep_scalar && !one(cs) && last_gate > 0) take_constant();
        int n = 0;
        for (int i = 0; i < 4; ++i) n += rat[i];
        if (scal && last_gate > 0 && n < 3) absorb_scalar();
        if (!keep_scalar && !one(cs)) {
            const cd all = cs;
            cs = 1.0;
            scalar(all, all, all, all);
        }
        if (8 * n + 16 * (int)scal > 31) {   // 31 products for everything at once
            emit(UO_FLA);
        } else {
            for (int i = 0; i < 4; ++i)
                if (rat[i]) emit(UO_FLB + i);
            if (scal) emit(UO_FLS).flags = scal_real ? UF_REAL : 0;
        }
        for (int i = 0; i < 4; ++i) {
            if (sign[i]) emit(UO_FLR + i).mask = sign[i];
            sign[i] = 0;
            rat[i] = false;
        }
        scal = false;
        scal_real = true;
        last_gate = joint = 0;
    }
    // The scalar's factors depend on the thread and tile alone: those that come
    // after the last gate move ahead of it, and the gate takes them.
    void absorb_scalar() {
        const size_t g = last_gate - 1;
        UnitRec r = recs[g];
        r.mask |= (unsigned)(UF_SCALAR | (scal_real ? UF_REAL : 0)) << (8 * last_bit);
        std::vector<UnitRec> before, after;
        for (size_t k = g + 1; k < recs.size(); ++k) (recs[k].code == UO_SC ? before : after).push_back(recs[k]);
        recs.resize(g);
        recs.insert(recs.end(), before.begin(), before.end());
        recs.push_back(r);
        recs.insert(recs.end(), after.begin(), after.end());
        scal = false;
        scal_real = true;
        last_gate = joint = 0;
    }
    void take_constant() {   // the constant scalar goes into the last gate's matrix
        cd k[4];
        for (int e = 0; e < 4; ++e) k[e] = cd(gate[e].x, gate[e].y) * cs;
        round_matrix_c64(k, 2, gate);
        packed(gate, mats.data() + recs[last_gate - 1].off[last_bit] + 2);
        cs = 1.0;
    }
    void g1(int i, const float2* m) {
        for (int e = 0; e < 4; ++e) gate[e] = m[e];
        if (!one(cp[i])) {
            cd k[4];
            for (int e = 0; e < 4; ++e) k[e] = cd(m[e].x, m[e].y) * ((e & 1) ? cp[i] : cd(1.0));
            round_matrix_c64(k, 2, gate);
            cp[i] = 1.0;
        }
        gate_record(i, gate, (rat[i] ? UF_DIAG : 0) | (sign[i] ? UF_SIGN : 0), sign[i]);
        rat[i] = false;
        sign[i] = 0;
        last_gate = joint;
    }
    void g2(int i, int j, const float2* m) {   // first qubit on register bit i, second on j
        for (int b : {i, j}) {
            if (!one(cp[b])) ratio(b, cp[b], cp[b]);
            cp[b] = 1.0;
            if (rat[b]) emit(UO_FLB + b);
            if (sign[b]) emit(UO_FLR + b).mask = sign[b];
            rat[b] = false;
            sign[b] = 0;
        }
        const int at = put(m, 16);
        UnitRec& r = emit(UO_G2 + unit_pair(std::min(i, j), std::max(i, j)) + (i > j ? 6 : 0));
        r.mat = (unsigned short)at;
    }
    static cd c(float2 f) { return cd(f.x, f.y); }
    // a diagonal on register bit i whose two values depend on the bit at `loc`;
    // one that vanishes where the bit is clear is applied as a dense gate
    void pair_op(int i, int loc, cd f00, cd f10, cd f01, cd f11) {   // f<bit i><bit loc>
        if (f00 == f01) cs *= f00;
        else scalar(f00, f01, f00, f01, loc);
        ratio(i, f10 / f00, f11 / f01, loc);
    }
    void d1(int la, const float2* m) {
        if (la >= kUnitRB) {
            scalar(c(m[0]), c(m[3]), c(m[0]), c(m[3]), la - LOC_THREAD);
        } else {
            cs *= c(m[0]);
            cp[la] *= c(m[3]) / c(m[0]);
        }
    }
    void d2(int la, int lb, const float2* m) {
        const cd d[4] = {c(m[0]), c(m[5]), c(m[10]), c(m[15])};   // 2 * bit a + bit b
        const bool ra = la < kUnitRB, rb = lb < kUnitRB;
        if (ra && rb) {
            cs *= d[0];
            cp[la] *= d[2] / d[0];
            cp[lb] *= d[1] / d[0];
            const cd k = d[3] * d[0] / (d[1] * d[2]);
            const int pr = unit_pair(std::min(la, lb), std::max(la, lb));
            if (is(round_c64(k), -1.f)) {
                negate(pr);
            } else if (!one(k)) {
                const int at = put_c({k, k});
                emit(UO_DG + pr).mat = (unsigned short)at;
            }
        } else if (ra) {
            pair_op(la, lb - LOC_THREAD, d[0], d[2], d[1], d[3]);
        } else if (rb) {
            pair_op(lb, la - LOC_THREAD, d[0], d[1], d[2], d[3]);
        } else {
            scalar(d[0], d[2], d[1], d[3], la - LOC_THREAD, lb - LOC_THREAD);
        }
    }
    cd scale() const { return cs; }
    void at_site() { flush(true); }
    // constants stay with their positions between phases
    void begin_phase(const std::vector<int>& R) {
        if (carry.empty()) carry.assign(kMaxTileQ, cd(1.0));
        regs = R;
        start_phase();
        for (int i = 0; i < 4; ++i) cp[i] = carry[R[i]];
        last_gate = joint = 0;
    }
    void at_end(bool last) {
        for (int i = 0; i < 4; ++i) {
            carry[regs[i]] = cp[i];
            if (!last) cp[i] = 1.0;
        }
        flush(!last);
        if (last)
            for (int i = 0; i < 4; ++i) carry[regs[i]] = 1.0;
    }
    // the constant of a tile position outside the registers, at thread bit loc
    void outside(int pos, int loc) {
        if (!one(carry[pos])) scalar(1.0, carry[pos], 1.0, carry[pos], loc);
        carry[pos] = 1.0;
    }
};

}  // namespace

namespace {

template <typename Asm>
UnitProgram assemble(const std::vector<DevOp>& dops, int off, int n, const int* local, int n_qubits,
                          const std::vector<float2>& tab, std::vector<uint4>& out) {
    static_assert(sizeof(UnitRec) == 16 && sizeof(UnitPhase) == 96 && sizeof(UnitHeader) == 64, "record sizes");
    constexpr int K = kMaxTileQ;
    UnitHeader hd{};
    int slot_site[kUnitSlots] = {};
    bool slot_used[kUnitSlots] = {}, slot_fwd[kUnitSlots] = {};
    bool in_tile[64] = {};
    for (int j = 0; j < K; ++j) {
        hd.local[j] = (unsigned char)local[j];
        in_tile[local[j]] = true;
    }
    // number of each qubit outside the tile among them: bit 8 + number of the
    // kernel's word of thread and tile bits
    int outer[64] = {}, n_outer = 0;
    for (int q = 0; q < n_qubits; ++q)
        if (!in_tile[q]) {
            outer[q] = n_outer++;
            hd.nl_mask |= 1ull << q;
        }
    // phases: runs of operations whose dense qubits fit in the register bits
    std::vector<std::pair<int, int>> ranges;
    std::vector<unsigned> regs;      // their tile positions
    unsigned cur = 0;
    int begin = 0;
    for (int o = 0; o < n; ++o) {
        const DevOp& d = dops[off + o];
        unsigned need = 0;
        if (d.type == OP_G1 || d.type == OP_SITE || d.type == OP_G2) need |= 1u << d.a;
        if (d.type == OP_G2) need |= 1u << d.b;
        if (__builtin_popcount(cur | need) > kUnitRB) {
            ranges.push_back({begin, o});
            regs.push_back(cur);
            cur = need;
            begin = o;
        } else {
            cur |= need;
        }
    }
    ranges.push_back({begin, n});
    regs.push_back(cur);

    Asm A;
    std::vector<UnitPhase> phases;
    for (size_t p = 0; p < ranges.size(); ++p) {
        std::vector<int> R;
        bool used[K] = {};
        for (int q = 0; q < K; ++q)
            if (regs[p] >> q & 1) {
                R.push_back(q);
                used[q] = true;
            }
        for (int q = K - 1; q >= 0 && (int)R.size() < kUnitRB; --q)
            if (!used[q]) {
                R.push_back(q);
                used[q] = true;
            }
        std::sort(R.begin(), R.end());
        // lanes 0-3 on free positions of distinct residue mod 4 (distinct bank
        // pairs of the padded buffers), lowest first; lane 4 on the lowest left
        std::vector<int> T;
        bool res_used[4] = {};
        for (int q = 0; q < K && (int)T.size() < 4; ++q)
            if (!used[q] && !res_used[q % 4]) {
                T.push_back(q);
                res_used[q % 4] = true;
            }
        for (int q : T) used[q] = true;
        for (int pass = 0; pass < 2; ++pass)   // lane 4 (and 3 where residues ran out), then the warps
            for (int q = 0; q < K; ++q)
                if (!used[q] && ((int)T.size() < 5 || pass)) {
                    T.push_back(q);
                    used[q] = true;
                }
        int loc[K];
        UnitPhase ph{};
        for (int i = 0; i < kUnitRB; ++i) {
            loc[R[i]] = i;
            ph.reg_j[i] = (unsigned short)(1 << R[i]);
        }
        for (int i = 0; i < K - kUnitRB; ++i) loc[T[i]] = LOC_THREAD + i;
        for (int l = 0; l < 32; ++l)
            for (int i = 0; i < 5; ++i)
                if (l >> i & 1) ph.lane_j[l] |= (unsigned short)(1 << T[i]);
        for (int w = 0; w < 8; ++w)
            for (int i = 0; i < 3; ++i)
                if (w >> i & 1) ph.warp_j[w] |= (unsigned short)(1 << T[5 + i]);
        ph.op_begin = (unsigned short)A.recs.size();
        A.begin_phase(R);
        auto at = [&](int pos, int q) { return pos >= 0 ? loc[pos] : LOC_THREAD + 8 + outer[q]; };
        for (int o = ranges[p].first; o < ranges[p].second; ++o) {
            const DevOp& d = dops[off + o];
            const float2* m = tab.data() + d.mat;
            if (d.type == OP_G1) {
                A.g1(loc[d.a], m);
            } else if (d.type == OP_G2) {
                A.g2(loc[d.a], loc[d.b], m);
            } else if (d.type == OP_D1) {
                A.d1(at(d.a, d.qa), m);
            } else if (d.type == OP_D2) {
                A.d2(at(d.a, d.qa), at(d.b, d.qb), m);
            } else if (d.type == OP_SITE) {
                const int i = loc[d.a], fl = d.flags & 0xff;
                if (fl & (FL_REDUCE | FL_SPAWN | FL_SAVE | FL_SAVE_FWD)) {
                    // the state itself is seen here
                    for (int q = 0; q < K; ++q)
                        if (loc[q] >= kUnitRB) A.outside(q, loc[q] - LOC_THREAD);
                    A.at_site();
                    UnitRec& r = A.site(i, m, (fl & FL_SPAWN) ? (d.flags >> 16) & 0xff : 0, A.scale());
                    r.flags = (unsigned char)(fl & ~(FL_APPLY | FL_KDIAG));
                    if (fl & FL_REDUCE) {
                        r.ev = (unsigned char)((d.flags >> 8) & 0xff);
                        slot_site[r.ev] = d.site;
                        slot_used[r.ev] = true;
                        hd.n_events = std::max(hd.n_events, (unsigned)r.ev + 1);
                        hd.n_slots = std::max<unsigned char>(hd.n_slots, r.ev + 1);
                    } else if (fl & (FL_SAVE | FL_SAVE_FWD)) {
                        r.ev = hd.n_slots++;
                        slot_site[r.ev] = d.site;
                        slot_used[r.ev] = true;
                        slot_fwd[r.ev] = (fl & FL_SAVE_FWD) != 0;
                    }
                    if (fl & FL_SPAWN) r.sp = (unsigned char)(d.flags >> 24);
                } else {
                    A.at_site();
                }
                if (fl & FL_APPLY) A.apply_site(i, m, (fl & FL_KDIAG) != 0);
            }
        }
        if (p + 1 == ranges.size())
            for (int q = 0; q < K; ++q)
                if (loc[q] >= kUnitRB) A.outside(q, loc[q] - LOC_THREAD);
        A.at_end(p + 1 == ranges.size());
        ph.op_end = (unsigned short)A.recs.size();
        phases.push_back(ph);
    }
    auto words = [&](const void* src, size_t bytes) {
        const size_t at = out.size(), n16 = (bytes + 15) / 16;
        out.resize(at + n16, make_uint4(0, 0, 0, 0));
        std::memcpy(out.data() + at, src, bytes);
    };
    UnitProgram info;
    info.word = (int)out.size();
    hd.n_phases = (unsigned)phases.size();
    hd.n_ops = (unsigned)A.recs.size();
    hd.ops_word = 4 + 6 * hd.n_phases;
    hd.mats_word = hd.ops_word + hd.n_ops;
    hd.words = hd.mats_word + (unsigned)((A.mats.size() + 1) / 2);
    // The sites of a pass are neighbours, however many the circuit has: slots keep
    // 15 bits, counted from the lowest one.  (The same with 32 bits a slot, in the
    // header or behind the matrices, made the sweeps 0.1 to 0.9 % slower.)
    int low = INT_MAX, high = 0;
    for (int k = 0; k < kUnitSlots; ++k)
        if (slot_used[k]) {
            low = std::min(low, slot_site[k]);
            high = std::max(high, slot_site[k]);
        }
    if (low <= high) info.site_base = low;
    for (int k = 0; k < kUnitSlots; ++k)
        if (slot_used[k]) hd.slot_site[k] = (unsigned short)((slot_site[k] - info.site_base) | (slot_fwd[k] ? 0x8000 : 0));
    if (high - info.site_base > 0x7fff) hd.words = 1u << 24;   // no planner makes one; no launch takes it
    words(&hd, sizeof(hd));
    words(phases.data(), phases.size() * sizeof(UnitPhase));
    words(A.recs.data(), A.recs.size() * sizeof(UnitRec));
    words(A.mats.data(), A.mats.size() * sizeof(float2));
    info.words = (int)hd.words;
    info.n_phases = (int)hd.n_phases;
    info.n_events = (int)hd.n_events;
    return info;
}

}  // namespace

UnitProgram assemble_unit(bool single, const std::vector<DevOp>& dops, int off, int n, const int* local, int n_qubits,
                          const std::vector<float2>& tab, std::vector<uint4>& out) {
    // pairs where the order of products shows: states swept alone through
    // diagonals that are not signs; and diagonals with zeros, which have no ratios
    bool phases = false, zeros = false;
    for (int o = off; o < off + n; ++o) {
        const DevOp& d = dops[o];
        if (d.type != OP_D1 && d.type != OP_D2) continue;
        const int dim = d.type == OP_D1 ? 2 : 4;
        for (int k = 0; k < dim; ++k) {
            const float2 f = tab[d.mat + (dim + 1) * k];
            zeros = zeros || (f.x == 0.f && f.y == 0.f);
            phases = phases || !(is(f, 1.f) || (is(f, -1.f) && d.type == OP_D2 && k == 3));
        }
    }
    UnitProgram u = (single && phases) || zeros ? assemble<PairAssembler>(dops, off, n, local, n_qubits, tab, out)
                                                : assemble<RatioAssembler>(dops, off, n, local, n_qubits, tab, out);
    u.mode = (single && phases) || zeros ? UM_PAIRS : UM_RATIOS;
    return u;
}

int unit_ctas(int n_units, long long n_tiles, int slots) {
    // Fewest tile times on the critical path: ceil(blocks / slots) rounds of
    // ceil(tiles / blocks per unit) tiles, plus a third of a tile per round for
    // a block's start (program copy, barriers, first tile not prefetched).
    const long long most = std::min<long long>(n_tiles, std::max<long long>(1, (4ll * slots) / n_units));
    double best = 1e300;
    int best_c = 1;
    for (long long c = 1; c <= most; ++c) {
        const double rounds = (double)((n_units * c + slots - 1) / slots);
        const double cost = rounds * ((double)((n_tiles + c - 1) / c) + 0.33);
        if (cost < best - 1e-9) {
            best = cost;
            best_c = (int)c;
        }
    }
    return best_c;
}

}  // namespace nqs
