// Assembler of the unit sweep kernel's programs (unit_program.h).
#include "unit_program.h"

#include <algorithm>
#include <cmath>
#include <complex>
#include <cstring>

#include "fp32_round.h"
#include "nqs_internal.h"

namespace nqs {

namespace {

struct Assembler {
    const std::vector<float2>& tab;
    std::vector<UnitRec> recs;
    std::vector<float2> mats;
    // pending diagonal of the current phase: constants known here, and flags of
    // the factors the kernel holds (scalar; one ratio per register bit)
    cd cs = 1.0, cp[4] = {1.0, 1.0, 1.0, 1.0};
    bool rs = false, rh[4] = {false, false, false, false};

    explicit Assembler(const std::vector<float2>& t) : tab(t) {}

    cd m(int off) const { return cd(tab[off].x, tab[off].y); }
    static bool one(cd c) {
        const float2 f = round_c64(c);
        return f.x == 1.f && f.y == 0.f;
    }
    int put(const std::vector<cd>& v) {   // matrix entries, 16-byte aligned
        if (mats.size() & 1) mats.push_back(make_float2(0.f, 0.f));
        const int at = (int)mats.size();
        for (cd c : v) mats.push_back(round_c64(c));
        return at;
    }
    UnitRec& emit(int code, int a = kNoLoc, int b = kNoLoc) {
        UnitRec r{};
        r.code = (unsigned char)code;
        r.a = (unsigned char)a;
        r.b = (unsigned char)b;
        recs.push_back(r);
        return recs.back();
    }
    void ratio(int i, cd c) {   // ratio of bit i *= constant
        const int at = put({c, c});
        emit(UO_HR + i).mat = (unsigned short)at;
        rh[i] = true;
    }
    void scalar_const(cd c) {
        const int at = put({c, c});
        emit(UO_SC).mat = (unsigned short)at;
        rs = true;
    }
    // multiply everything pending into the amplitudes; keep_scalar leaves the
    // constant scalar pending (the caller scales what it writes)
    void flush(bool keep_scalar) {
        for (int i = 0; i < 4; ++i)
            if (!one(cp[i])) {
                ratio(i, cp[i]);
                cp[i] = 1.0;
            }
        int bits = 0;
        for (int i = 0; i < 4; ++i) bits += rh[i];
        if (!keep_scalar && !one(cs)) {
            scalar_const(cs);
            cs = 1.0;
        }
        // 8 products per ratio and 16 for the scalar one by one, 31 for all at once
        if (8 * bits + 16 * (int)rs > 31) {
            emit(UO_FLA);
        } else {
            for (int i = 0; i < 4; ++i)
                if (rh[i]) emit(UO_FLB + i);
            if (rs) emit(UO_FLS);
        }
        rs = false;
        for (bool& r : rh) r = false;
    }
    void g1(int i, const cd* g) {
        std::vector<cd> k = {g[0] * cs, g[1] * cs * cp[i], g[2] * cs, g[3] * cs * cp[i]};
        if (mats.size() & 1) mats.push_back(make_float2(0.f, 0.f));
        const int at = (int)mats.size();
        float2 f[4];
        if (cs == 1.0 && cp[i] == 1.0)
            for (int e = 0; e < 4; ++e) f[e] = make_float2((float)g[e].real(), (float)g[e].imag());
        else
            round_matrix_c64(k.data(), 2, f);
        mats.insert(mats.end(), f, f + 4);
        cs = 1.0;
        cp[i] = 1.0;
        emit((rh[i] ? UO_G1H : UO_G1) + i).mat = (unsigned short)at;
        rh[i] = false;
    }
    void g2(int i, int j, const cd* g) {   // first qubit on register bit i, second on j
        for (int b : {i, j})
            if (rh[b]) {
                emit(UO_FLB + b);
                rh[b] = false;
            }
        std::vector<cd> k(16);
        for (int r = 0; r < 4; ++r)
            for (int c = 0; c < 4; ++c)
                k[4 * r + c] = g[4 * r + c] * cs * ((c & 2) ? cp[i] : cd(1.0)) * ((c & 1) ? cp[j] : cd(1.0));
        if (i > j) {   // index by the lower register bit first
            auto sw = [](int x) { return ((x & 1) << 1) | (x >> 1); };
            std::vector<cd> t(16);
            for (int r = 0; r < 4; ++r)
                for (int c = 0; c < 4; ++c) t[4 * sw(r) + sw(c)] = k[4 * r + c];
            k.swap(t);
        }
        float2 f[16];
        round_matrix_c64(k.data(), 4, f);
        if (mats.size() & 1) mats.push_back(make_float2(0.f, 0.f));
        const int at = (int)mats.size();
        mats.insert(mats.end(), f, f + 16);
        cs = cp[i] = cp[j] = 1.0;
        emit(UO_G2 + unit_pair(std::min(i, j), std::max(i, j))).mat = (unsigned short)at;
    }
    // a diagonal on register bit i whose two values depend on the bit at `loc`
    void pair_op(int i, int loc, cd f00, cd f10, cd f01, cd f11) {   // f<bit i><bit loc>
        if (f00 == 0.0 || f01 == 0.0) {
            const int at = put({f00, f10, f01, f11});
            emit(UO_DP, loc, i).mat = (unsigned short)at;
        } else if (f00 == f01) {
            cs *= f00;
            const int at = put({f10 / f00, f11 / f01});
            emit(UO_HR + i, loc).mat = (unsigned short)at;
            rh[i] = true;
        } else {
            const int at = put({f00, f10 / f00, f01, f11 / f01});
            emit(UO_HP + i, loc).mat = (unsigned short)at;
            rh[i] = rs = true;
        }
    }
    void d1(int la, const cd* g) {   // g[0], g[3]
        if (la < kUnitRB) {
            if (g[0] == 0.0) {
                g1(la, g);
            } else {
                cs *= g[0];
                cp[la] *= g[3] / g[0];
            }
            return;
        }
        const int at = put({g[0], g[3]});
        emit(UO_SC, la - LOC_THREAD).mat = (unsigned short)at;
        rs = true;
    }
    void d2(int la, int lb, const cd* d) {   // d[2 * bit a + bit b]
        const bool ra = la < kUnitRB, rb = lb < kUnitRB;
        if (ra && rb) {
            if (d[0] == 0.0 || d[1] == 0.0 || d[2] == 0.0) {
                const int at = put({d[0], d[1], d[2], d[3]});
                emit(UO_DG, la, lb).mat = (unsigned short)at;
                return;
            }
            cs *= d[0];
            cp[la] *= d[2] / d[0];
            cp[lb] *= d[1] / d[0];
            const cd k = d[3] * d[0] / (d[1] * d[2]);
            if (!one(k)) {
                const int at = put({k, k});
                emit(UO_DD + unit_pair(std::min(la, lb), std::max(la, lb))).mat = (unsigned short)at;
            }
        } else if (ra) {
            pair_op(la, lb - LOC_THREAD, d[0], d[2], d[1], d[3]);
        } else if (rb) {
            pair_op(lb, la - LOC_THREAD, d[0], d[1], d[2], d[3]);
        } else {
            const int at = put({d[0], d[2], d[1], d[3]});   // index bit a + 2 * bit b
            emit(UO_SC, la - LOC_THREAD, lb - LOC_THREAD).mat = (unsigned short)at;
            rs = true;
        }
    }
};

}  // namespace

UnitProgram assemble_unit(const std::vector<DevOp>& dops, int off, int n, const int* local, int n_qubits,
                          const std::vector<float2>& tab, std::vector<uint4>& out) {
    static_assert(sizeof(UnitRec) == 16 && sizeof(UnitPhase) == 96 && sizeof(UnitHeader) == 64, "record sizes");
    constexpr int K = kMaxTileQ;
    UnitHeader hd{};
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
    std::vector<std::vector<int>> regs;
    std::vector<int> cur;
    int begin = 0;
    for (int o = 0; o < n; ++o) {
        const DevOp& d = dops[off + o];
        int need[2], cnt = 0;
        if (d.type == OP_G1 || d.type == OP_SITE || d.type == OP_G2) need[cnt++] = d.a;
        if (d.type == OP_G2) need[cnt++] = d.b;
        std::vector<int> u = cur;
        for (int c = 0; c < cnt; ++c)
            if (std::find(u.begin(), u.end(), need[c]) == u.end()) u.push_back(need[c]);
        if ((int)u.size() > kUnitRB) {
            ranges.push_back({begin, o});
            regs.push_back(cur);
            cur.assign(need, need + cnt);
            begin = o;
        } else {
            cur.swap(u);
        }
    }
    ranges.push_back({begin, n});
    regs.push_back(cur);

    Assembler A(tab);
    std::vector<UnitPhase> phases;
    cd carry[K];   // constant ratio pending on each tile position across phases
    for (cd& c : carry) c = 1.0;
    for (size_t p = 0; p < ranges.size(); ++p) {
        std::vector<int> R = regs[p];
        bool used[K] = {};
        for (int q : R) used[q] = true;
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
        auto at = [&](int pos, int q) { return pos >= 0 ? loc[pos] : LOC_THREAD + 8 + outer[q]; };
        for (int i = 0; i < kUnitRB; ++i) A.cp[i] = carry[R[i]];
        for (int o = ranges[p].first; o < ranges[p].second; ++o) {
            const DevOp& d = dops[off + o];
            cd g[16];
            const int cnt = (d.type == OP_G2 || d.type == OP_D2) ? 16 : 4;
            for (int e = 0; e < cnt; ++e) g[e] = A.m(d.mat + e);
            if (d.type == OP_G1) {
                A.g1(loc[d.a], g);
            } else if (d.type == OP_G2) {
                A.g2(loc[d.a], loc[d.b], g);
            } else if (d.type == OP_D1) {
                A.d1(at(d.a, d.qa), g);
            } else if (d.type == OP_D2) {
                const cd dd[4] = {g[0], g[5], g[10], g[15]};
                A.d2(at(d.a, d.qa), at(d.b, d.qb), dd);
            } else if (d.type == OP_SITE) {
                const int i = loc[d.a], fl = d.flags & 0xff;
                if (fl & (FL_REDUCE | FL_SPAWN | FL_SAVE | FL_SAVE_FWD)) {
                    // the state itself is seen here: constant ratios of the other
                    // positions too
                    for (int q = 0; q < K; ++q)
                        if (loc[q] >= kUnitRB && !A.one(carry[q])) {
                            const int mt = A.put({1.0, carry[q]});
                            A.emit(UO_SC, loc[q] - LOC_THREAD).mat = (unsigned short)mt;
                            A.rs = true;
                            carry[q] = 1.0;
                        }
                    A.flush(true);
                    std::vector<cd> k = {A.cs, A.cs};
                    const int ns = (fl & FL_SPAWN) ? (d.flags >> 16) & 0xff : 0;
                    for (int f = 0; f < ns; ++f)
                        for (int e = 0; e < 4; ++e) k.push_back(A.m(d.mat + 4 * (f + 1) + e) * A.cs);
                    const int mt = A.put(k);
                    UnitRec& r = A.emit(UO_SITE + i);
                    r.mat = (unsigned short)mt;
                    r.flags = (unsigned char)(fl & ~(FL_APPLY | FL_KDIAG));
                    r.nspawn = (unsigned char)ns;
                    r.site = (unsigned short)d.site;
                    if (fl & FL_REDUCE) {
                        r.ev = (unsigned char)((d.flags >> 8) & 0xff);
                        hd.slot_site[r.ev] = (unsigned short)d.site;
                        hd.n_events = std::max(hd.n_events, (unsigned)r.ev + 1);
                        hd.n_slots = std::max<unsigned char>(hd.n_slots, r.ev + 1);
                    } else if (fl & (FL_SAVE | FL_SAVE_FWD)) {
                        r.ev = hd.n_slots++;
                        hd.slot_site[r.ev] = (unsigned short)(d.site | ((fl & FL_SAVE_FWD) ? 0x8000 : 0));
                    }
                    if (fl & FL_SPAWN) r.sp = (unsigned char)(d.flags >> 24);
                }
                if (fl & FL_APPLY) {
                    if (fl & FL_KDIAG) A.d1(i, g);
                    else A.g1(i, g);
                }
            }
        }
        for (int i = 0; i < kUnitRB; ++i) carry[R[i]] = A.cp[i];
        if (p + 1 == ranges.size()) {
            for (int q = 0; q < K; ++q)
                if (loc[q] >= kUnitRB && !A.one(carry[q])) {
                    const int mt = A.put({1.0, carry[q]});
                    A.emit(UO_SC, loc[q] - LOC_THREAD).mat = (unsigned short)mt;
                    A.rs = true;
                }
            A.flush(false);
        } else {
            // constants stay with their positions; what the threads hold does not
            for (cd& c : A.cp) c = 1.0;
            A.flush(true);
        }
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
    words(&hd, sizeof(hd));
    words(phases.data(), phases.size() * sizeof(UnitPhase));
    words(A.recs.data(), A.recs.size() * sizeof(UnitRec));
    words(A.mats.data(), A.mats.size() * sizeof(float2));
    info.words = (int)hd.words;
    info.n_phases = (int)hd.n_phases;
    info.n_events = (int)hd.n_events;
    return info;
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
