"""Host-side checks of the unit sweep kernel's program assembler
(csrc/unit_program.cpp), compiled with the host compiler."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_17028_gb300", "csrc")

HEAD = r'''
#include <cmath>
#include <cstdio>
#include <cstring>
#include "fp32_round.h"
#include "small.h"
#include "unit_program.h"
#include "nqs_internal.h"
using namespace nqs;
static const int kLocal[12] = {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11};
struct Program {
    std::vector<uint4> words;
    UnitProgram info;
    UnitHeader hd;
    const UnitRec* recs;
    const float2* mats;
    Program(bool single, const std::vector<DevOp>& ops, const std::vector<float2>& table, int n_qubits) {
        info = assemble_unit(single, ops, 0, (int)ops.size(), kLocal, n_qubits, table, words);
        std::memcpy(&hd, words.data(), sizeof(hd));
        recs = reinterpret_cast<const UnitRec*>(words.data() + hd.ops_word);
        mats = reinterpret_cast<const float2*>(words.data() + hd.mats_word);
    }
};
'''


def run_host(tmp_path, body):
    cxx = shutil.which("g++")
    inc = "/usr/local/cuda/include"
    if not cxx or not os.path.isdir(inc):
        pytest.skip("no host C++ compiler or CUDA headers")
    src = tmp_path / "check.cpp"
    src.write_text(HEAD + body)
    exe = tmp_path / "check"
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-I", inc, str(src),
                    os.path.join(CSRC, "unit_program.cpp"), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


def test_checkpoint_slots_hold_any_site(tmp_path):
    """A slot names its site, counted from the program's first one, and its table
    (phi or chi) whatever the number of sites of the circuit; the other records
    with a site index do as well."""
    out = run_host(tmp_path, r'''
int main() {
    for (int from : {0, 32766, 70000})
    for (int fwd = 0; fwd < 3; ++fwd) {   // reductions and saves of phi, saves of chi
        std::vector<float2> table = {{1, 0}, {0, 0}, {0, 0}, {1, 0}};
        std::vector<DevOp> ops;
        for (int k = 0; k < 4; ++k) {
            DevOp d{};
            d.type = OP_SITE;
            d.a = d.qa = k;
            d.b = d.qb = -1;
            d.site = from + k;
            d.flags = FL_APPLY | (fwd == 0 ? FL_REDUCE | (k << 8) : fwd == 1 ? FL_SAVE : FL_SAVE_FWD);
            ops.push_back(d);
        }
        Program p(true, ops, table, 12);
        for (int k = 0; k < 4; ++k) {   // as the kernel reads it from tables that start at site_base
            const unsigned s = p.hd.slot_site[k];
            printf("%d %d\n", p.info.site_base + (int)(s & 0x7fff), (s & 0x8000) != 0);
        }
    }
    OpRec r{};
    SmallUnit u{};
    r.site = 70000;
    u.site[0] = 70000;
    printf("%lld %lld\n", (long long)r.site, (long long)u.site[0]);
}
''')
    got = [(int(a), int(b)) for a, b in zip(out[::2], out[1::2])]
    assert got[:36] == [(s + k, int(t == 2)) for s in (0, 32766, 70000) for t in range(3) for k in range(4)]
    assert got[36] == (70000, 70000)


def test_repeated_phases_keep_the_norm(tmp_path):
    """Branch groups hold a diagonal as its value at 0 and a ratio.  The ratio is
    rounded to single precision, with a modulus off 1, and a circuit repeats its
    phases: 128 equal ones must not add those errors up.  The mean of
    |factor|^2 over the amplitudes against the exact product of the matrices:
    what is left is the rounding of the one constant that takes the errors out,
    2^-24 on each part, 1.2e-7 of its square; twice that is allowed."""
    out = run_host(tmp_path, r'''
typedef std::complex<double> cdd;
static cdd f(float2 v) { return cdd(v.x, v.y); }
int main() {
    // the angle of 2000 whose rounded ratio is farthest from modulus 1
    double angle = 0, far = 0;
    for (int k = 1; k < 2000; ++k) {
        const double g = 0.001571 * k;
        const cdd q = f(round_c64(std::polar(1.0, g))) / f(round_c64(std::polar(1.0, -g)));
        const double off = std::fabs(std::abs(f(round_c64(q))) / std::abs(q) - 1.0);
        if (off > far) { far = off; angle = g; }
    }
    // 128 times the ZZ phase of tile position 8, a register bit, and qubit 12, outside the tile
    std::vector<float2> table(16, make_float2(0.f, 0.f));
    for (int k = 0; k < 4; ++k) table[5 * k] = round_c64(std::polar(1.0, k == 0 || k == 3 ? -angle : angle));
    std::vector<DevOp> ops(128);
    for (DevOp& d : ops) {
        d = DevOp{};
        d.type = OP_D2;
        d.a = d.qa = 8;
        d.b = -1;
        d.qb = 12;
        d.site = -1;
    }
    Program p(false, ops, table, 13);
    // the records as the kernel executes them, in FP64; the tile's number (qubit 12) is bit 8
    double got = 0, want = 0;
    for (int tile = 0; tile < 2; ++tile) {
        const unsigned bits = (unsigned)tile << 8;
        cdd d = 1.0, h[4] = {1.0, 1.0, 1.0, 1.0}, x[16];
        for (cdd& a : x) a = 1.0;
        for (unsigned o = 0; o < p.hd.n_ops; ++o) {
            const UnitRec& r = p.recs[o];
            const float2* const m = p.mats + r.mat;
            const int c = (bits >> r.a) & 1, c2 = (bits >> r.b) & 1;
            if (r.code == UO_SC) {
                d *= f(m[c + 2 * c2]);
            } else if (r.code >= UO_HP && r.code < UO_HP + 4) {
                h[r.code - UO_HP] *= f(m[c]);
            } else if (r.code >= UO_FLB && r.code < UO_FLB + 4) {
                for (int k = 0; k < 16; ++k)
                    if (k >> (r.code - UO_FLB) & 1) x[k] *= h[r.code - UO_FLB];
                h[r.code - UO_FLB] = 1.0;
            } else if (r.code == UO_FLS) {
                for (cdd& a : x) a *= d;
                d = 1.0;
            } else if (r.code == UO_FLA) {
                for (int k = 0; k < 16; ++k) {
                    x[k] *= d;
                    for (int i = 0; i < 4; ++i)
                        if (k >> i & 1) x[k] *= h[i];
                }
                d = h[0] = h[1] = h[2] = h[3] = 1.0;
            } else {
                printf("unexpected record %d\n", r.code);
                return 1;
            }
        }
        for (int k = 0; k < 16; ++k) {
            got += std::norm(x[k]) / 32;
            want += std::norm(std::pow(f(table[5 * (2 * (k & 1) + tile)]), 128)) / 32;
        }
    }
    printf("%.17g %.17g %d\n", far, got / want - 1.0, (int)p.info.mode);
}
''')
    far, off, mode = float(out[0]), float(out[1]), int(out[2])
    assert mode == 0 and 128 * far > 1e-6   # ratios; what adds up if nothing takes it out
    assert abs(off) <= 2.4e-7, off
