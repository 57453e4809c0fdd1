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
    """A slot names its site and its table (phi or chi) whatever the number of
    sites of the circuit; the other records with a site index do as well."""
    out = run_host(tmp_path, r'''
int main() {
    const int sites[4] = {5, 32768, 40000, 70000};
    for (int fwd = 0; fwd < 3; ++fwd) {   // reductions and saves of phi, saves of chi
        std::vector<float2> table = {{1, 0}, {0, 0}, {0, 0}, {1, 0}};
        std::vector<DevOp> ops;
        for (int k = 0; k < 4; ++k) {
            DevOp d{};
            d.type = OP_SITE;
            d.a = d.qa = k;
            d.b = d.qb = -1;
            d.site = sites[k];
            d.flags = FL_APPLY | (fwd == 0 ? FL_REDUCE | (k << 8) : fwd == 1 ? FL_SAVE : FL_SAVE_FWD);
            ops.push_back(d);
        }
        Program p(true, ops, table, 12);
        for (int k = 0; k < 4; ++k) {   // as the kernel reads it: the top bit selects the table
            const auto s = p.hd.slot_site[k];
            const auto top = (decltype(s))(1ull << (8 * sizeof(s) - 1));
            printf("%lld %d\n", (long long)(s & (decltype(s))~top), (s & top) != 0);
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
    sites = [5, 32768, 40000, 70000]
    assert got[:12] == [(s, int(t == 2)) for t in range(3) for s in sites]
    assert got[12] == (70000, 70000)
