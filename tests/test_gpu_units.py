"""Unit sweep launches (one state per block, all branch groups of a wave in one
launch per pass) at the sizes where they can go wrong: one tile and two tiles
of a 12-qubit tile, a level whose children do not fit in one wave, pruned
factors (groups of fewer than three states), passes with several spawning
sites, and two-qubit gates, diagonals and sites on register, thread and
outer qubits.  Against the FP64 oracle at the tolerance of the parity tests
(1e-5 of F), and bit for bit against the same call again."""

import numpy as np
import pytest

import workloads as W
from oracle import expansion as OEX
from oracle import ir as OIR

from _gpu_util import compare, oracle_result

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    yield


# n, gates, noises, level, v: 12 qubits is a single tile, 13 two; 9 noises at
# level 3 make 324 depth-2 states; 40 noises put four sites into a pass
@pytest.mark.parametrize("n,gates,noises,level,v", [
    (12, 60, 6, 2, "basis"), (12, 90, 4, 4, "ideal"), (13, 70, 9, 3, "ideal"), (13, 150, 40, 1, "dense"),
    (14, 110, 20, 2, "ideal"), (15, 60, 3, 3, "dense")])
def test_unit_sweeps_match_oracle(n, gates, noises, level, v):
    from paper_2211_17028_gb300 import nqs
    from _gpu_util import gpu_state
    w = W.random_circuit(700 + n + noises, n, gates, noises, rate_lo=1e-3, rate_hi=3e-2, v_kind=v)
    ref = oracle_result(w, level)
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    psi, keep1 = gpu_state(w.psi, w.n)
    vs, keep2 = gpu_state(w.v, w.n)
    res = circ.fidelity(psi, vs, level)
    terms = circ.term_values()
    if ref["F"].real > 0:
        compare(w, level, res, terms, ref)
    again = circ.fidelity(psi, vs, level)
    assert again["F"] == res["F"] and np.array_equal(circ.term_values(), terms)
    circ.close()


@pytest.mark.parametrize("noises", [3, 7])
def test_pruned_factors_leave_smaller_groups(noises):
    """Amplitude damping has one non-dominant factor of nonzero weight: with
    NQS_PREP_PRUNE_ZERO_RANK a branch group holds one state."""
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(800 + noises, 13, 60, noises, noise_kinds=("ad",), v_kind="ideal")
    full = nqs.NoisyCircuit(W.to_ir_text(w))
    pruned = nqs.NoisyCircuit(W.to_ir_text(w), None, nqs.NQS_PREP_PRUNE_ZERO_RANK)
    psi = nqs.basis(w.psi["bits"])
    a, b = full.fidelity(psi, nqs.ideal(), 2), pruned.fidelity(psi, nqs.ideal(), 2)
    assert b["n_terms"] < a["n_terms"]
    for u in range(3):
        assert abs(a["T"][u] - b["T"][u]) <= 1e-5 * a["F"]
    ref = OEX.approximate(OIR.parse(W.to_ir_text(w)), w.psi, w.v, 2) if w.n <= 10 else oracle_result(w, 2, False)
    assert abs(b["F"] - ref["F"].real) <= 1e-5 * ref["F"].real
    full.close()
    pruned.close()
