"""Circuits narrower than a sweep tile (two launches, one block per prefix of
insertions) at the sizes where they can go wrong: one and two qubits, the
widest (11), one noise, more than 32 later sites (terms are written out in
chunks of 32 reductions), operation lists around the chunk of 32 operations,
deep levels, dense states, pruned factors and shards.  Against the FP64 oracle
at the tolerance of the parity tests (1e-5 of F)."""

import numpy as np
import pytest

import workloads as W

from _gpu_util import compare, gpu_state, oracle_result

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    yield


@pytest.mark.parametrize("n,gates,noises,level,v", [
    (1, 6, 3, 3, "ideal"), (2, 31, 1, 1, "dense"), (3, 32, 4, 4, "ideal"), (5, 33, 5, 4, "ideal"),
    (7, 64, 6, 3, "dense"), (11, 90, 36, 2, "ideal"), (11, 40, 7, 3, "dense"), (9, 20, 8, 0, "ideal")])
def test_small_circuits_match_oracle(n, gates, noises, level, v):
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(900 + n + noises, n, gates, noises, rate_lo=1e-3, rate_hi=3e-2, v_kind=v)
    ref = oracle_result(w, level)
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    psi, keep1 = gpu_state(w.psi, w.n)
    vs, keep2 = gpu_state(w.v, w.n)
    res = circ.fidelity(psi, vs, level)
    terms = circ.term_values()
    assert [l["kind"] for l in nqs.nqs_schedule_launches(circ.h)] == ["small", "sum"]
    compare(w, level, res, terms, ref)
    again = circ.fidelity(psi, vs, level)
    assert again["F"] == res["F"] and np.array_equal(circ.term_values(), terms)
    circ.close()


@pytest.mark.parametrize("n,noises", [(6, 5), (10, 9)])
def test_small_pruned_and_sharded(n, noises):
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(950 + n, n, 50, noises, noise_kinds=("ad", "depol"), v_kind="ideal")
    psi = nqs.basis(w.psi["bits"])
    full = nqs.NoisyCircuit(W.to_ir_text(w))
    a = full.fidelity(psi, nqs.ideal(), 3)
    full.close()
    pruned = nqs.NoisyCircuit(W.to_ir_text(w), None, nqs.NQS_PREP_PRUNE_ZERO_RANK)
    b = pruned.fidelity(psi, nqs.ideal(), 3)
    parts = []
    for r in range(3):
        nqs.nqs_set_option(pruned.h, nqs.NQS_OPT_SHARD_COUNT, 3)
        nqs.nqs_set_option(pruned.h, nqs.NQS_OPT_SHARD_RANK, r)
        parts.append(pruned.fidelity(psi, nqs.ideal(), 3)["T"])
    pruned.close()
    T, F = nqs.merge_level_sums(parts)
    assert b["n_terms"] <= a["n_terms"]
    for u in range(4):
        assert abs(a["T"][u] - b["T"][u]) <= 1e-5 * a["F"]
        assert abs(T[u] - b["T"][u]) <= 1e-14 * b["F"]
