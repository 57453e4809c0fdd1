"""Site triples evaluated by sweeps that meet at the middle site, against the
FP64 oracle and against the forward sweeps of many triples that share a pair:
widths of one and several tiles, neighbouring sites, sites of one qubit, few
and many triples per call (one and several lanes)."""

import itertools

import numpy as np
import pytest

import workloads as W

from _gpu_util import REL_TOL, oracle_result, site_sets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,seed,gates,noise", [(12, 81, 40, 9), (13, 82, 30, 8), (15, 83, 45, 7)])
def test_triples_that_meet_in_the_middle(n, seed, gates, noise):
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    w = W.random_circuit(seed, n, gates, noise, v_kind="ideal", rate_lo=1e-3, rate_hi=3e-2)
    ref = oracle_result(w, 3)
    want = site_sets([r for r, _ in ref["terms"]], [x.real for _, x in ref["terms"]])
    F = ref["F"].real
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    nqs.nqs_prepare_sets(circ.h, nqs.basis(w.psi["bits"]), nqs.ideal())
    every = np.array(list(itertools.combinations(range(w.n_noise), 3)), dtype=np.int32)
    rng = np.random.default_rng(seed)
    # one third site for each pair of a few: all of them meet
    few = {}
    for s in rng.permutation(every):
        few.setdefault((int(s[0]), int(s[1])), s)
    for sets in (every, np.array(list(few.values())), rng.permutation(every)[:12]):
        got = nqs.nqs_eval_sets(circ.h, sets)
        for s, g in zip(sets, got):
            assert abs(g - want[tuple(int(x) for x in s)]) <= REL_TOL * abs(F), (len(sets), s)
    for s in rng.permutation(every)[:8]:   # alone
        assert abs(nqs.nqs_eval_sets(circ.h, s[None])[0] - want[tuple(int(x) for x in s)]) <= REL_TOL * abs(F), s
    circ.close()
