"""Branch groups and site triples where they can go wrong: test states of one
basis amplitude, a deep level whose states do not fit in the group buffers
together, and triples of sites with one or two kept factors.  Against the FP64
oracle at the tolerance of the parity tests (1e-5 of F)."""

import itertools

import numpy as np
import pytest

import workloads as W
from oracle import csim
from oracle import expansion as OEX
from oracle import ir as OIR
from oracle.statevector import basis_state

from _gpu_util import REL_TOL, compare, oracle_result, site_sets

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    yield


@pytest.mark.parametrize("n,gates,noises,level", [(12, 60, 6, 2), (13, 80, 7, 2), (14, 110, 12, 2), (16, 90, 5, 3)])
def test_basis_test_states(n, gates, noises, level):
    """v is the bit string that the circuit makes most likely, so F is one
    amplitude and not zero."""
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(750 + n, n, gates, noises, rate_lo=1e-3, rate_hi=3e-2, v_kind="ideal")
    bits = int(np.argmax(np.abs(csim.ideal_state(OIR.parse(W.to_ir_text(w)), basis_state(n, w.psi["bits"])))))
    w.v = {"kind": "basis", "bits": bits}
    ref = oracle_result(w, level)
    assert ref["F"].real > 1e-6
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    res = circ.fidelity(nqs.basis(w.psi["bits"]), nqs.basis(bits), level)
    compare(w, level, res, circ.term_values(), ref)
    circ.close()


@pytest.mark.parametrize("short", [False, True], ids=["room", "short"])
def test_states_of_several_waves(short):
    """252 states of depth 2 against the 126 that the buffer holds, and against
    nine where memory is short."""
    import torch
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(718, 18, 60, 8, rate_lo=1e-1, rate_hi=3e-1, v_kind="ideal",
                         noise_kinds=("depol", "adpd", "pd"))
    ref = oracle_result(w, 3)
    assert ref["T"][3].real > 1e-3 * ref["F"].real
    refused = []

    def alloc(nbytes, stream, ctx):
        if nbytes > (8 + 1 + 3 + 9) * (8 << 18):
            refused.append(nbytes)
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))

    def free(ptr, nbytes, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    hooks = nqs.ALLOC_FN(alloc), nqs.FREE_FN(free)
    if short:
        nqs.nqs_set_allocator(*hooks)
    try:
        circ = nqs.NoisyCircuit(W.to_ir_text(w))
        res = circ.fidelity(nqs.basis(w.psi["bits"]), nqs.ideal(), 3)
        compare(w, 3, res, circ.term_values(), ref)
        info = nqs.nqs_get_info(circ.h)
        assert info["ckpt_spacing"] == 0 and info["n_states"] == (21 if short else 8 + 1 + 24 + 126)
        assert len(refused) == int(short)
        circ.close()
    finally:
        nqs.use_torch_allocator()


@pytest.mark.parametrize("kinds,seed", [(("ad", "depol"), 92), (("adpd", "pd", "depol"), 93), (("adpd", "pd"), 94)])
def test_triples_of_sites_with_fewer_factors(kinds, seed):
    """Amplitude and phase damping keep one factor, both together two.  A term's
    amplitude is at most the product of its factors' norms, sqrt(d_i) each, and
    rounded relative to that: W(S) within 1e-5 of the product of the sites' sums
    of d_i."""
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(seed, 13, 250, 8, noise_kinds=kinds, v_kind="ideal", rate_lo=1e-1, rate_hi=3e-1)
    ref = oracle_result(w, 3)
    want = site_sets([r for r, _ in ref["terms"]], [x.real for _, x in ref["terms"]])
    d = [float(np.sum(OEX.svd_factors(z.kraus)[0][1:])) for z in w.noises]
    every = np.array(list(itertools.combinations(range(w.n_noise), 3)), dtype=np.int32)
    size = {tuple(s): d[s[0]] * d[s[1]] * d[s[2]] for s in every.tolist()}
    assert sum(want[s] > 10 * REL_TOL * size[s] for s in size) >= 8   # what is compared is there
    circ = nqs.NoisyCircuit(W.to_ir_text(w), None, nqs.NQS_PREP_PRUNE_ZERO_RANK)
    nqs.nqs_prepare_sets(circ.h, nqs.basis(w.psi["bits"]), nqs.ideal())
    rng = np.random.default_rng(seed)
    few = {}   # one third site for each pair: these meet at the second
    for s in rng.permutation(every):
        few.setdefault((int(s[0]), int(s[1])), s)
    for sets in (every, np.array(list(few.values())), rng.permutation(every)[:12], every[5:6]):
        for s, g in zip(sets.tolist(), nqs.nqs_eval_sets(circ.h, sets)):
            assert abs(g - want[tuple(s)]) <= REL_TOL * size[tuple(s)], (len(sets), s)
    circ.close()
