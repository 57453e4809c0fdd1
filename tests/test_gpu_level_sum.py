"""Per-level sums of a result against the exactly rounded sums of its own term
values (math.fsum), at term counts on both sides of the line between the
one-warp and the whole-block sums (512 terms): 9 C(11, 2) = 495 and
9 C(12, 2) = 594 level-2 terms, and a five-level expansion.  The compensated
sums are good to a few ulps of the sum: 4 * 2^-53 relative."""

import math

import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,noises,level", [(6, 11, 2), (6, 12, 2), (7, 5, 4), (13, 12, 2)])
def test_level_sums_equal_fsum_of_terms(n, noises, level):
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    w = W.random_circuit(300 + noises, n, 40, noises, rate_lo=1e-3, rate_hi=3e-2, v_kind="ideal")
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    res = circ.fidelity(nqs.basis(w.psi["bits"]), nqs.ideal(), level)
    terms = list(circ.term_values())
    circ.close()
    at = 0
    for u in range(level + 1):
        count = math.comb(noises, u) * 3 ** u
        want = math.fsum(terms[at:at + count])
        assert abs(res["T"][u] - want) <= 4 * 2.0 ** -53 * want, (u, res["T"][u], want)
        at += count
    assert at == len(terms) == res["n_terms"]
    total = math.fsum(terms)
    assert abs(res["F"] - total) <= 4 * 2.0 ** -53 * total
