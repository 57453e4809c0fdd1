"""General noises on both sides of the line between whole states on chip (at
most 14 qubits) and one launch per gate over all siblings, against the FP64
oracle O3: the smallest widths, the line itself, levels that spawn twice, and
the same handle at one level after another.  Tolerance of the general-noise
tests: 1e-5 of F on F and on every site-set sum."""

import pytest

import workloads as W
from workloads import channels as ch
from workloads.circuits import Noise
from oracle import ir as OIR
from oracle import o3 as O3

from test_gpu_general_noise import REL, _site_sets

pytestmark = pytest.mark.gpu


def _workload(n, gates, noises):
    rng = W.SplitMix64(500 + n)
    w = W.random_circuit(500 + n, n, gates, 0, v_kind="ideal")
    w.noises = []
    for k in range(noises):
        q = rng.randbelow(n)
        at = (k + 1) * gates // (noises + 1)
        if n > 1 and k % 2 == 0:
            p = (q + 1 + rng.randbelow(n - 1)) % n
            w.noises.append(Noise(at, q, ch.depolarizing2(0.02 + 0.01 * k), "", p))
        else:   # two factor sets: the matrix is not positive semidefinite
            w.noises.append(Noise(at, q, [], "", -1, ch.perturbed_superop(rng, ch.amplitude_damping(0.04), 0.01)))
    return w


@pytest.mark.parametrize("n,gates,noises,levels", [
    (1, 6, 3, (3, 1)), (2, 12, 3, (2, 0)), (13, 40, 3, (2, 3)), (14, 50, 3, (1, 2)), (15, 40, 3, (2, 3, 1))])
def test_general_noise_matches_o3(n, gates, noises, levels):
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    w = _workload(n, gates, noises)
    c = OIR.parse(W.to_ir_text(w))
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    for level in levels:
        ref = O3.approximate(c, w.psi, w.v, level)
        res = circ.fidelity(nqs.basis(w.psi["bits"]), nqs.ideal(), level)
        vals = circ.term_values()
        F = ref["F"].real
        assert res["n_terms"] == len(vals)
        assert abs(res["F"] - F) <= REL * abs(F)
        got, want = _site_sets(c, level, vals), _site_sets(c, level, ref["terms"].real)
        assert max(abs(got[k] - want[k]) for k in want) <= REL * abs(F)
    circ.close()
