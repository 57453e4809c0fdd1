"""The two forms of the unit kernel (two blocks per SM for launches that do not
fill the chip, three for those that do) and records that hold the gates of
several register bits: launches just below and above the line, layers of gates
with signs, phases and controlled phases between them, both directions.
Against the FP64 oracle at the tolerance of the parity tests (1e-5 of F), and
bit for bit against the same call again."""

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


# tiles of the widest launch: 2^(n - 12) x 3 per noise; 304 blocks are two per SM
@pytest.mark.parametrize("n,gates,noises,v", [(15, 90, 12, "ideal"), (16, 100, 6, "ideal"), (16, 100, 7, "dense"),
                                              (17, 120, 8, "ideal"), (18, 140, 5, "dense")])
def test_forms_match_oracle(n, gates, noises, v):
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(900 + n + noises, n, gates, noises, v_kind=v)
    ref = oracle_result(w, 2)
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    psi, keep1 = gpu_state(w.psi, n)
    vs, keep2 = gpu_state(w.v, n)
    res = circ.fidelity(psi, vs, 2)
    terms = circ.term_values()
    compare(w, 2, res, terms, ref)
    again = circ.fidelity(psi, vs, 2)
    assert again["F"] == res["F"] and np.array_equal(circ.term_values(), terms)
    circ.close()
