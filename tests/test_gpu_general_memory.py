"""General noises on more than 14 qubits (one launch per gate over all siblings):
the lifetime of a call's uploads, and calls that are short of memory."""

import ctypes

import pytest

import workloads as W
from workloads import channels as ch
from workloads.circuits import Noise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    yield


def _workload():
    w = W.random_circuit(615, 15, 40, 0, v_kind="ideal")
    w.noises = [Noise(9, 0, ch.depolarizing2(0.02), "", 1), Noise(19, 3, ch.depolarizing2(0.03), "", 2),
                Noise(29, 1, ch.depolarizing2(0.04), "", 4)]
    return w


def test_uploads_are_read_before_the_call_returns():
    """With a pinned result nothing at the end of a call waits for the stream;
    its tables come from host memory that is gone when the call returns."""
    import torch
    from paper_2211_17028_gb300 import nqs
    w = _workload()
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    psi = nqs.basis(w.psi["bits"])
    want = circ.fidelity(psi, nqs.ideal(), 2)
    pinned = torch.zeros(ctypes.sizeof(nqs.nqs_result), dtype=torch.uint8, pin_memory=True)
    out = nqs.nqs_result.from_address(pinned.data_ptr())
    side, reached = torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(side):
        torch.cuda._sleep(200_000_000)   # about 100 ms ahead of the uploads
        reached.record()
    nqs.nqs_fidelity(circ.h, psi, nqs.ideal(), 2, side, out=out)
    assert reached.query()
    side.synchronize()
    assert out.F == want["F"] and out.status == 0
    circ.close()


def test_one_sibling_where_fifteen_do_not_fit():
    """N + level + 3 states of 256 KiB fit, the siblings' 15 per depth do not."""
    import torch
    from paper_2211_17028_gb300 import nqs
    w = _workload()
    text, psi = W.to_ir_text(w), nqs.basis(w.psi["bits"])
    circ = nqs.NoisyCircuit(text)
    want = circ.fidelity(psi, nqs.ideal(), 2)
    terms = circ.term_values()
    circ.close()
    refused = []

    def alloc(nbytes, stream, ctx):
        if nbytes > (3 + 2 + 3) * (8 << 15):
            refused.append(nbytes)
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))

    def free(ptr, nbytes, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    hooks = nqs.ALLOC_FN(alloc), nqs.FREE_FN(free)
    nqs.nqs_set_allocator(*hooks)
    try:
        circ = nqs.NoisyCircuit(text)
        got = circ.fidelity(psi, nqs.ideal(), 2)
        assert refused and got["F"] == want["F"] and got["T"] == want["T"]
        assert list(circ.term_values()) == list(terms)
        asked = len(refused)   # the next call keeps what it has
        assert circ.fidelity(psi, nqs.ideal(), 2)["F"] == want["F"] and len(refused) == asked
        circ.close()
    finally:
        nqs.use_torch_allocator()
