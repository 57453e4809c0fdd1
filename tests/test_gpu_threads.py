"""Two handles on two threads: what one call sets for its own launches must not
reach the launches of another.  The calls have different needs of shared
memory (13 and 14 qubits of general noises; unit programs of different
lengths) or want the same generated kernels at the same time."""

import ctypes
import threading

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
    torch.cuda.synchronize()


def _general(n):
    w = W.random_circuit(600 + n, n, 8, 0, v_kind="ideal")
    w.noises = [Noise(3, 0, ch.depolarizing2(0.02), "", 1), Noise(6, 1, ch.depolarizing2(0.03), "", 2)]
    return w, 1


def _units(n):
    # many operations and sites to a pass against a single one of each
    if n == 13:
        return W.random_circuit(613, 13, 300, 30, v_kind="ideal"), 1
    return W.random_circuit(612, 12, 2, 1, v_kind="ideal"), 1


@pytest.mark.parametrize("make,widths", [(_general, (13, 14)), (_units, (12, 13))], ids=["general", "units"])
def test_two_threads_do_not_disturb_each_other(make, widths):
    import torch
    from paper_2211_17028_gb300 import nqs
    work = []
    for n in widths:
        w, level = make(n)
        circ = nqs.NoisyCircuit(W.to_ir_text(w))
        psi = nqs.basis(w.psi["bits"])
        work.append((circ, psi, level, circ.fidelity(psi, nqs.ideal(), level)["F"]))
    failed = []

    def calls(circ, psi, level, F):
        # the result goes to pinned memory: nothing between two calls waits for the GPU
        stream = torch.cuda.Stream()
        pinned = torch.zeros(ctypes.sizeof(nqs.nqs_result), dtype=torch.uint8, pin_memory=True)
        out = nqs.nqs_result.from_address(pinned.data_ptr())
        for k in range(4000):
            try:
                nqs.nqs_fidelity(circ.h, psi, nqs.ideal(), level, stream, out=out)
            except nqs.NqsError as e:
                failed.append(e.code)
            if k % 100 == 99:
                stream.synchronize()
                if out.status != 0 or out.F != F:
                    failed.append((out.status, out.F, F))

    threads = [threading.Thread(target=calls, args=a) for a in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, (len(failed), failed[:4])
    for a in work:
        a[0].close()


def test_generated_kernels_wanted_by_two_threads_at_once():
    """The second thread waits for the kernels that the first one compiles."""
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(640, 14, 60, 4, v_kind="ideal")
    circs = [nqs.NoisyCircuit(W.to_ir_text(w)) for _ in range(2)]
    psi = nqs.basis(w.psi["bits"])
    start = threading.Barrier(2)
    got = [None, None]

    def call(i):
        nqs.nqs_set_option(circs[i].h, nqs.NQS_OPT_JIT, 1)
        start.wait()
        F = circs[i].fidelity(psi, nqs.ideal(), 2)["F"]
        got[i] = (F, nqs.nqs_get_info(circs[i].h)["jit_state"])

    threads = [threading.Thread(target=call, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert got[0] == got[1] and got[0][1] == 1, got
    for c in circs:
        c.close()
