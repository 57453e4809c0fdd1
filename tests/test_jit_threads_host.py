"""The cache of generated kernels with several threads (no device needed): a
thread that wants a kernel which another one is compiling waits for it."""

import threading

import workloads as W


def test_two_handles_want_the_same_kernels_at_once():
    from paper_2211_17028_gb300 import nqs
    w = W.random_circuit(641, 14, 60, 4, v_kind="ideal")
    circs = [nqs.NoisyCircuit(W.to_ir_text(w)) for _ in range(2)]
    start, got = threading.Barrier(2), [None, None]

    def check(i):
        start.wait()
        try:
            got[i] = nqs.nqs_jit_compile_check(circs[i].h, 1, 2)
        except nqs.NqsError as e:
            got[i] = e.code

    threads = [threading.Thread(target=check, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for c in circs:
        c.close()
    # passes of the forward sweep and of the backward one, at most two each
    assert got[0] == got[1] and 2 <= got[0] <= 4, got
