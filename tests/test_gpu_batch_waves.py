"""A batch whose circuits do not fit in memory together: waves of circuits, each
with the schedule that it has on its own, so the results are those of the plain
path bit for bit, in the first call and in later ones."""

import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_waves_give_the_plain_results():
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    ws = [W.random_circuit(960 + i, 15, 70, 8 + i % 3, v_kind="ideal") for i in range(10)]
    texts, psis = [W.to_ir_text(w) for w in ws], [nqs.basis(w.psi["bits"]) for w in ws]
    n, vs, levels = len(ws), [nqs.ideal()] * len(ws), [1 + (i % 4 > 0) for i in range(len(ws))]
    plain, states = [], []
    for t, p, l in zip(texts, psis, levels):
        c = nqs.NoisyCircuit(t)
        plain.append(c.fidelity(p, nqs.ideal(), l))
        states.append(nqs.nqs_get_info(c.h)["n_states"] * (8 << 15))
        c.close()
    room, least = 3 * max(states), min(s for s, l in zip(states, levels) if l == 2)
    held, refused = {}, []

    def alloc(nbytes, stream, ctx):   # room for the states of about three circuits
        if nbytes >= least and sum(held.values()) + nbytes > room:
            refused.append(nbytes)
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))
        if nbytes >= least:
            held[p] = nbytes
        return p

    def free(ptr, nbytes, stream, ctx):
        held.pop(int(ptr), None)
        torch.cuda.caching_allocator_delete(int(ptr))

    hooks = nqs.ALLOC_FN(alloc), nqs.FREE_FN(free)
    nqs.nqs_set_allocator(*hooks)
    try:
        circs = [nqs.NoisyCircuit(t) for t in texts]
        for call in range(2):
            outs = nqs.nqs_batch_fidelity([c.h for c in circs], psis, vs, levels)
            for k in range(n):
                got = outs[k].to_dict()
                assert got["F"] == plain[k]["F"] and got["T"] == plain[k]["T"], (call, k)
        assert len(refused) >= 2
        # a wave's buffers are given back for the next one, the term values with them
        with pytest.raises(nqs.NqsError) as e:
            circs[0].term_values()
        assert e.value.code == nqs.NQS_ERR_ORDER
        for c in circs:
            c.close()
    finally:
        nqs.use_torch_allocator()
