"""What a handle holds beside its checkpoints: hundreds of handles of a study
live side by side, so branch groups are held together only as far as that
fills the chip, and wide ones only while the device is free."""

import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,level,full,most", [(20, 2, False, 36), (20, 3, False, 96), (23, 2, False, 12), (23, 2, True, 3)])
def test_states_held_for_branch_groups(n, level, full, most):
    """At most 256 MiB per depth or the children of one pass; on a device that is
    half full, three states of 64 MiB at a time."""
    import torch
    from paper_2211_17028_gb300 import nqs
    torch.cuda.set_device(0)
    nqs.use_torch_allocator()
    torch.cuda.empty_cache()
    other = torch.empty(torch.cuda.mem_get_info()[1] * 11 // 20 if full else 1, dtype=torch.uint8, device="cuda")
    w = W.random_circuit(900 + n, n, 60, 12, v_kind="ideal")
    circ = nqs.NoisyCircuit(W.to_ir_text(w))
    assert circ.fidelity(nqs.basis(w.psi["bits"]), nqs.ideal(), level)["status"] == 0
    info = nqs.nqs_get_info(circ.h)
    assert info["ckpt_spacing"] == 0
    assert info["n_states"] <= w.n_noise + 1 + most
    # tables, programs, partial sums and term values
    assert info["workspace_bytes"] - info["n_states"] * (8 << n) <= 24 << 20
    circ.close()
    del other
    torch.cuda.empty_cache()
