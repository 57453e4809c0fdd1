"""Loss and gradient of the proposal network where its tiles have edges (one
row, ragged widths and batches, scalar and vector loads, one and many partial
products, several groups of rows per block of the output layer) against FP64.

Every fp32 operand of a product enters as two bf16 parts, within 2^-17 of its
size; at most 2 (layers + 1) = 8 such products follow one another, and the sum
of the products' sizes is at most a few times the largest result: 8 * 4 * 2^-17
= 2^-12 at the very worst, 1e-4 of the largest entry as errors add at random.
Rows with a ReLU input next to its kink are left out of the data."""

import numpy as np
import pytest

from oracle import mlp as OM

pytestmark = pytest.mark.gpu


def _rows(rng, params, dims, B):
    X = rng.normal(size=(2 * B + 8, dims[0])).astype(np.float32)
    clear = np.ones(len(X), dtype=bool)
    h = X.astype(np.float64)
    for W, b in OM.unflatten(params, dims)[:-1]:
        z = h @ OM.to_bf16(W).T + b
        clear &= (np.abs(z) >= 1e-5 * np.abs(z).max()).all(axis=1)
        h = np.maximum(z, 0.0)
    assert clear.sum() >= B
    return X[clear][:B]


@pytest.mark.parametrize("n_in,hidden,layers,B,shift", [
    (8, 256, 3, 1, 0),
    (8, 256, 3, 1025, 0),
    (8, 256, 3, 1024, 1),       # inputs that are not 16-byte aligned
    (1, 1, 1, 2, 0),
    (3, 5, 1, 17, 0),
    (33, 40, 2, 300, 0),
    (4, 100, 8, 65, 0),
    (8, 64, 1, 4999, 0),        # 32 rows per block of the output layer
])
def test_loss_and_gradient_at_the_edges(n_in, hidden, layers, B, shift):
    import torch
    from paper_2211_17028_gb300 import nqs
    nqs.use_torch_allocator()
    rng = np.random.default_rng([n_in, hidden, B])
    m = nqs.nqs_mlp_create(n_in, hidden, layers, seed=5)
    dims = [n_in] + [hidden] * layers + [1]
    params = nqs.nqs_mlp_get_params(m)
    params += rng.normal(size=params.size).astype(np.float32) * 0.02   # biases too
    nqs.nqs_mlp_set_params(m, params)
    # a larger batch first: the partial products are then laid out anew
    X = _rows(rng, params, dims, B)
    y = np.cos(X).sum(axis=1).astype(np.float32)
    buf = torch.zeros(B * n_in + shift, device="cuda")
    Xd = buf[shift:].view(B, n_in)
    Xd.copy_(torch.from_numpy(X))
    yd = torch.from_numpy(y).cuda()
    nqs.nqs_mlp_loss_grad(m, torch.zeros(B + 130, n_in, device="cuda"), torch.zeros(B + 130, device="cuda"))
    loss, g = nqs.nqs_mlp_loss_grad(m, Xd, yd)
    lo, go = OM.loss_and_grad(params, dims, X, y)
    assert abs(loss - lo) <= 1e-4 * lo
    assert np.abs(g - go).max() <= 1e-4 * np.abs(go).max()
    out = torch.zeros(B, device="cuda")
    nqs.nqs_mlp_forward(m, Xd, out)
    want = OM.forward(params, dims, X)[-1][:, 0]
    assert np.abs(out.cpu().numpy() - want).max() <= 1e-4 * max(np.abs(want).max(), 1e-3)
    nqs.nqs_mlp_destroy(m)
