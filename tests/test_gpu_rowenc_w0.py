"""dW_0 of the H = 128 encoder without dX (needs a GB300): every width of the
input, aligned rows and rows 4 bytes off, against the oracle and against the kernel
that forms dW_0 and dX together.

Tolerances: 5e-2 against the oracle, as for the other BF16 gradients. Against the
other kernel 1e-5: the same FP32 products, in sums of at most 70001 rows taken in
another order, off by 2^-24 sqrt(70001) = 1.6e-5 of the products' root sum of
squares at the worst and by a few 2^-24 in the mean."""
import numpy as np
import pytest
import torch

from oracle import model as om
from paper_2410_01657_gb300 import binding as B
from paper_2410_01657_gb300 import nn as gnn
from gpu_util import rel_l2
from test_gpu_rowmlp import DEV, _mlp_params, built  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 127, 70001])
@pytest.mark.parametrize("n_in", [4, 5, 7, 8, 9, 12, 16])
def test_encoder_h128_without_dx(n_in, rows):
    dims = [n_in, 128, 128, 128]
    P = _mlp_params(dims, True, n_in)
    rng = np.random.default_rng(rows)
    X, dY = rng.standard_normal((rows, n_in)), rng.standard_normal((rows, 128))
    _, cache = om.mlp_forward(P, X)
    ref = om.mlp_backward(P, cache, dY)[1]["W"][0]
    ts = [torch.as_tensor(t, dtype=torch.float32, device=DEV) for t in [*P["W"], *P["b"], P["gamma"], P["beta"]]]
    dYt = torch.as_tensor(dY, dtype=torch.float32, device=DEV)
    aligned = torch.as_tensor(X, dtype=torch.float32, device=DEV)
    off = torch.empty(rows * n_in + 1, device=DEV)[1:].view(rows, n_in).copy_(aligned)
    assert off.data_ptr() % 16 == 4

    def dw0(Xt, need_dx):
        params = [t.clone().requires_grad_() for t in ts]
        y = gnn.RowMLPFunction.apply(Xt, dims, True, False, 1e-5, need_dx, True, False, *params)
        g = torch.autograd.grad(y, params[0], dYt)[0]
        B.call("gnn_check", None)
        return g

    a = dw0(aligned, False)
    assert torch.equal(a, dw0(off, False))
    assert rel_l2(a.cpu().numpy(), ref) < 5e-2
    assert rel_l2(a.cpu().numpy(), dw0(aligned, True).cpu().numpy()) < 1e-5
