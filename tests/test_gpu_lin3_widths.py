"""The FP32 path's Linears at the widths where the number of accumulators changes:
three sums up to 80 (weight gradients and the adjoint chain: 64), two above
(needs a GB300). The reference is the same MLP in 64 bits; tolerance 1e-5
relative L2, as for the other widths: K <= 96 inputs and three layers in FP32
are off by sqrt(K) 2^-24 per layer, below 2e-6."""
import pytest
import torch

from gpu_util import rel_l2
from test_gpu_lin3 import DEV, TOL, _mlp64, _params, _run, built  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [[64, 63, 64, 64], [66, 65, 65], [79, 80, 80], [80, 81, 96, 80], [96, 17, 81]])
@pytest.mark.parametrize("rows", [127, 152 * 128 * 2 + 1])
def test_widths(dims, rows):
    P = _params(dims, True, 11)
    g = torch.Generator(device=DEV).manual_seed(rows)
    X = torch.randn(rows, dims[0], device=DEV, generator=g)
    dY = torch.randn(rows, dims[-1], device=DEV, generator=g)
    y, dx, dw = _run(P, dims, True, X, dY)
    Xd = X.double().requires_grad_()
    yr, ps = _mlp64(P, Xd)
    dxr, *dwr = torch.autograd.grad(yr, [Xd, *ps], dY.double())
    assert rel_l2(y.cpu().numpy(), yr.detach().cpu().numpy()) < TOL
    assert rel_l2(dx.cpu().numpy(), dxr.cpu().numpy()) < TOL
    for k, (a, r) in enumerate(zip(dw, dwr)):
        err = float((a.double() - r).norm() / max(float(r.norm()), 1e-3 * rows ** 0.5))
        assert err < TOL, k
