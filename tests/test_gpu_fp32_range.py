"""The FP32 path over the whole range of FP32 numbers (needs a GB300): infinities,
NaN, numbers near the largest and the smallest, in inputs, upstream gradients and
weights, against the same MLP in 64 bits.

Where 64 bits give a NaN or an infinity (or a number above FP32's largest), FP32
has to give the same; every other value is within 1e-5 of the row's norm (the
bound of the FP32 path at ordinary sizes: rounding is relative, so a power of two in
front of the inputs changes nothing as long as results are normal numbers), a
gradient that cancels over its n rows within 1e-5 of sqrt(n), the size of a sum of n
numbers near 1 of either sign. Rows beside a special one keep their bits. The
gradients of a NaN row are not compared (ELU' of a NaN is a NaN here and 1 in
PyTorch)."""
import ctypes as C

import pytest
import torch

from paper_2410_01657_gb300 import binding as B
from paper_2410_01657_gb300 import nn as gnn
from test_gpu_lin3 import DEV, built  # noqa: F401

pytestmark = pytest.mark.gpu
DIMS = [[1, 1, 1], [5, 20, 20, 3], [64, 64, 64], [64, 64, 64, 64], [100, 128, 70], [128, 128, 9]]
INF, NAN, MAX = float("inf"), float("nan"), 3.4028234e38


def _weights(dims, g):
    n = len(dims) - 1
    W = [(torch.rand(dims[k + 1], dims[k], device=DEV, generator=g) + 0.5) / dims[k] for k in range(n)]   # all positive
    return W + [0.1 * torch.randn(dims[k + 1], device=DEV, generator=g) for k in range(n)]


def _run(dims, ts, X, dY):
    rows = X.shape[0]
    d = [torch.zeros_like(t) for t in ts]
    S, dS = gnn.mlp_struct(dims, ts, False), gnn.mlp_struct(dims, d, False)
    f, b = C.c_size_t(), C.c_size_t()
    B.call("gnn_mlp_workspace_size", C.byref(S), rows, C.byref(f), C.byref(b))
    ws = gnn.workspace(max(f.value, b.value), DEV)
    Y, dX = torch.empty(rows, dims[-1], device=DEV), torch.empty_like(X)
    B.call("gnn_mlp_forward", C.byref(S), rows, B.ptr(X), B.ptr(Y), 0, 1e-5, B.ptr(ws), ws.numel(), None)
    B.call("gnn_mlp_backward", C.byref(S), rows, B.ptr(X), B.ptr(dY), 0, B.ptr(dX), C.byref(dS), 1e-5, B.ptr(ws),
           ws.numel(), None)
    B.call("gnn_check", None)
    return Y, dX, d


def _ref(dims, ts, X, dY):
    n = len(dims) - 1
    p = [t.double().requires_grad_() for t in ts]
    x = X.double().requires_grad_()
    z = x
    for k in range(n):
        z = torch.nn.functional.linear(z if k == 0 else torch.nn.functional.elu(z), p[k], p[n + k])
    dx, *dp = torch.autograd.grad(z, [x, *p], dY.double())
    return z.detach(), dx, dp


def _close(a, r, dim=1, least=0.0):
    """Equal special values; the rest within 1e-5 of the row's norm, or of `least`."""
    big = r.abs() > MAX
    r = torch.where(big, r.sign() * INF, r)
    assert torch.equal(torch.isnan(a), torch.isnan(r))
    inf = torch.isinf(r)
    assert torch.equal(torch.isinf(a), inf) and bool((a[inf].double() == r[inf]).all())
    ok = torch.isfinite(r)
    err = torch.where(ok, (a.double() - r).abs(), 0.0)
    norm = torch.where(ok, r, 0.0).norm(dim=dim, keepdim=True)
    assert bool((err <= 1e-5 * norm.clamp_min(least)).all())


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("value", [-INF, INF, NAN, -MAX, MAX, 1e30])
def test_special_rows(dims, value):
    if abs(value) == MAX and dims[0] == 1:
        pytest.skip("a weight above 1 takes the largest number out of range half way")
    rows, at = 300, [3, 130, 299] if abs(value) > MAX or value != value else [130]
    g = torch.Generator(device=DEV).manual_seed(1)
    ts = _weights(dims, g)
    X, dY = torch.randn(rows, dims[0], device=DEV, generator=g), torch.randn(rows, dims[-1], device=DEV, generator=g)
    Y0, dX0, _ = _run(dims, ts, X, dY)
    X[at, 0] = value
    Y, dX, d = _run(dims, ts, X, dY)
    Yr, dXr, dr = _ref(dims, ts, X, dY)
    _close(Y, Yr)
    keep = torch.ones(rows, dtype=torch.bool, device=DEV)
    keep[at] = False
    assert torch.equal(Y[keep], Y0[keep]) and torch.equal(dX[keep], dX0[keep])
    if value == value:
        _close(dX, dXr)
        for a, r in zip(d, dr):
            _close(a.view(a.shape[0], -1), r.view(r.shape[0], -1), dim=0, least=rows ** 0.5)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("value", [-INF, MAX, 1e30])
def test_special_upstream_gradient(dims, value):
    if value == MAX and dims[0] == 1:
        pytest.skip("a weight above 1 takes the largest number out of range half way")
    rows = 200
    g = torch.Generator(device=DEV).manual_seed(2)
    ts = _weights(dims, g)
    X, dY = torch.randn(rows, dims[0], device=DEV, generator=g), torch.randn(rows, dims[-1], device=DEV, generator=g)
    dY[17, 0] = value
    _, dX, d = _run(dims, ts, X, dY)
    _, dXr, dr = _ref(dims, ts, X, dY)
    _close(dX, dXr)
    n = len(dims) - 1
    for k in range(n):
        _close(d[k].reshape(1, -1), dr[k].reshape(1, -1), least=rows ** 0.5)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("power", [-140, -126, -116, -100, 100, 120])
def test_scaled_inputs(dims, power):
    # X (then W_0) times 2^power and W_0 (then X) times 2^-100 of it: no digit of the small operand is lost
    rows = 300
    g = torch.Generator(device=DEV).manual_seed(3)
    ts = _weights(dims, g)
    X, dY = torch.randn(rows, dims[0], device=DEV, generator=g), torch.randn(rows, dims[-1], device=DEV, generator=g)
    up = 2.0 ** (-power if abs(power) <= 120 else 120)
    for swap in (False, True):
        tt = [t.clone() for t in ts]
        x = X.clone()
        (tt[0] if swap else x).mul_(2.0 ** power)
        (x if swap else tt[0]).mul_(up)
        Y, dX, d = _run(dims, tt, x, dY)
        Yr, dXr, dr = _ref(dims, tt, x, dY)
        _close(Y, Yr)
        for a, r in zip([dX, *d], [dXr, *dr]):
            a, r = a.reshape(1, -1), r.reshape(1, -1)
            if 2.0 ** -126 < float(r.abs().max()) < 2.0 ** 126 and r.numel() > 1:   # (one number may have cancelled)
                _close(a, r)
