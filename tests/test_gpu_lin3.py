"""The FP32 path's tensor-core Linears (lin3.cu) against 64 bits, at the sizes
where tiles, pieces of rows and 16-byte accesses have their edges (needs a GB300).

Tolerance 1e-5 relative L2, the FP32 path's bound against the FP64 oracle: a
Linear of K <= 256 inputs in FP32 is off by at most (K + 8) 2^-24 = 1.6e-5 of
sum |x||w|, in the mean by sqrt(K) 2^-24 = 1e-6 of the result, and a chain of
seven such layers with LayerNorm stays below 1e-5."""
import ctypes as C

import numpy as np
import pytest
import torch

import synthetic as syn
from oracle import model as om
from paper_2410_01657_gb300 import _build
from paper_2410_01657_gb300 import binding as B
from paper_2410_01657_gb300 import nn as gnn
from paper_2410_01657_gb300.graph import MeshGraph

from gpu_util import oracle_subgraphs, rel_l2, split_edges, split_rows

pytestmark = pytest.mark.gpu
DEV = "cuda"
TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()
    B.load()


def _params(dims, has_ln, seed):
    return syn.xavier_mlp(np.random.default_rng(seed), dims, has_ln, randomize_affine=True)


def _mlp64(P, X):
    W = [torch.tensor(w, dtype=torch.float32, device=DEV).double().requires_grad_() for w in P["W"]]
    b = [torch.tensor(v, dtype=torch.float32, device=DEV).double().requires_grad_() for v in P["b"]]
    ln = [torch.tensor(P[k], dtype=torch.float32, device=DEV).double().requires_grad_() for k in ("gamma", "beta") if k in P]
    z = X
    for k in range(len(W)):
        z = torch.nn.functional.linear(z if k == 0 else torch.nn.functional.elu(z), W[k], b[k])
    y = torch.nn.functional.layer_norm(z, z.shape[1:], ln[0], ln[1], 1e-5) if ln else z
    return y, W + b + ln


def _run(P, dims, has_ln, X, dY):
    ts = [torch.as_tensor(t, dtype=torch.float32, device=DEV).requires_grad_()
          for t in [*P["W"], *P["b"]] + ([P["gamma"], P["beta"]] if has_ln else [])]
    Xr = X.clone().requires_grad_()
    y = gnn.RowMLPFunction.apply(Xr, dims, has_ln, False, 1e-5, True, False, False, *ts)
    dx, *dw = torch.autograd.grad(y, [Xr, *ts], dY)
    B.call("gnn_check", None)
    return y.detach(), dx, dw


@pytest.mark.parametrize("dims,has_ln", [
    ([1, 1, 1], False), ([3, 5, 5, 9], True), ([4, 16, 16, 16], True), ([17, 33, 30, 2], False), ([32, 64, 64, 3], False),
    ([64, 64, 64], True), ([65, 100, 100, 100], True), ([128, 128, 128, 128], True), ([128, 128, 128, 128, 128, 7], False)])
@pytest.mark.parametrize("rows", [1, 31, 128, 129, 152 * 128 * 3 + 65])
def test_row_mlp_matches_64_bits(dims, has_ln, rows):
    P = _params(dims, has_ln, 3)
    g = torch.Generator(device=DEV).manual_seed(rows)
    X = torch.randn(rows, dims[0], device=DEV, generator=g)
    dY = torch.randn(rows, dims[-1], device=DEV, generator=g)
    y, dx, dw = _run(P, dims, has_ln, X, dY)
    Xd = X.double().requires_grad_()
    yr, ps = _mlp64(P, Xd)
    dxr, *dwr = torch.autograd.grad(yr, [Xd, *ps], dY.double())
    assert rel_l2(y.cpu().numpy(), yr.detach().cpu().numpy()) < TOL
    assert rel_l2(dx.cpu().numpy(), dxr.cpu().numpy()) < TOL
    for k, (a, r) in enumerate(zip(dw, dwr)):
        # a gradient that cancels over the rows is held to the sum's scale
        err = float((a.double() - r).norm() / max(float(r.norm()), 1e-3 * rows ** 0.5))
        assert err < TOL, k


def test_unaligned_rows_and_pieces():
    # X and dY start 4 bytes off a 16-byte boundary: the scalar accesses give the same bits as the wide ones
    dims, rows = [64, 64, 64, 64], 300
    P = _params(dims, True, 5)
    g = torch.Generator(device=DEV).manual_seed(1)
    X, dY = torch.randn(rows, 64, device=DEV, generator=g), torch.randn(rows, 64, device=DEV, generator=g)
    off = [torch.empty(rows * 64 + 1, device=DEV)[1:].view(rows, 64).copy_(t) for t in (X, dY)]
    assert off[0].data_ptr() % 16 == 4
    ts = [torch.as_tensor(t, dtype=torch.float32, device=DEV) for t in [*P["W"], *P["b"], P["gamma"], P["beta"]]]
    S = gnn.mlp_struct(dims, ts, True)
    f, b = C.c_size_t(), C.c_size_t()
    B.call("gnn_mlp_workspace_size", C.byref(S), rows, C.byref(f), C.byref(b))
    ws = gnn.workspace(max(f.value, b.value), DEV)
    res = []
    for x, dy in ((X, dY), off):
        Y, dX = torch.empty(rows, 64, device=DEV), torch.empty(rows, 64, device=DEV)
        d = [torch.zeros_like(t) for t in ts]
        dS = gnn.mlp_struct(dims, d, True)
        B.call("gnn_mlp_forward", C.byref(S), rows, B.ptr(x), B.ptr(Y), 0, 1e-5, B.ptr(ws), ws.numel(), None)
        B.call("gnn_mlp_backward", C.byref(S), rows, B.ptr(x), B.ptr(dy), 0, B.ptr(dX), C.byref(dS), 1e-5, B.ptr(ws),
               ws.numel(), None)
        B.call("gnn_check", None)
        res.append([Y, dX, *d])
    for a, c in zip(*res):
        assert torch.equal(a, c)


def test_elu_and_special_values():
    # W = 1, b = 0: y = ELU(x) of every magnitude, and rows with NaN or infinity stay their own
    P = {"W": [np.ones((1, 1)), np.ones((1, 1))], "b": [np.zeros(1), np.zeros(1)]}
    g = torch.Generator(device=DEV).manual_seed(2)
    x = torch.exp(torch.rand(20000, 1, device=DEV, generator=g) * 70 - 60) * torch.sign(torch.randn(20000, 1, device=DEV, generator=g))
    x[5], x[900] = float("nan"), float("inf")
    y, _, _ = _run(P, [1, 1, 1], False, x, torch.zeros_like(x))
    keep = torch.isfinite(x)
    ref = torch.nn.functional.elu(x.double())
    # one rounding of the result, the reduction's and the series' (together below 1 ulp), one per Linear sum
    assert float(((y.double() - ref).abs() / ref.abs().clamp_min(1e-30))[keep].max()) < 4 * 2.0 ** -24 * 2
    assert not torch.isfinite(y[~keep]).any()


@pytest.mark.parametrize("H,n_hidden", [(1, 0), (3, 2), (20, 1), (64, 5), (100, 2), (128, 2)])
def test_layer_matches_oracle(H, n_hidden):
    nel, p, R = (3, 2, 3), 2, 4
    brick, subs = oracle_subgraphs(nel, p, R, "rcb")
    part = MeshGraph(nel, p).partition(R, "rcb")
    G = part.to_device(DEV)
    lp = syn.gnn_params(4, H, n_hidden, 1, randomize_affine=True)["layers"][0]
    rng = np.random.default_rng(7)
    x = rng.standard_normal((part.graph.n_nodes, H)).astype(np.float32).astype(np.float64)[part.array("row_gid")]
    e = rng.standard_normal((part.n_edges, H)).astype(np.float32).astype(np.float64)
    x1, e1, cache = om.layer_forward(lp, subs, split_rows(x, subs), split_edges(e, subs))
    dx1 = [rng.standard_normal(a.shape) for a in x1]
    de1 = [rng.standard_normal(a.shape) for a in e1]
    dx0, de0, _ = om.layer_backward(lp, subs, cache, dx1, de1)
    params = syn.gnn_params(4, H, n_hidden, 1, randomize_affine=True)
    layer = gnn.ConsistentGNN(params, precision="fp32", device=DEV).layers[0]
    tens = layer.edge.tensors() + layer.node.tensors()
    W = gnn.mp_params(layer.edge.dims, layer.node.dims, tens)
    cfg = gnn.mp_config(H, "fp32")
    to = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device=DEV)  # noqa: E731
    xt, et = to(x), to(e)
    xo, eo, a = torch.empty_like(xt), torch.empty_like(et), torch.empty_like(xt)
    gnn.gnn_mp_forward(G, cfg, W, xt, et, xo, eo, a)
    # (H = 1: LayerNorm maps every row to beta, and the oracle's zero gradients have no relative error)
    assert rel_l2(xo.cpu().numpy(), np.concatenate(x1)) < TOL
    assert rel_l2(eo.cpu().numpy(), np.concatenate(e1)) < TOL
    gx, ge = to(np.concatenate(dx1)), to(np.concatenate(de1))
    res = []
    for alias, star in ((False, a), (True, a), (False, None)):
        dts = [torch.zeros_like(t) for t in tens]
        dW = gnn.mp_params(layer.edge.dims, layer.node.dims, dts)
        up = ge.clone()
        dx, de = torch.empty_like(xt), up if alias else torch.empty_like(et)
        gnn.gnn_mp_backward(G, cfg, W, xt, et, star, gx, up, dx, de, dW)
        B.call("gnn_check", None)
        res.append([dx, de.clone(), *dts])
    assert rel_l2(res[0][0].cpu().numpy(), np.concatenate(dx0)) < TOL
    assert rel_l2(res[0][1].cpu().numpy(), np.concatenate(de0)) < TOL
    for other in res[1:]:   # de_in may be de_out's buffer; a* may be recomputed
        for u, v in zip(res[0], other):
            assert torch.equal(u, v)
