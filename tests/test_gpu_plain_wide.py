"""The FP32 path above width 128, where the SIMT kernels of plain.cu run, and at
the border between the two forms, against the FP64 oracle (needs a GB300).

Tolerance 1e-5 relative L2 per output and gradient, the FP32 path's bound; a row
MLP's gradient that cancels over its rows is held to the scale of the sum, as
for the narrower widths."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle import model as om
from paper_2410_01657_gb300 import binding as B
from paper_2410_01657_gb300 import nn as gnn
from paper_2410_01657_gb300.graph import MeshGraph
from gpu_util import oracle_subgraphs, rel_l2, split_edges, split_rows
from test_gpu_lin3 import DEV, TOL, _mlp64, _params, _run, built  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,n_hidden", [(128, 1), (129, 2), (136, 0), (256, 1)])
def test_layer(H, n_hidden):
    nel, p, R = (3, 2, 2), 2, 3
    brick, subs = oracle_subgraphs(nel, p, R, "rcb")
    part = MeshGraph(nel, p).partition(R, "rcb")
    G = part.to_device(DEV)
    params = syn.gnn_params(4, H, n_hidden, 1, randomize_affine=True)
    rng = np.random.default_rng(7)
    x = rng.standard_normal((part.graph.n_nodes, H)).astype(np.float32).astype(np.float64)[part.array("row_gid")]
    e = rng.standard_normal((part.n_edges, H)).astype(np.float32).astype(np.float64)
    x1, e1, cache = om.layer_forward(params["layers"][0], subs, split_rows(x, subs), split_edges(e, subs))
    dx1 = [rng.standard_normal(a.shape) for a in x1]
    de1 = [rng.standard_normal(a.shape) for a in e1]
    dx0, de0, grads = om.layer_backward(params["layers"][0], subs, cache, dx1, de1)
    layer = gnn.ConsistentGNN(params, precision="fp32", device=DEV).layers[0]
    tens = layer.edge.tensors() + layer.node.tensors()
    W, cfg = gnn.mp_params(layer.edge.dims, layer.node.dims, tens), gnn.mp_config(H, "fp32")
    to = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device=DEV)  # noqa: E731
    xt, et, gx, ge = to(x), to(e), to(np.concatenate(dx1)), to(np.concatenate(de1))
    xo, eo, a = torch.empty_like(xt), torch.empty_like(et), torch.empty_like(xt)
    gnn.gnn_mp_forward(G, cfg, W, xt, et, xo, eo, a)
    assert rel_l2(xo.cpu().numpy(), np.concatenate(x1)) < TOL
    assert rel_l2(eo.cpu().numpy(), np.concatenate(e1)) < TOL
    flat = [t for k in ("edge", "node") for t in [*grads[k]["W"], *grads[k]["b"], grads[k]["gamma"], grads[k]["beta"]]]
    for star in (a, None):
        d = [torch.zeros_like(t) for t in tens]
        dx, de = torch.empty_like(xt), torch.empty_like(et)
        gnn.gnn_mp_backward(G, cfg, W, xt, et, star, gx, ge, dx, de, gnn.mp_params(layer.edge.dims, layer.node.dims, d))
        B.call("gnn_check", None)
        assert rel_l2(dx.cpu().numpy(), np.concatenate(dx0)) < TOL
        assert rel_l2(de.cpu().numpy(), np.concatenate(de0)) < TOL
        for k, (u, v) in enumerate(zip(d, flat)):
            assert rel_l2(u.cpu().numpy(), v) < TOL, k


@pytest.mark.parametrize("dims,has_ln", [
    (d, ln) for d in ([128, 128, 128], [129, 64, 64], [64, 130, 64], [64, 64, 129], [4, 256, 256, 256], [300, 17, 3])
    for ln in (True, False) if not (ln and d[-1] < 64)])
@pytest.mark.parametrize("rows", [1, 129, 9001])
def test_row_mlp(dims, has_ln, rows):
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
        err = float((a.double() - r).norm() / max(float(r.norm()), 1e-3 * rows ** 0.5))
        assert err < TOL, k
