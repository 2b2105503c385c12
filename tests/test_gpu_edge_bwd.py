"""The edge adjoint of the fused BF16 backward (edge_bwd.cu), H <= 64, where its
tile groups have their edges: one tile, fewer tiles than groups, uneven shares,
every depth that fits (needs a GB300).

Tolerances: the BF16 path's 5e-2 relative L2 on gradients against the FP32 path
(2e-2 on outputs); the recomputing and the saved-activation forms load the same
BF16 hidden activations, so their results are equal bit for bit, as are two runs."""
import numpy as np
import pytest
import torch

import synthetic as syn
from paper_2410_01657_gb300 import _build
from paper_2410_01657_gb300 import binding as B
from paper_2410_01657_gb300 import nn as gnn
from paper_2410_01657_gb300.graph import MeshGraph

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()
    B.load()


def _grads(G, part, H, n_hidden, precision, x, e, dx1, de1, save):
    params = syn.gnn_params(5, H, n_hidden, 1, randomize_affine=True)
    layer = gnn.ConsistentGNN(params, precision=precision, device=DEV).layers[0]
    tens = [t.detach().requires_grad_() for t in (*layer.edge.tensors(), *layer.node.tensors())]
    xt = x.clone().requires_grad_()
    et = e.to(torch.bfloat16 if precision == "bf16" else torch.float32).requires_grad_()
    xo, eo = gnn.ConsistentMPFunction.apply(xt, et, G, (H, precision, True, 1e-5, 0), layer.edge.dims, layer.node.dims,
                                            save, *tens)
    outs, ups = ([xo, eo], [dx1, de1.to(eo.dtype)]) if de1 is not None else ([xo], [dx1])
    g = torch.autograd.grad(outs, [xt, et, *tens], ups)
    B.call("gnn_check", None)
    return [t.float() for t in g]


def _rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm().clamp_min(1e-30))


@pytest.mark.parametrize("H,n_hidden", [(16, 0), (16, 6), (32, 1), (32, 2), (32, 3), (32, 5), (64, 0), (64, 1), (64, 2)])
@pytest.mark.parametrize("nel,p,R", [((1, 1, 1), 1, 1), ((2, 2, 1), 2, 3), ((7, 6, 9), 4, 5)])
@pytest.mark.parametrize("edge_up", [False, True])
def test_edge_adjoint(H, n_hidden, nel, p, R, edge_up):
    part = MeshGraph(nel, p).partition(min(R, nel[0] * nel[1] * nel[2]), "rcb")
    G = part.to_device(DEV)
    g = torch.Generator(device=DEV).manual_seed(11)
    gid = torch.from_numpy(part.array("row_gid")).to(DEV)
    x = torch.randn(part.graph.n_nodes, H, device=DEV, generator=g)[gid]
    e = torch.randn(part.n_edges, H, device=DEV, generator=g).bfloat16().float()
    dx1 = torch.randn(part.n_rows, H, device=DEV, generator=g)
    de1 = torch.randn(part.n_edges, H, device=DEV, generator=g).bfloat16().float() if edge_up else None
    runs = [_grads(G, part, H, n_hidden, "bf16", x, e, dx1, de1, save) for save in (False, False, True)]
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert torch.equal(a, b)
    ref = _grads(G, part, H, n_hidden, "fp32", x, e, dx1, de1, False)
    assert _rel(runs[0][0], ref[0]) < 5e-2 and _rel(runs[0][1], ref[1]) < 5e-2
    for k, (a, b) in enumerate(zip(runs[0][2:], ref[2:])):
        # a gradient that nearly cancels over the edges is held to the sum's scale
        scale = max(float(b.norm()), 0.1 * part.n_edges ** 0.5)
        assert float((a - b).norm()) < 5e-2 * scale, k
