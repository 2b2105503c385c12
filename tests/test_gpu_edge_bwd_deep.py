"""The fused BF16 backward at H <= 64 at the deepest MLPs it takes, against the FP64
oracle, and where it refuses (needs a GB300). Tolerance 5e-2 relative L2 on
gradients, the BF16 path's; a parameter gradient that nearly cancels over the edges
is held to the sum's scale."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle import model as om
from paper_2410_01657_gb300 import binding as B
from paper_2410_01657_gb300 import nn as gnn
from paper_2410_01657_gb300.graph import MeshGraph
from gpu_util import oracle_subgraphs, rel_l2, split_edges, split_rows
from test_gpu_lin3 import DEV, built  # noqa: F401

pytestmark = pytest.mark.gpu


def _layer(H, n_hidden):
    params = syn.gnn_params(6, H, n_hidden, 1, randomize_affine=True)
    return params["layers"][0], gnn.ConsistentGNN(params, precision="bf16", device=DEV).layers[0]


@pytest.mark.parametrize("H,n_hidden", [(16, 6), (32, 3), (32, 4), (32, 6), (64, 2)])
def test_deep_layer(H, n_hidden):
    nel, p, R = (4, 3, 3), 3, 3
    brick, subs = oracle_subgraphs(nel, p, R, "rcb")
    part = MeshGraph(nel, p).partition(R, "rcb")
    G = part.to_device(DEV)
    lp, layer = _layer(H, n_hidden)
    rng = np.random.default_rng(5)
    x = rng.standard_normal((part.graph.n_nodes, H)).astype(np.float32).astype(np.float64)[part.array("row_gid")]
    et = torch.as_tensor(rng.standard_normal((part.n_edges, H)), device=DEV).bfloat16()
    e = et.double().cpu().numpy()
    _, _, cache = om.layer_forward(lp, subs, split_rows(x, subs), split_edges(e, subs))
    dx1, de1 = rng.standard_normal(x.shape), rng.standard_normal(e.shape)
    dx0, de0, grads = om.layer_backward(lp, subs, cache, split_rows(dx1, subs), split_edges(de1, subs))
    xt = torch.as_tensor(x, dtype=torch.float32, device=DEV).requires_grad_()
    et.requires_grad_()
    tens = [t.detach().requires_grad_() for t in (*layer.edge.tensors(), *layer.node.tensors())]
    for save in (False, True):
        xo, eo = gnn.ConsistentMPFunction.apply(xt, et, G, (H, "bf16", True, 1e-5, 0), layer.edge.dims, layer.node.dims,
                                                save, *tens)
        dx, de, *dw = torch.autograd.grad([xo, eo], [xt, et, *tens], [
            torch.as_tensor(dx1, dtype=torch.float32, device=DEV), torch.as_tensor(de1, device=DEV).bfloat16()])
        B.call("gnn_check", None)
        assert rel_l2(dx.cpu().numpy(), np.concatenate(dx0)) < 5e-2
        assert rel_l2(de.float().cpu().numpy(), np.concatenate(de0)) < 5e-2
        flat = [t for k in ("edge", "node") for t in [*grads[k]["W"], *grads[k]["b"], grads[k]["gamma"], grads[k]["beta"]]]
        for k, (a, r) in enumerate(zip(dw, flat)):
            scale = max(float(np.linalg.norm(r)), 0.1 * part.n_edges ** 0.5)
            assert float(np.linalg.norm(a.double().cpu().numpy() - r)) < 5e-2 * scale, (save, k)


def test_too_deep_names_the_limit():
    part = MeshGraph((2, 2, 1), 2).partition(1, "rcb")
    G = part.to_device(DEV)
    _, layer = _layer(64, 3)
    tens = layer.edge.tensors() + layer.node.tensors()
    W, cfg = gnn.mp_params(layer.edge.dims, layer.node.dims, tens), gnn.mp_config(64, "bf16")
    x, e = torch.zeros(part.n_rows, 64, device=DEV), torch.zeros(part.n_edges, 64, device=DEV, dtype=torch.bfloat16)
    with pytest.raises(B.GnnError, match="H=64 supports at most 4 Linear"):
        gnn.gnn_mp_backward(G, cfg, W, x, e, x.clone(), x.clone(), None, x.clone(), e.clone(),
                            gnn.mp_params(layer.edge.dims, layer.node.dims, [torch.zeros_like(t) for t in tens]))
