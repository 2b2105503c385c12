"""FP32 layer backward with its gradient outputs in the buffers of its inputs or
upstream gradients (needs a GB300): the same bits as with buffers of their own."""
import pytest
import torch

import synthetic as syn
from paper_2410_01657_gb300 import binding as B
from paper_2410_01657_gb300 import nn as gnn
from paper_2410_01657_gb300.graph import MeshGraph
from test_gpu_lin3 import DEV, built  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,n_hidden", [(7, 1), (64, 2), (128, 2), (136, 1)])
@pytest.mark.parametrize("star,with_de", [(True, True), (False, True), (True, False)])
def test_gradients_in_place(H, n_hidden, star, with_de):
    part = MeshGraph((3, 2, 3), 3).partition(3, "rcb")
    G = part.to_device(DEV)
    layer = gnn.ConsistentGNN(syn.gnn_params(2, H, n_hidden, 1, randomize_affine=True), precision="fp32", device=DEV).layers[0]
    tens = layer.edge.tensors() + layer.node.tensors()
    W, cfg = gnn.mp_params(layer.edge.dims, layer.node.dims, tens), gnn.mp_config(H, "fp32")
    g = torch.Generator(device=DEV).manual_seed(H)
    x, gx = (torch.randn(part.n_rows, H, device=DEV, generator=g) for _ in range(2))
    e, ge = (torch.randn(part.n_edges, H, device=DEV, generator=g) for _ in range(2))
    xo, eo, a = torch.empty_like(x), torch.empty_like(e), torch.empty_like(x)
    gnn.gnn_mp_forward(G, cfg, W, x, e, xo, eo, a)

    def back(dx_at, de_at):
        t = {"x": x.clone(), "e": e.clone(), "gx": gx.clone(), "ge": ge.clone(), "a": a.clone()}
        t["dx"], t["de"] = torch.empty_like(x), torch.empty_like(e)
        d = [torch.zeros_like(q) for q in tens]
        gnn.gnn_mp_backward(G, cfg, W, t["x"], t["e"], t["a"] if star else None, t["gx"], t["ge"] if with_de else None,
                            t[dx_at], t[de_at], gnn.mp_params(layer.edge.dims, layer.node.dims, d))
        B.call("gnn_check", None)
        return [t[dx_at], t[de_at], *d]

    ref = back("dx", "de")
    for at in (("dx", "e"), ("x", "de"), ("x", "e"), ("gx", "ge" if with_de else "e")) + ((("a", "e"),) if star else ()):
        for u, v in zip(ref, back(*at)):
            assert torch.equal(u, v), at
