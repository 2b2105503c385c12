"""Parameters of a layer tied to each other: one gradient buffer for several of
them receives the sum of their gradients (needs a GB300).

Tolerance 1e-6 relative: the sums are the same FP32 numbers added in FP32, at
most eight of them, in another order."""
import numpy as np
import pytest
import torch

import synthetic as syn
from paper_2410_01657_gb300 import binding as B
from paper_2410_01657_gb300 import nn as gnn
from paper_2410_01657_gb300.graph import MeshGraph
from test_gpu_lin3 import DEV, built  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,precision", [(20, "fp32"), (64, "fp32"), (128, "fp32"), (136, "fp32"), (16, "bf16"),
                                         (64, "bf16"), (128, "bf16")])
def test_tied_layer(H, precision):
    part = MeshGraph((3, 2, 3), 3).partition(2, "rcb")
    G = part.to_device(DEV)
    layer = gnn.ConsistentGNN(syn.gnn_params(2, H, 2, 1, randomize_affine=True), precision=precision, device=DEV).layers[0]
    te, tn = layer.edge.tensors(), layer.node.tensors()
    tens, n = te + tn, len(layer.edge.dims) - 1
    W, cfg = gnn.mp_params(layer.edge.dims, layer.node.dims, tens), gnn.mp_config(H, precision)
    g = torch.Generator(device=DEV).manual_seed(H)
    x, gx = (torch.randn(part.n_rows, H, device=DEV, generator=g) for _ in range(2))
    e = torch.randn(part.n_edges, H, device=DEV, generator=g).to(torch.bfloat16 if precision == "bf16" else torch.float32)
    xo, eo, a = torch.empty_like(x), torch.empty_like(e), torch.empty_like(x)
    gnn.gnn_mp_forward(G, cfg, W, x, e, xo, eo, a)

    def back(d):
        gnn.gnn_mp_backward(G, cfg, W, x, e, a, gx, None, torch.empty_like(x), torch.empty_like(e),
                            gnn.mp_params(layer.edge.dims, layer.node.dims, d))
        B.call("gnn_check", None)

    apart = [torch.zeros_like(t) for t in tens]
    back(apart)
    # every hidden weight of both MLPs, every bias with every beta, and both gammas have one buffer each
    m = len(te)
    groups = [[1, 2, 3, m + 1, m + 2, m + 3], [*range(n, 2 * n), 2 * n + 1, *range(m + n, m + 2 * n), m + 2 * n + 1],
              [2 * n, m + 2 * n]]
    tied = [torch.zeros_like(t) for t in tens]
    for idx in groups:
        for i in idx:
            tied[i] = tied[idx[0]]
    back(tied)
    for idx in groups:
        ref = sum(apart[i].double() for i in idx)
        assert float((tied[idx[0]].double() - ref).norm() / ref.norm()) < 1e-6, idx
    for i in (0, m):
        assert torch.equal(tied[i], apart[i])


def test_tied_row_mlp():
    rows, C = 1000, gnn.C
    for precision, has_ln, d0 in (("fp32", True, 64), ("bf16", True, 4)):
        dims = [d0, 64, 64, 64]
        P = syn.xavier_mlp(np.random.default_rng(1), dims, has_ln, randomize_affine=True)
        ts = [torch.as_tensor(t, dtype=torch.float32, device=DEV) for t in [*P["W"], *P["b"], P["gamma"], P["beta"]]]
        g = torch.Generator(device=DEV).manual_seed(3)
        X, dY = torch.randn(rows, d0, device=DEV, generator=g), torch.randn(rows, 64, device=DEV, generator=g)
        S, sfx = gnn.mlp_struct(dims, ts, has_ln), "_bf16" if precision == "bf16" else ""
        f, b = C.c_size_t(), C.c_size_t()
        B.call("gnn_mlp_workspace_size" + sfx, C.byref(S), rows, C.byref(f), C.byref(b))
        ws = gnn.workspace(b.value, DEV)

        def back(d):
            dS = gnn.mlp_struct(dims, d, has_ln)
            B.call("gnn_mlp_backward" + sfx, C.byref(S), rows, B.ptr(X), B.ptr(dY), 0, None, C.byref(dS), 1e-5, B.ptr(ws),
                   ws.numel(), None)
            B.call("gnn_check", None)

        apart = [torch.zeros_like(t) for t in ts]
        back(apart)
        tied = [torch.zeros_like(t) for t in ts]
        tied[2], tied[4], tied[5] = tied[1], tied[3], tied[3]
        back(tied)
        for idx in ([1, 2], [3, 4, 5]):
            ref = sum(apart[i].double() for i in idx)
            assert float((tied[idx[0]].double() - ref).norm() / ref.norm()) < 1e-6, (precision, idx)
