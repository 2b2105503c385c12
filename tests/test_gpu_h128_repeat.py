"""The H = 128 backward gives the same bits on every run (needs a GB300).

The node recomputation keeps its input, hidden and dz tiles in one buffer: the
next tile's rows may be written only after the TMA store of dz has read it. On
graphs whose node states stay in L2 a missing wait let some rows of dz be
overwritten, and results changed from run to run; on these meshes (four to five
node tiles per SM) most runs showed it."""
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


@pytest.mark.parametrize("mesh", ["mixed", "brick"])
def test_backward_repeats_bit_for_bit(mesh):
    H = 128
    if mesh == "mixed":
        m = syn.mixed_element_mesh(40, 0)
        g = MeshGraph.from_elements(m["pos"], m["elem_ptr"], m["elem_nodes"], m["edge_ptr"], m["edge_pairs"])
    else:
        g = MeshGraph((23, 25, 17), 2)
    part = g.partition(5, "rcb")
    G = part.to_device(DEV)
    gen = torch.Generator(device=DEV).manual_seed(3)
    rnd = lambda n, dt: torch.randn(n, H, device=DEV, generator=gen, dtype=dt)  # noqa: E731
    x, e = rnd(part.n_rows, torch.float32), rnd(part.n_edges, torch.bfloat16)
    dx, de = rnd(part.n_rows, torch.float32), rnd(part.n_edges, torch.bfloat16)
    net = gnn.ConsistentGNN(syn.gnn_params(2, H, 2, 1, randomize_affine=True), precision="bf16", device=DEV)
    ref = None
    for _ in range(6):
        xr, er = x.clone().requires_grad_(), e.clone().requires_grad_()
        xo, eo = net.process(G, xr, er)
        res = torch.autograd.grad([xo, eo], [xr, er, *net.layers.parameters()], [dx, de])
        B.call("gnn_check", None)
        if ref is None:
            ref = res
        for a, b in zip(ref, res):
            assert torch.equal(a, b)
