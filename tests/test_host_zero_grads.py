"""Gradient buffers of one allocation behave as tensors of their own (CPU)."""
import torch

from paper_2410_01657_gb300 import nn as gnn


def test_pieces_are_independent_tensors():
    like = [torch.empty(3, 5), torch.empty(7), torch.empty(64, 2), torch.empty(1)]
    flat, g = gnn.zero_grads(like)
    for t, p in zip(like, g):
        assert p.shape == t.shape and p.dtype == torch.float32 and p.is_contiguous() and not p.any()
        assert p.data_ptr() % 16 == 0 and not p._is_view()
    # a gradient saved in a graph, another one changed in place (an optimizer, a second backward)
    w = torch.ones(3, 5, requires_grad=True)
    loss = (g[0] * w).sum()
    g[1].add_(1.0)
    loss.backward()
    assert torch.equal(w.grad, g[0])
    assert torch.equal(g[1], torch.ones(7)) and not g[2].any() and not g[0].any()
    flat.zero_()   # one launch for all of them
    assert not any(p.any() for p in g)
