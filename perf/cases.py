"""Performance cases of the consistent mesh-GNN framework, through its public entry points.

A case is a mesh (a GLL brick or a mixed hex/tet mesh with a hub node), its
partition into sub-graphs, a width, a precision and the work done on it:

* ``forward``   one consistent layer forward on preallocated buffers (``nn.gnn_mp_forward``);
* ``train``     one consistent layer forward and backward through autograd
  (``ConsistentGNN.process``), with upstream gradients on both states;
* ``stack``     a ``LayerStack`` training step (zero_grad, forward, backward), optionally
  replayed from a captured CUDA graph;
* ``infer``     an inference ``LayerStack`` (no edge output of the last layer);
* ``encoder`` / ``decoder``  one row MLP forward and backward (the edge encoder over the
  edge attributes, the node decoder over the node states);
* ``network``   a whole training step: encoders, layer, decoder, consistent loss, backward.

Node and edge states are N(0,1), the per-feature scale that the encoders'
LayerNorm produces; the network takes a smooth Fourier velocity field and the
field one step later as its target. Weights are Xavier-uniform with random
biases and LayerNorm parameters.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import synthetic as syn
from paper_2410_01657_gb300 import nn as gnn
from paper_2410_01657_gb300.graph import MeshGraph

DEV = "cuda"
LN_EPS = 1e-5
EXACT_CHUNK = 1 << 20   # rows of one piece of the 64-bit evaluation

_BASE = {"mesh": "brick", "nx": 4, "ny": 4, "nz": 4, "p": 3, "parts": 2, "method": "slab", "uneven": False,
         "work": "train", "precision": "bf16", "hidden": 64, "n_hidden": 2, "layers": 1, "save_act": False,
         "captured": False}


def _case(**kw):
    return {**_BASE, **kw}


def listed():
    return [
        # Plain FP32 layer of a small mesh in two slabs: the smallest call, one layer evaluated on its own.
        _case(name="fp32_forward_4cube_h16", work="forward", precision="fp32", hidden=16),
        # A small model stepped many times (an inner training loop captured in a CUDA graph): launch latency.
        _case(name="bf16_stack_graph_4cube_h16", work="stack", hidden=16, layers=2, captured=True),
        # FP32 training of one layer on the mid-size brick, 8 RCB parts: the precision chosen for gradient checks.
        _case(name="fp32_train_16cube_h64", precision="fp32", nx=16, ny=16, nz=16, p=5, parts=8, method="rcb"),
        # A whole FP32 training step (encoders, layer, decoder, loss) on a small brick: development and validation.
        _case(name="fp32_network_8cube_h64", work="network", precision="fp32", nx=8, ny=8, nz=8, p=5, parts=8,
              method="rcb"),
        # BF16 training of one layer on the mid-size brick: the everyday training path, activations recomputed.
        _case(name="bf16_train_16cube_h64", nx=16, ny=16, nz=16, p=5, parts=8, method="rcb"),
        # The same path with the activations kept, on sub-graphs of uneven size from a non-cubic brick.
        _case(name="bf16_train_saved_uneven_h64", nx=19, ny=17, nz=13, p=5, parts=24, method="rcb", uneven=True,
              save_act=True),
        # The wide model: one layer of the H = 128 training step on a p = 7 brick.
        _case(name="bf16_stack_16cube_h128", work="stack", nx=16, ny=16, nz=16, p=7, parts=8, method="rcb", hidden=128),
        # One H = 128 layer forward (evaluation) on an odd-sized brick.
        _case(name="bf16_forward_odd_h128", work="forward", nx=11, ny=13, nz=9, p=6, parts=5, method="rcb", hidden=128),
        # Large-graph inference: four layers at H = 32, 16 parts, no edge output of the last layer.
        _case(name="bf16_infer_24cube_h32", work="infer", nx=24, ny=24, nz=24, p=7, parts=16, method="rcb", hidden=32,
              layers=4),
        # The deep narrow model (5 hidden layers, H = 32) in training.
        _case(name="bf16_train_deep_h32", nx=16, ny=16, nz=16, p=5, parts=8, method="rcb", hidden=32, n_hidden=5),
        # A general mixed-element mesh with a hub node held as many copy rows.
        _case(name="bf16_train_mixed_h64", mesh="mixed", nx=40, ny=40, nz=40, p=1, parts=8, method="rcb"),
        # The edge encoder of the wide model over every edge of a p = 7 brick, forward and backward.
        _case(name="bf16_encoder_h128", work="encoder", nx=12, ny=12, nz=12, p=7, parts=8, method="rcb", hidden=128),
    ]


def _brick_edges(c):
    l = [c["nx"] * c["p"] + 1, c["ny"] * c["p"] + 1, c["nz"] * c["p"] + 1]
    return 2 * sum(math.prod(l) // l[a] * (l[a] - 1) for a in range(3))


# MP-layer work (edges x H^2 x Linear layers x layers) that a drawn case may have at most, by precision:
# FP32 and BF16 stay below the listed cases of the same precision
_MOST = {"fp32": 3.1e6 * 64 * 64 * 4, "bf16": 8.6e6 * 128 * 128 * 4}


def draw(rng):
    precision = rng.choice(["bf16", "bf16", "bf16", "fp32"])
    work = rng.choice(["train", "train", "stack", "forward", "infer", "encoder", "decoder", "network"])
    hidden = rng.choice([16, 32, 64, 128] if precision == "bf16" else [16, 24, 32, 64, 100, 128])
    n_hidden = rng.choice([1, 2, 2, 2, 5])
    if hidden == 128 and work in ("encoder", "decoder", "network"):
        n_hidden = min(n_hidden, 2)
    if work == "network":
        n_hidden = min(n_hidden, 2)   # the outputs are every gradient tensor
    layers = {"stack": 1 if n_hidden == 5 else rng.choice([1, 2]), "infer": rng.choice([1, 2, 4])}.get(work, 1)
    c = _case(precision=precision, work=work, hidden=hidden, n_hidden=n_hidden, layers=layers,
              save_act=precision == "bf16" and hidden < 128 and work in ("train", "stack") and rng.random() < 0.3)
    most = min(4e7, _MOST[precision] / (hidden * hidden * (n_hidden + 2) * layers))
    edges = math.exp(rng.uniform(math.log(2e3), math.log(most)))
    if rng.random() < 0.15 and edges > 2e4:
        n = max(6, min(40, int((edges / 11.5) ** (1 / 3))))
        c.update(mesh="mixed", nx=n, ny=n, nz=n, p=1)
    else:
        p = rng.choice([1, 2, 3, 4, 5, 6, 7])
        side = max(1.0, (edges / 6) ** (1 / 3) / p)
        nel = [max(1, round(side * rng.uniform(0.6, 1.6))) for _ in range(3)]
        c.update(nx=nel[0], ny=nel[1], nz=nel[2], p=p)
        while _brick_edges(c) > most:
            a = max(("nx", "ny", "nz"), key=lambda k: c[k])
            c[a] -= 1
    elems = c["nx"] * c["ny"] * c["nz"]
    c["parts"] = max(1, min(rng.choice([1, 2, 3, 5, 8, 16, 64]), elems // 8))
    c["method"] = rng.choice(["rcb", "rcb", "slab"])
    if c["method"] == "slab":
        c["parts"] = min(c["parts"], c["nz"])
    c["uneven"] = c["method"] == "rcb" and c["mesh"] == "brick" and elems >= 16 * c["parts"] and rng.random() < 0.3
    c["captured"] = work == "stack" and rng.random() < 0.5
    return c


# ------------------------------------------------------------------ inputs

def _partition(c):
    if c["mesh"] == "mixed":
        m = syn.mixed_element_mesh(c["nx"], 0)
        g = MeshGraph.from_elements(m["pos"], m["elem_ptr"], m["elem_nodes"], m["edge_ptr"], m["edge_pairs"])
    else:
        g = MeshGraph((c["nx"], c["ny"], c["nz"]), c["p"])
    w = None
    if c["uneven"]:
        n = c["nx"] * c["ny"] * c["nz"]
        w = syn.rescale_counts(syn.log_uniform_counts(c["parts"], 5, 500, 0), n).astype(np.float64)
    return g.partition(c["parts"], c["method"], w)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _inputs(c, part, seed):
    """The tensors that the program holds: states, fields, upstream gradients (FP32, or BF16 for the edge state)."""
    g, H = _gen(seed), c["hidden"]
    NR, E = part.n_rows, part.n_edges
    edt = torch.bfloat16 if c["precision"] == "bf16" else torch.float32
    rows = lambda n, w, dt=torch.float32: torch.randn(n, w, device=DEV, generator=g, dtype=dt)  # noqa: E731
    t = {}
    if c["work"] in ("encoder", "network"):
        t["attr"] = torch.from_numpy(part.array("edge_attr")).to(DEV)
    if c["work"] == "network":
        pos = torch.from_numpy(part.array("row_pos")).to(DEV)
        m = syn.fourier_modes(seed, 8)
        k, amp, ph = (torch.from_numpy(np.asarray(m[n], dtype=np.float64)).to(DEV) for n in ("k", "amp", "phase"))
        shift = 0.1 * k.norm(dim=1)
        arg = 2 * math.pi * (pos @ k.T)
        for name, adv in (("u", 0.0), ("target", 1.0)):
            t[name] = sum(amp[i] * torch.sin(arg[:, i:i + 1] + ph[i] + adv * shift[i]) for i in range(8)).float()
        return t
    if c["work"] == "encoder":
        t["dy"] = rows(E, H, edt)
        return t
    t["x"] = rows(NR, H)
    if c["work"] == "decoder":
        t["dy"] = rows(NR, 3)
        return t
    t["e"] = rows(E, H, edt)
    if c["work"] in ("train", "stack"):
        t["dx"] = rows(NR, H)
    if c["work"] == "train":
        t["de"] = rows(E, H, edt)
    return t


def _params(c, seed):
    return syn.gnn_params(seed, c["hidden"], c["n_hidden"], c["layers"], randomize_affine=True)


def prepare(case, seed):
    c = case
    part = _partition(c)
    G = part.to_device(DEV)
    t = _inputs(c, part, seed)
    net = gnn.ConsistentGNN(_params(c, seed), precision=c["precision"], device=DEV, save_act=c["save_act"])
    s = {"case": c, "G": G, "net": net, **t}
    if c["work"] == "forward":
        s["cfg"] = gnn.mp_config(c["hidden"], c["precision"])
        L = net.layers[0]
        s["keep"] = [q.detach() for q in (*L.edge.tensors(), *L.node.tensors())]
        s["W"] = gnn.mp_params(L.edge.dims, L.node.dims, s["keep"])
        s["x_out"], s["e_out"], s["a"] = torch.empty_like(t["x"]), torch.empty_like(t["e"]), torch.empty_like(t["x"])
        s["ws"] = gnn.workspace(gnn.mp_workspace_sizes(G, s["cfg"], s["W"])[0], DEV)
    elif c["work"] in ("stack", "infer"):
        layers = [([q.detach() for q in m.edge.tensors()], [q.detach() for q in m.node.tensors()], m.edge.dims,
                   m.node.dims) for m in net.layers]
        s["stack"] = gnn.LayerStack(G, layers, c["hidden"], c["precision"], t["x"], t["e"],
                                    inference=c["work"] == "infer", save_act=c["save_act"])
        if c["captured"]:
            s["stack"].capture(t["dx"])
    elif c["work"] == "train":
        s["x"].requires_grad_()
        s["e"].requires_grad_()
    elif c["work"] == "decoder":
        s["x"].requires_grad_()
    return s


# ------------------------------------------------------------------ one pass

def run(state):
    s = state
    c, net, G = s["case"], s["net"], s["G"]
    if c["work"] == "forward":
        gnn.gnn_mp_forward(G, s["cfg"], s["W"], s["x"], s["e"], s["x_out"], s["e_out"], s["a"], s["ws"])
        return {"x": s["x_out"], "e": s["e_out"], "a": s["a"]}
    if c["work"] == "infer":
        s["stack"].forward()
        return {"x": s["stack"].x_out}
    if c["work"] == "stack":
        st = s["stack"]
        st.zero_grad()
        if c["captured"]:
            st.replay()
        else:
            st.step(s["dx"])
        return {"x": st.x_out, "e": st.e[-1], "dx": st.dx[0], "de": st.de[0], "dw": st.dparams}
    if c["work"] == "train":
        x, e = net.process(G, s["x"], s["e"])
        ps = list(net.layers.parameters())
        dx, de, *dw = torch.autograd.grad([x, e], [s["x"], s["e"], *ps], [s["dx"], s["de"]])
        return {"x": x, "e": e, "dx": dx, "de": de, "dw": dw}
    if c["work"] == "encoder":
        m = net.enc_edge
        y = gnn.RowMLPFunction.apply(s["attr"], m.dims, m.has_ln, c["precision"] == "bf16", LN_EPS, False,
                                     c["precision"] == "bf16", False, *m.tensors())
        return {"y": y, "dw": list(torch.autograd.grad(y, m.tensors(), s["dy"]))}
    if c["work"] == "decoder":
        m = net.dec
        y = gnn.RowMLPFunction.apply(s["x"], m.dims, m.has_ln, False, LN_EPS, True, c["precision"] == "bf16", False,
                                     *m.tensors())
        dx, *dw = torch.autograd.grad(y, [s["x"], *m.tensors()], s["dy"])
        return {"y": y, "dx": dx, "dw": dw}
    y = net(G, s["u"], s["attr"])
    loss = gnn.consistent_loss(y, s["target"], G)
    return {"y": y, "loss": loss, "dw": list(torch.autograd.grad(loss, list(net.parameters())))}


# ------------------------------------------------------------------ work

def work(case):
    """Bytes: node states 4H and edge states s_e H per row/edge, each input read and each output written
    once, 12 bytes of graph per edge. FLOPs: the first edge Linear split into two products per node and one
    per edge; the backward has twice the forward's."""
    c = case
    part = _partition(c)
    NR, E, H, L = part.n_rows, part.n_edges, c["hidden"], c["n_hidden"] + 2
    se = 2 if c["precision"] == "bf16" else 4
    mlp = 2 * H * H * (L - 1)
    layer = E * 2 * H * H * L + NR * (4 * H * H + 4 * H * H + 2 * H * H * (L - 1))
    w = c["work"]
    if w == "encoder":
        return {"bytes": E * (16 + 2 * se * H), "flops": 3 * E * (8 * H + mlp)}
    if w == "decoder":
        return {"bytes": NR * (8 * H + 24), "flops": 3 * NR * (6 * H + mlp)}
    if w == "network":
        return {"bytes": E * (16 + 12) + NR * 36,
                "flops": 3 * (layer * c["layers"] + E * (8 * H + mlp) + NR * (12 * H + 2 * mlp))}
    graph = 12 * E
    if w == "forward":
        return {"bytes": graph + 2 * se * H * E + 12 * H * NR, "flops": layer}
    if w == "infer":
        return {"bytes": graph + se * H * E + 8 * H * NR, "flops": c["layers"] * layer}
    grads = 2 if w == "train" else 1
    return {"bytes": graph + (2 + grads) * se * H * E + 16 * H * NR, "flops": 3 * c["layers"] * layer}


# ------------------------------------------------------------------ the same in 64 bits

def _mlp64(P, z):
    """The layers after the first Linear, which gave z: ELU, Linear, ..., LayerNorm."""
    W, b, ln = P
    for k in range(1, len(W)):
        z = torch.nn.functional.linear(torch.nn.functional.elu(z), W[k], b[k])
    return torch.nn.functional.layer_norm(z, z.shape[1:], ln[0], ln[1], LN_EPS) if ln else z


def _pieces(fn, n, *tens):
    """fn over pieces of n rows of the tensors, keeping only the pieces' inputs for the backward."""
    out = []
    for i in range(0, n, EXACT_CHUNK):
        a = [t[i:i + EXACT_CHUNK] for t in tens]
        out.append(checkpoint(fn, *a, use_reentrant=False) if torch.is_grad_enabled() else fn(*a))
    return torch.cat(out)


def _row64(P, X):
    return _pieces(lambda x: _mlp64(P, torch.nn.functional.linear(x.double(), P[0][0], P[1][0])), X.shape[0], X)


def _layer64(c, part, Pe, Pn, x, e):
    """Edge update with residual, 1/d-weighted receiver sums completed over all copies of a node, node update
    with residual; returns x', e' and a*."""
    H = c["hidden"]
    recv = torch.from_numpy(part.receivers()).to(DEV)
    col = torch.from_numpy(part.array("col").astype(np.int64)).to(DEV)
    w = torch.from_numpy(part.array("edge_w")).to(DEV).double()
    Wa, Wb, Wc = Pe[0][0].split(H, dim=1)

    def edge(ei, r, s):
        ei = ei.double()
        return ei + _mlp64(Pe, (x @ Wa.T)[r] + (x @ Wb.T)[s] + ei @ Wc.T + Pe[1][0])

    e1 = _pieces(edge, part.n_edges, e, recv, col)
    a = torch.zeros(part.n_rows, H, device=DEV, dtype=torch.float64).index_add(0, recv, e1 * w[:, None])
    hp = torch.from_numpy(part.array("halo_ptr").astype(np.int64)).to(DEV)
    hr = torch.from_numpy(part.array("halo_rows").astype(np.int64)).to(DEV)
    if hr.numel():
        of = torch.repeat_interleave(torch.arange(hp.numel() - 1, device=DEV), hp.diff())
        sums = torch.zeros(hp.numel() - 1, H, device=DEV, dtype=torch.float64).index_add(0, of, a[hr])
        a = a.index_copy(0, hr, sums[of])
    x1 = _pieces(lambda ai, xi: xi + _mlp64(Pn, torch.nn.functional.linear(torch.cat([ai, xi], 1), Pn[0][0], Pn[1][0])),
                 part.n_rows, a, x)
    return x1, e1, a


def exact(case, seed):
    c = case
    part = _partition(c)
    t = _inputs(c, part, seed)
    p = _params(c, seed)
    train = c["work"] not in ("forward", "infer")
    flat = {}

    def mlp(q, key):   # parameters as FP32 holds them, in the order W..., b..., gamma, beta
        ts = [torch.as_tensor(v, dtype=torch.float32, device=DEV).double().requires_grad_(train)
              for v in (*q["W"], *q["b"], *((q["gamma"], q["beta"]) if "gamma" in q else ()))]
        n = len(q["W"])
        flat[key] = ts
        return ts[:n], ts[n:2 * n], ts[2 * n:]

    with torch.set_grad_enabled(train):
        if c["work"] == "encoder":
            y = _row64(mlp(p["enc_edge"], "m"), t["attr"])
            return {"y": y.detach(), "dw": list(torch.autograd.grad(y, flat["m"], t["dy"].double()))}
        if c["work"] == "decoder":
            x = t["x"].double().requires_grad_()
            y = _row64(mlp(p["dec"], "m"), x)
            dx, *dw = torch.autograd.grad(y, [x, *flat["m"]], t["dy"].double())
            return {"y": y.detach(), "dx": dx, "dw": dw}
        layers = [(mlp(q["edge"], f"{i}e"), mlp(q["node"], f"{i}n")) for i, q in enumerate(p["layers"])]
        per_layer = [flat[f"{i}e"] + flat[f"{i}n"] for i in range(c["layers"])]
        if c["work"] == "network":
            x, e = _row64(mlp(p["enc_node"], "u"), t["u"]), _row64(mlp(p["enc_edge"], "a"), t["attr"])
            for Pe, Pn in layers:
                x, e, _ = _layer64(c, part, Pe, Pn, x, e)
            y = _row64(mlp(p["dec"], "d"), x)
            w = torch.from_numpy(part.array("node_w")).to(DEV).double()
            loss = (w[:, None] * (y - t["target"].double()) ** 2).sum() / (w.sum() * 3)
            ps = flat["u"] + flat["a"] + [q for l in per_layer for q in l] + flat["d"]
            return {"y": y.detach(), "loss": loss.detach(), "dw": list(torch.autograd.grad(loss, ps))}
        x0, e0 = t["x"].double().requires_grad_(train), t["e"].double().requires_grad_(train)
        x, e, a = x0, e0, None
        for Pe, Pn in layers:
            x, e, a = _layer64(c, part, Pe, Pn, x, e)
        if c["work"] == "forward":
            return {"x": x, "e": e, "a": a}
        if c["work"] == "infer":
            return {"x": x}
        outs, ups = ([x, e], [t["dx"].double(), t["de"].double()]) if c["work"] == "train" else ([x], [t["dx"].double()])
        dx, de, *dw = torch.autograd.grad(outs, [x0, e0, *(q for l in per_layer for q in l)], ups)
        if c["work"] == "train":
            return {"x": x.detach(), "e": e.detach(), "dx": dx, "de": de, "dw": dw}
        grads, k = [], 0
        for l in per_layer:
            grads.append(dw[k:k + len(l)])
            k += len(l)
        return {"x": x.detach(), "e": e.detach(), "dx": dx, "de": de, "dw": grads}
