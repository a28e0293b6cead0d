"""The work that is timed: what a user has this library do, through its public entry points.

A case is one problem (graph, layers, options) and one thing done with it:

  "train"    a stretch of training on a problem that is already on the device: `iters` iterations, then the objective and
             the model (W, b of every layer) on the host, as a driver that reports and checkpoints now and then does
  "epoch"    one iteration with everything the paper's figures record after every epoch: the objective, the residuals and
             the accuracy of the model on all nodes
  "predict"  the trained model on every node: logits, classes, counts
  "fit"      a new problem from host arrays: set-up, `iters` iterations, objective, model, release
  "grow"     the greedy layer-wise schedule: 2, 5, then all layers, `iters` iterations at each depth, from host arrays

The sizes are those of the benchmark's five workloads (c1..c5, the wide ones with fewer layers, so that a state fits the
card three times) and general ones; `draw` spreads over the same ranges.
"""

import math

import numpy as np
import torch

from paper_2105_09837_b200 import binding as B
from paper_2105_09837_b200 import greedy, synth

RHO = NU = 1e-3


def _case(name, op, nodes, degree, feat, hops, classes, layers, hidden, levels=0, neg=0, step=0.0, quant_q=False, slope=0.0,
          act=0, table=0, iters=1):
    """levels 0: pdADMM-G; m >= 2: pdADMM-G-Q with m levels, `neg` of them below zero, spacing `step` (0: from the data);
    slope: leaky ReLU; act 1 or 2: tanh or sigmoid with a lookup table of `table` candidates."""
    c = dict(op=op, nodes=nodes, degree=degree, feat=feat, hops=hops, classes=classes, layers=layers, hidden=hidden, levels=levels,
             neg=neg, step=step, quant_q=quant_q, slope=slope, act=act, table=table, iters=iters)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # c1, the small citation graph: an interactive run that records everything after every epoch.  Latency counts.
        _case("c1 epoch", "epoch", 2000, 4, 250, 2, 7, 10, 100),
        # the same problem trained in stretches of 20 iterations, its iteration count in the benchmark
        _case("c1 train", "train", 2000, 4, 250, 2, 7, 10, 100, iters=20),
        # c1's problem through the greedy schedule 2, 5, 10 layers that the paper trains with, from host arrays
        _case("c1 grow", "grow", 2000, 4, 250, 2, 7, 10, 100, iters=20),
        # c2, the benchmark's headline workload: a medium graph, 10 x 500
        _case("c2 train", "train", 20000, 10, 700, 3, 10, 10, 500, iters=10),
        # the whole job on it as a user meets it: host arrays in, trained model out
        _case("c2 fit", "fit", 20000, 10, 700, 3, 10, 10, 500, iters=20),
        # inference with its model
        _case("c2 predict", "predict", 20000, 10, 700, 3, 10, 10, 500),
        # c3: the same with p on 256 levels (8-bit codes)
        _case("c3 train", "train", 20000, 10, 700, 3, 10, 10, 500, levels=256, iters=5),
        # c4's shape: a large graph, layers of 1000, 8-bit codes
        _case("c4 train", "train", 170000, 14, 128, 4, 40, 5, 1000, levels=256, iters=2),
        # c5's shape: the widest layers, 16 levels
        _case("c5 train", "train", 90000, 10, 500, 3, 7, 8, 2000, levels=16, iters=2),
        # odd sizes throughout, leaky ReLU: nothing is a multiple of a tile
        _case("odd train", "train", 7013, 7, 77, 3, 5, 7, 333, slope=0.1, iters=10),
        # the paper's own level set {-1, 0, ..., 20} for p and q
        _case("signed levels train", "train", 12007, 8, 190, 2, 6, 6, 250, levels=22, neg=1, step=1.0, quant_q=True, iters=5),
        # a smooth activation, its z-update from a lookup table
        _case("tanh train", "train", 10000, 8, 300, 2, 8, 6, 256, act=1, table=513, iters=5),
    ]


def _state_bytes(c):
    return 26.0 * c["nodes"] * c["hidden"] * c["layers"] + 12.0 * c["nodes"] * (c["hops"] + 1) * c["feat"]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        op = rng.choice(["train", "train", "train", "epoch", "predict", "fit", "grow"])
        small = op in ("epoch", "grow")
        layers = rng.randint(3, 12)
        hidden = log_int(64, 500 if small else 2000)
        nodes = log_int(800, 8000 if small else (40000 if op == "fit" else 170000))
        feat, hops = log_int(32, 700), rng.randint(0, 4)
        levels = rng.choice([0, 0, 0, 16, 256, 1024, 22])
        neg, step = (1, 1.0) if levels == 22 else (0, 0.0)
        quant_q = levels > 0 and rng.random() < 0.3
        slope = rng.choice([0.0, 0.0, 0.0, 0.1])
        act = table = 0
        if rng.random() < 0.12 and levels == 0 and nodes * hidden * layers < 3e7:
            act, table, slope = rng.choice([1, 2]), log_int(128, 1025), 0.0
        iters = {"train": rng.randint(2, 12), "epoch": 1, "predict": 1, "fit": rng.randint(10, 40), "grow": rng.randint(5, 20)}[op]
        if levels or act:                 # few: see tolerance()
            iters = min(iters, 3 if op == "grow" else 5)
        c = _case(None, op, nodes, rng.randint(3, 16), feat, hops, rng.randint(3, 48), layers, hidden, levels, neg, step, quant_q, slope,
                  act, table, iters)
        w = work(c)
        if _state_bytes(c) < 2e10 and w["flops"] < 2e13 and w["bytes"] < 4e10:
            return c


def _rand(gen, *shape):
    return torch.rand(shape, generator=gen, device="cuda")


def _inputs(c, seed, layers=None):
    """Host arrays of one problem.  The graph is undirected with a heavy-tailed degree distribution (one end of an edge
    is uniform, the other lands on node i with density ~ i^(-1/2): hubs of degree ~ sqrt(N))."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, d, edges = c["nodes"], c["feat"], c["nodes"] * c["degree"] // 2
    host = lambda t: t.cpu().numpy()  # noqa: E731
    src = host((_rand(gen, edges) * n).int().clamp_(max=n - 1))
    dst = host((_rand(gen, edges).square() * n).int().clamp_(max=n - 1))
    feat = host(torch.randn((n, d), generator=gen, device="cuda"))
    labels = host(torch.randint(0, c["classes"], (n,), generator=gen, device="cuda", dtype=torch.int32))
    mask = host((_rand(gen, n) < 0.5).to(torch.uint8))
    w = synth.Workload("case", seed, n, "ba", c["degree"] // 2, d, "normal", 0.0, c["classes"], c["hops"], layers or c["layers"], c["hidden"],
                       c["levels"], c["iters"], RHO, NU)
    weights, n_in = [], w.n0
    for n_out in w.widths:
        weights.append(host(torch.randn((n_out, n_in), generator=gen, device="cuda") * math.sqrt(2.0 / n_in)))
        n_in = n_out
    return synth.Inputs(w, src, dst, feat, labels, mask, weights)


def _options(c):
    return dict(flags=B.FLAG_QUANT_Q if c["quant_q"] else 0, quant_neg_levels=c["neg"], quant_step=c["step"], leaky_slope=c["slope"],
                activation=c["act"], table=(c["table"], -6.0, 6.0) if c["act"] else (0, 0.0, 0.0))


def _depths(c):
    return sorted({2, min(5, c["layers"]), c["layers"]})


def prepare(case, seed):
    c = case
    s = dict(case=c, options=_options(c))
    # where the model goes: W_1, b_1, W_2, b_2, ... in one flat array
    widths = [(c["hops"] + 1) * c["feat"]] + [c["hidden"]] * (c["layers"] - 1) + [c["classes"]]
    s["model"] = np.zeros(sum(i * o + o for i, o in zip(widths, widths[1:])), dtype=np.float32)
    if c["op"] == "grow":
        s["inputs"] = {L: _inputs(c, seed, L) for L in _depths(c)}
        return s
    inp = _inputs(c, seed)
    if c["op"] == "fit":
        s["inputs"] = inp
        return s
    s["ctx"] = B.from_inputs(inp, **s["options"])
    if c["op"] in ("predict", "epoch"):          # a model in training: at the very start the residuals are rounding noise
        s["ctx"].step(3)
    return s


def _read_model(ctx, flat):
    at = 0
    for layer in range(1, ctx.n_layers + 1):
        for kind in (B.T_W, B.T_B):
            t = ctx.get_tensor(kind, layer)
            flat[at:at + t.size] = t.reshape(-1)
            at += t.size
    return flat


def run(state):
    c = state["case"]
    if c["op"] == "predict":
        logits, classes, counts = state["ctx"].predict()
        return {"logits": logits, "classes": classes, "counts": counts}
    if c["op"] == "epoch":
        ctx = state["ctx"]
        ctx.step(1)
        out = {"objective": ctx.objective(), "residuals": ctx.residuals()}
        out["logits"], out["classes"], out["counts"] = ctx.predict()
        return out
    if c["op"] == "train":
        ctx = state["ctx"]
        ctx.step(c["iters"])
        return {"objective": ctx.objective(), "model": _read_model(ctx, state["model"])}
    if c["op"] == "fit":
        ctx = B.from_inputs(state["inputs"], **state["options"])
        ctx.step(c["iters"])
    else:
        depths = _depths(c)
        ctx = greedy.train(lambda L: state["inputs"][L], depths, [c["iters"]] * len(depths), **state["options"])
    out = {"objective": ctx.objective(), "model": _read_model(ctx, state["model"])}
    ctx.destroy()
    return out


def _iteration(c, layers):
    """Bytes and operations that one iteration cannot do without: p, z, q, u of every layer read and written once (p as its
    codes in pdADMM-G-Q), X once, W read and written; the four products of a layer (two of layer 1), and one more for the
    quantised p."""
    n, n_in = c["nodes"], (c["hops"] + 1) * c["feat"]
    nbytes, flops = 4.0 * n * n_in, 0.0
    code = 4.0 if not c["levels"] else (1.0 if c["levels"] <= 256 else 2.0)
    for l in range(layers):
        n_out = c["hidden"] if l + 1 < layers else c["classes"]
        nbytes += 8.0 * n * n_out * (3 if l + 1 < layers else 1) + 8.0 * n_in * n_out
        flops += 2.0 * n * n_in * n_out * (2 if l == 0 else (5 if c["levels"] else 4))
        if l > 0:
            nbytes += 2.0 * code * n * n_in
        n_in = n_out
    return nbytes, flops


def _forward(c, layers):
    """One pass through the layers: X and W read, logits written; and the products."""
    n, n_in = c["nodes"], (c["hops"] + 1) * c["feat"]
    nbytes, flops = 4.0 * n * n_in, 0.0
    for l in range(layers):
        n_out = c["hidden"] if l + 1 < layers else c["classes"]
        nbytes += 4.0 * n_in * n_out
        flops += 2.0 * n * n_in * n_out
        n_in = n_out
    return nbytes + 4.0 * n * n_in, flops


def work(case):
    c, op = case, case["op"]
    nbytes = flops = 0.0
    for layers in (_depths(c) if op == "grow" else [c["layers"]]):
        b, f = _iteration(c, layers)
        if op != "predict":
            nbytes, flops = nbytes + c["iters"] * b, flops + c["iters"] * f
        if op in ("epoch", "predict", "fit", "grow"):          # a forward pass: the prediction, or the start of Algorithm 1
            b, f = _forward(c, layers)
            nbytes, flops = nbytes + b, flops + f
        if op in ("fit", "grow"):                              # the sparse products that make X
            nbytes += 4.0 * c["nodes"] * c["feat"] * (c["hops"] + 1) + 8.0 * c["nodes"] * (c["degree"] + 1)
            flops += 2.0 * c["nodes"] * (c["degree"] + 1) * c["feat"] * c["hops"]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Single precision through some tens of iterations (two implementations of the products, tensor cores and CUDA cores,
    differ by 1e-7 after one and by 2e-6, 2e-4 of single entries, after thirty).  A projection on a level set and the
    choice among table candidates are decisions: where a value lies within its rounding error of a boundary either side is
    right, and both are followed from there on (the two implementations differ by 2e-5 to 4e-4, 2e-2 of single entries).
    The class of a node whose two largest logits agree in single precision may differ as well."""
    if case["levels"] or case["act"]:
        return {"rel": 1e-3, "max": 0.1, "differ": 1e-3}
    return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
