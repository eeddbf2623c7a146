"""The performance cases of this framework: what its users have it do, each as one timed pass.

A case is a dict of plain values.  ``kind`` names the use:

  train      one full-graph GCN training iteration on resident inputs (``GcnTrainer.epoch``: forward, loss,
             backward, Adam)
  infer      the forward pass alone (``GcnTrainer.forward``): class scores of every node from trained weights
  sage, gin  one training iteration of the two other architectures (``SageTrainer.epoch``, ``GinTrainer.epoch``)
  step_host  one training iteration whose features, labels, mask, weights and moments live in pinned host memory
             (``train_step_host``), predictions for every node returned
  propagate  a graph that arrives as an edge list on the device is built (``graph_create``) and features are
             propagated over it ``hops`` times (``spmm``): inductive use, where every request brings its own graph

The other fields: ``n`` nodes, ``edges`` undirected R-MAT edges before symmetrisation, ``dims`` the layer widths
("64-32-8"), ``precision`` of the dense products, ``mask`` the share of train nodes, ``dropout`` on hidden layers.

The timed pass is the call itself; graphs, trainers, parameters and contexts are made in ``prepare``, where a training
program makes them once.  Training state is that of a run in progress (step count and Adam moments not zero): after a
first step from zero moments the update is the bare sign of the gradient, whose rounding noise says nothing.
"""
import math

import torch

from paper_2501_01951_b200 import binding as mg
from paper_2501_01951_b200 import synth
from paper_2501_01951_b200.sage_gin import GinTrainer, SageTrainer
from paper_2501_01951_b200.train import GcnTrainer

_DEV = "cuda:0"


def _config(key, scale=1.0):
    """Shape of one of the repository's own workloads, node and edge counts scaled."""
    wl = synth.CONFIGS[key]
    return dict(n=int(wl.n * scale), edges=int(wl.undirected_edges * scale), dims="-".join(map(str, wl.dims)),
                precision=wl.precision, mask=wl.mask_p, dropout=0.0)


def listed():
    return [
        # The tiny workload of the repository: an iteration that lasts as long as its launches.  What unit tests, tutorials and
        # hyper-parameter sweeps over small graphs run thousands of times.
        dict(name="train-tiny", kind="train", **_config("C1")),
        # A small citation-like graph with wide bag-of-words features, a narrow hidden layer, few labels and dropout: the
        # classical two-layer use, at the trainer's default precision.
        dict(name="train-small-dropout", kind="train", n=20011, edges=60000, dims="500-32-7", precision="fp32", mask=0.03, dropout=0.5),
        # A medium graph at strict precision with dropout, three layers, more than half of the nodes labelled: FMA products
        # and byte masks beside the aggregation.
        dict(name="train-medium-fp32", kind="train", n=170003, edges=1200000, dims="128-256-256-40", precision="fp32", mask=0.54, dropout=0.5),
        # The dense-neighbourhood workload: aggregations served by the L2 (mean degree 500).
        dict(name="train-dense", kind="train", **_config("C2")),
        # The co-purchase-shaped workload: aggregations served by DRAM, 8 % of the nodes labelled.
        dict(name="train-copurchase", kind="train", **_config("C3")),
        # The wide-feature workload (bf16 products, 1024-wide) at a size whose state fits the card several times.
        dict(name="train-wide-bf16", kind="train", **_config("C4", 0.3)),
        # The large citation-shaped workload (172 classes, 1 % labelled: row-sparse backward), scaled likewise.
        dict(name="train-citation", kind="train", **_config("C5", 0.2)),
        # Scores for every node with odd widths and a ragged node count, bf16 products: a deployed model.
        dict(name="infer-ragged-bf16", kind="infer", n=700001, edges=7000000, dims="301-130-47", precision="bf16", mask=0.1, dropout=0.0),
        # Mean-aggregator GraphSAGE and GIN, medium graphs.
        dict(name="sage", kind="sage", n=400000, edges=6000000, dims="100-256-47", precision="tf32", mask=0.3, dropout=0.0),
        dict(name="gin-ragged", kind="gin", n=150001, edges=1500000, dims="75-128-33", precision="tf32", mask=0.5, dropout=0.0),
        # Host-resident training data: every step copies the features in and the results out.
        dict(name="step-host", kind="step_host", n=500000, edges=4000000, dims="128-128-64", precision="tf32", mask=0.1, dropout=0.0),
        # A graph per request: built on the device from its edge list, then two hops of propagation.
        dict(name="propagate-new-graph", kind="propagate", n=250007, edges=2000000, dims="96-96", precision="fp32", mask=0.0, dropout=0.0, hops=2),
    ]


# ------------------------------------------------------------------------------------------------ drawn cases

def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(case):
    return tuple(int(d) for d in case["dims"].split("-"))


def _entries(case):
    return 2 * case["edges"] + case["n"]


def _estimate(case):
    """(seconds, bytes held) of a case, roughly: gathers at 10 TB/s, products at a rate by precision, host copies at 50 GB/s."""
    d, n, nnz = _dims(case), case["n"], _entries(case)
    passes = {"train": 2, "infer": 1, "sage": 2, "gin": 2, "step_host": 2, "propagate": 1}[case["kind"]]
    gather = sum(4.0 * nnz * min(a, b) for a, b in zip(d, d[1:])) * passes * (case.get("hops") or 1)
    flops = sum(2.0 * n * a * b for a, b in zip(d, d[1:])) * (3 if passes == 2 else 1)
    rate = {"fp32": 40e12, "tf32": 300e12, "bf16": 700e12}[case["precision"]]
    sec = gather / 10e12 + flops / rate
    if case["kind"] == "step_host":
        sec += 4.0 * n * d[0] / 50e9
    if case["kind"] == "propagate":
        sec += nnz * 40 / 1e12
    return sec, 4.0 * n * (sum(d) * 3 + max(d) * 2) + 24.0 * nnz


def draw(rng):
    kind = rng.choice(["train"] * 6 + ["infer"] * 2 + ["sage", "gin", "step_host", "propagate"])
    most_s = max(_estimate(c)[0] for c in listed())
    most_b = max(_estimate(c)[1] for c in listed())
    n = int(_log(rng, 2000, {"train": 3e6, "infer": 3e6, "step_host": 1e6, "propagate": 1e6}.get(kind, 1e6)))
    degree = _log(rng, 3, 40 if kind == "gin" else 300)     # mean, undirected edges counted at both ends
    layers = rng.choice([2, 3] if kind == "gin" else [2, 2, 3, 3, 4])
    precision = rng.choice({"infer": ["fp32", "tf32", "bf16", "bf16"]}.get(kind, ["fp32", "fp32", "tf32", "tf32", "bf16"]))
    wide = precision == "bf16" and rng.random() < 0.5
    hidden = int(_log(rng, 16, 1024 if wide else 300))
    if rng.random() < 0.5:
        hidden = max(16, hidden // 16 * 16)
    first, last = int(_log(rng, 24, 1024 if wide else 700)), int(_log(rng, 2, 180))
    dims = [first] + [hidden] * (layers - 1) + [last]
    hops = None
    if kind == "propagate":
        hops = rng.choice([1, 2, 3])
        w = int(_log(rng, 8, 300))
        dims, precision = [w, w], "fp32"
    case = dict(kind=kind, n=n, edges=0, dims="-".join(map(str, dims)), precision=precision,
                mask=round(0.0 if kind == "propagate" else _log(rng, 0.01, 0.7), 4),
                dropout=rng.choice([0.0, 0.0, 0.5]) if kind == "train" else 0.0)
    if hops:
        case["hops"] = hops
    for _ in range(200):
        case["edges"] = max(case["n"], int(min(case["n"] * degree / 2, 60e6, case["n"] ** 2 / 250)))
        sec, held = _estimate(case)
        if sec <= 0.8 * most_s and held <= 0.8 * most_b and (not case["dropout"] or case["n"] * max(dims) <= 2e8):
            break
        case["n"] = max(2000, int(case["n"] * 0.8))
        degree = max(3.0, degree * 0.95)
    return case


# ------------------------------------------------------------------------------------------------ inputs and handles

def _weights(dims, gen, scale=1.0):
    Ws = [(torch.rand((a, b), generator=gen, device=_DEV) * 2 - 1) * (scale * math.sqrt(6.0 / (a + b))) for a, b in zip(dims, dims[1:])]
    bs = [torch.randn(b, generator=gen, device=_DEV) * 0.05 for b in dims[1:]]
    return Ws, bs


def _moments(ms, vs, gen):
    for m, v in zip(ms, vs):
        m.copy_(torch.randn(m.shape, generator=gen, device=_DEV) * 1e-3)
        v.copy_((torch.rand(v.shape, generator=gen, device=_DEV) + 0.5) * 1e-6)


def prepare(case, seed):
    dims, n, kind = _dims(case), case["n"], case["kind"]
    prec = mg.PRECISIONS[case["precision"]]
    gen = torch.Generator(device=_DEV).manual_seed(seed)
    src, dst = synth.rmat_graph(n, case["edges"], seed, device=_DEV)
    ctx = mg.ctx_create(0)
    ld0 = (dims[0] + 3) // 4 * 4
    X = torch.zeros((n, ld0), device=_DEV)
    X[:, : dims[0]] = torch.randn((n, dims[0]), generator=gen, device=_DEV)
    st = dict(kind=kind, ctx=ctx, dims=dims, prec=prec, t=50)
    if kind == "propagate":
        st.update(n=n, src=src, dst=dst, X=X, hops=case["hops"], Z=[torch.zeros_like(X) for _ in range(2)])
        return st
    y = torch.randint(0, dims[-1], (n,), generator=gen, device=_DEV, dtype=torch.int32)
    m = (torch.rand(n, generator=gen, device=_DEV) < case["mask"]).to(torch.uint8)
    m[: 8] = 1                                      # never empty
    if kind in ("sage", "gin"):
        flags = mg.GRAPH_SYMMETRISE | (mg.GRAPH_NORM_ROW if kind == "sage" else mg.GRAPH_NORM_NONE)
        g = mg.graph_create(ctx, n, src, dst, flags)
        Ws, bs = _weights(dims, gen, 0.7)
        if kind == "sage":
            tr = SageTrainer(ctx, g, dims, prec)
            tr.set_params([w.cpu() for w in Ws], [w.cpu() for w in _weights(dims, gen, 0.7)[0]], bs)
        else:
            hidden = dims[1]
            tr = GinTrainer(ctx, g, dims, hidden, prec)
            inner = [_weights((d, hidden), gen, n / _entries(case)) for d in dims[:-1]]     # a node sums over all its neighbours
            outer = [_weights((hidden, d), gen) for d in dims[1:]]
            tr.set_params([w[0][0] for w in inner], [w[1][0] for w in inner], [w[0][0] for w in outer], [w[1][0] for w in outer])
        tr.set_inputs(X, y, m)
        _moments(tr.m, tr.v, gen)
        st.update(g=g, tr=tr)
        return st
    g = mg.graph_create(ctx, n, src, dst)
    Ws, bs = _weights(dims, gen)
    if kind == "step_host":
        pin = lambda t: t.cpu().pin_memory()
        st.update(g=g, X=pin(X[:, : dims[0]].contiguous()), y=pin(y), m=pin(m), W=[pin(w) for w in Ws], b=[pin(b) for b in bs],
                  pred=torch.zeros(n, dtype=torch.int32).pin_memory())
        for name, like in (("mW", Ws), ("mb", bs)):
            st[name] = [pin(torch.randn(t.shape, generator=gen, device=_DEV) * 1e-3) for t in like]
        for name, like in (("vW", Ws), ("vb", bs)):
            st[name] = [pin((torch.rand(t.shape, generator=gen, device=_DEV) + 0.5) * 1e-6) for t in like]
        return st
    keep = 1.0 - case["dropout"]
    tr = GcnTrainer(ctx, g, dims, prec, keep_scale=1.0 / keep)
    tr.set_params(Ws, bs)
    masks = None
    if case["dropout"]:
        masks = [(torch.rand((n, d), generator=gen, device=_DEV) < keep).to(torch.uint8) for d in dims[1:-1]]
    tr.set_inputs(X, y, m, masks)
    _moments(tr.mW + tr.mb, tr.vW + tr.vb, gen)
    st.update(g=g, tr=tr)
    return st


# ------------------------------------------------------------------------------------------------ the timed pass

def run(st):
    kind = st["kind"]
    if kind == "propagate":
        ctx, w = st["ctx"], st["dims"][0]
        g = mg.graph_create(ctx, st["n"], st["src"], st["dst"])
        Y = st["X"]
        for hop in range(st["hops"]):
            Z = st["Z"][hop % 2]
            mg.spmm(ctx, g, Y, Z, w)
            Y = Z
        out = dict(Z=Y[:, :w], nnz=g.nnz, max_deg=g.max_deg, symmetric=g.symmetric)
        g.close()
        return out
    st["t"] += 1
    if kind == "step_host":
        loss = mg.train_step_host(st["ctx"], st["g"], st["dims"], st["prec"], st["X"], st["y"], st["m"], st["W"], st["b"],
                                  st["mW"], st["vW"], st["mb"], st["vb"], st["t"], pred=st["pred"])
        return dict(loss=loss, pred=st["pred"], **{k: list(st[k]) for k in ("W", "b", "mW", "vW", "mb", "vb")})
    tr = st["tr"]
    if kind == "infer":
        tr.forward()
        return tr.X[tr.L][:, : tr.dims[-1]]
    tr.epoch(st["t"])
    if kind == "train":
        return dict(loss=tr.loss, pred=tr.pred, W=tr.W, b=tr.b, dW=tr.dW, db=tr.db, mW=tr.mW, vW=tr.vW, mb=tr.mb, vb=tr.vb,
                    hidden=[tr.X[l][:, : tr.dims[l]] for l in range(1, tr.L)])
    hidden = [tr.S[l][:, : tr.dims[l]] if kind == "sage" else tr.H[l][:, : tr.dims[l]] for l in range(1, tr.L)]
    return dict(loss=tr.loss, pred=tr.pred, params=tr.params, grads=tr.grads, m=tr.m, v=tr.v, hidden=hidden)


# ------------------------------------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """Per aggregation of width w over a matrix of e entries: 8 e + 8 n bytes of index and value, its input rows and its output
    rows once, 2 e w operations.  Per dense product: both operands and the result once.  Backward passes count the rows that
    can be non-zero only (train rows below the loss, their neighbours one aggregation later); layers aggregate at the narrower
    of their widths.  step_host adds the copies over the host link, propagate the edge list, the sort of its keys being one
    read and one write of each."""
    d, n, nnz, kind = _dims(case), case["n"], _entries(case), case["kind"]
    L = len(d) - 1
    by = fl = 0.0

    def aggregate(w, rows_in, rows_out, entries):
        nonlocal by, fl
        by += 8.0 * entries + 8.0 * rows_out + 4.0 * w * (rows_in + rows_out)
        fl += 2.0 * entries * w

    def product(m, a, b, weight_gradient=False):
        nonlocal by, fl
        by += 4.0 * (m * (a + b) + a * b)
        fl += 2.0 * m * a * b

    if kind == "propagate":
        for _ in range(case["hops"]):
            aggregate(d[0], n, n, nnz)
        return dict(bytes=by + 8.0 * case["edges"] + 32.0 * case["edges"] + 12.0 * nnz, flops=fl)
    self_terms = {"sage": 2, "gin": 1}.get(kind, 1)
    for l in range(L):
        aggregate(d[l] if kind in ("sage", "gin") else min(d[l], d[l + 1]), n, n, nnz)
        product(n, self_terms * d[l], d[1] if kind == "gin" else d[l + 1])
        if kind == "gin":
            product(n, d[1], d[l + 1])
    if kind != "infer":
        share = max(case["mask"], 1.0 / n)
        by += 4.0 * n + 5.0 * n                     # predictions out; labels and mask in
        for l in range(L - 1, -1, -1):
            rows = n * share
            wider = min(1.0, share * (nnz / n))
            entries = nnz * min(1.0, share)
            product(rows, self_terms * d[l], d[1] if kind == "gin" else d[l + 1])           # weight gradient
            if kind == "gin":
                product(rows, d[1], d[l + 1])
                product(rows, d[1], d[l + 1])
            if l > 0:
                product(rows, d[l + 1] if kind != "gin" else d[1], self_terms * d[l])        # gradient of the layer's input
                aggregate(d[l] if kind in ("sage", "gin") else min(d[l], d[l + 1]), rows, n * wider, entries)
                by += n * wider * d[l] / 8.0                                                  # sign of the activation below
            share = wider
        by += sum(28.0 * a * b for a, b in zip(d, d[1:]))                                     # Adam: p, g, m, v in; p, m, v out
    if kind == "step_host":
        by += 4.0 * n * d[0] + 9.0 * n + sum(24.0 * a * b for a, b in zip(d, d[1:]))
    if case["dropout"]:
        by += sum(2.0 * n * w for w in d[1:-1])
    return dict(bytes=by, flops=fl)


def tolerance(case):
    """Sums in another order move a hidden pre-activation by its rounding error; where that crosses zero the ReLU mask of the
    backward pass flips, and each flip changes an entry of the gradient below by its whole value, so a gradient moves by about
    the square root of the share of flips (2e-7 of the entries at fp32: 4e-4).  Without a backward pass only the rounding of
    the sums remains.  Arg-max predictions may change where two scores are that close."""
    prec, kind = case["precision"], case["kind"]
    if kind == "propagate":
        return dict(rel=1e-5, max=1e-4)
    if kind == "infer":
        return dict(rel={"fp32": 1e-5, "tf32": 2e-3, "bf16": 1e-2}[prec], max={"fp32": 1e-3, "tf32": 5e-2, "bf16": 0.2}[prec])
    return dict(rel={"fp32": 1e-3, "tf32": 1e-2, "bf16": 2e-2}[prec], max={"fp32": 0.05, "tf32": 0.2, "bf16": 0.4}[prec],
                differ={"fp32": 1e-3, "tf32": 5e-3, "bf16": 1e-2}[prec])
