"""weight_grad (A^T B with B's column sums from the same pass) where one, two and three rows of tiles share the sums, and
GraphSAGE / GIN whose first layer aggregates after its product, against the oracle."""
import numpy as np
import pytest
import torch

from helpers import ADAM, TOL_FP32, padded, rel_fro, round4
from oracle import gcn_oracle as orc
from paper_2501_01951_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    from paper_2501_01951_b200 import build
    build.build()
    from paper_2501_01951_b200 import binding
    return binding


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("M,N,K", [(4, 4, 1), (30, 7, 31), (128, 33, 257), (129, 256, 5000), (300, 100, 33333), (256, 300, 70001)])
def test_weight_and_bias_gradient(mg, prec, M, N, K):
    ctx = mg.ctx_create(0)
    A, B = synth.uniform_tensor((K, M), 41, -1, 1), synth.uniform_tensor((K, N), 42, -1, 1)
    C, cs = torch.zeros(M, round4(N), device="cuda"), torch.full((N + 1,), 5.0, device="cuda")
    mg.weight_grad(ctx, prec, M, N, K, padded(A), padded(B), C, cs)
    cut = {0: lambda t: t.double(), 1: lambda t: (t.contiguous().view(torch.int32) & -8192).view(torch.float32).double(), 2: lambda t: t.to(torch.bfloat16).double()}[prec]
    assert rel_fro(C[:, :N].cpu().numpy(), (cut(A).T @ cut(B)).numpy()) <= (TOL_FP32 if prec == 0 else 2e-5)
    want = B.double().sum(0).numpy()
    assert np.abs(cs[:N].cpu().numpy() - want).max() <= 1e-6 * B.double().abs().sum(0).max().item() and cs[N].item() == 5.0
    with pytest.raises(mg.MixgcnError):
        mg.weight_grad(ctx, prec, M, N, K, padded(A), padded(B)[:, 1:], C, cs)
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
    ctx.close()


@pytest.mark.parametrize("kind", ["sage", "gin"])
def test_first_layer_updates_first(mg, kind):
    from paper_2501_01951_b200.sage_gin import GinTrainer, SageTrainer
    dims, L, hidden, n = (64, 10, 21, 6), 3, 12, 3000
    s, d = synth.rmat_graph(n, 15000, 8)
    X, y, m = synth.uniform_tensor((n, 64), 1, -1, 1), synth.uniform_labels(n, 6, 2), synth.bernoulli_mask(n, 0.3, 3)
    go = orc.graph_build(n, s.numpy(), d.numpy(), orc.SYMMETRISE, norm="row" if kind == "sage" else "none")
    ctx = mg.ctx_create(0)
    gg = mg.graph_create(ctx, n, s, d, mg.GRAPH_SYMMETRISE | (mg.GRAPH_NORM_ROW if kind == "sage" else mg.GRAPH_NORM_NONE))
    npl = lambda lst: [t.numpy() for t in lst]
    bias = lambda k, w: [synth.uniform_tensor((x,), k + i, -0.1, 0.1) for i, x in enumerate(w)]
    if kind == "sage":
        Ws, Wn = ([synth.glorot_uniform(a, b, k + a) for a, b in zip(dims, dims[1:])] for k in (500, 600))
        b = bias(700, dims[1:])
        tr = SageTrainer(ctx, gg, dims, mg.PREC_FP32)
        tr.set_params(Ws, Wn, b)
        ref = orc.sage_epoch(go, X.numpy(), npl(Ws), npl(Wn), npl(b), y.numpy(), m.numpy(), None, 1, **ADAM)
    else:
        W1 = [synth.glorot_uniform(a, hidden, 500 + a) * 0.1 for a in dims[:-1]]
        W2 = [synth.glorot_uniform(hidden, a, 600 + a) * 0.3 for a in dims[1:]]
        b1, b2 = bias(700, [hidden] * L), bias(800, dims[1:])
        tr = GinTrainer(ctx, gg, dims, hidden, mg.PREC_FP32, gin_eps=0.25)
        tr.set_params(W1, b1, W2, b2)
        ref = orc.gin_epoch(go, X.numpy(), npl(W1), npl(b1), npl(W2), npl(b2), y.numpy(), m.numpy(), 0.25, None, 1, **ADAM)
    assert tr.upd[0] and not tr.upd[1]
    tr.set_inputs(padded(X), y.cuda(), m.cuda())
    for _ in range(2):                                    # twice: nothing of the first pass is left over
        tr.forward()
        assert rel_fro(tr.logits[:, :6].cpu().numpy(), ref["logits"]) <= TOL_FP32
        tr.compute_loss(); tr.backward()
    if kind == "gin":
        for i in range(4 * L):
            assert rel_fro(tr.grads[i].cpu().numpy(), ref["grads"][i]) <= 2 * TOL_FP32, i
    else:
        for l in range(L):
            g, dl, ld = tr.grads[l].cpu().numpy(), dims[l], round4(dims[l])
            assert rel_fro(g[:dl], ref["grads"][l]) <= TOL_FP32 and rel_fro(g[ld:ld + dl], ref["grads"][L + l]) <= TOL_FP32
            assert rel_fro(tr.grads[L + l].cpu().numpy(), ref["grads"][2 * L + l]) <= TOL_FP32
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
