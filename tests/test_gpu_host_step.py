"""train_step_host with features whose rows are padded on the device (odd widths on either side of a warp's 128 columns), one to
three layers, with and without announced features, against the trainer on device buffers, bit for bit."""
import pytest
import torch

from helpers import ADAM, padded
from paper_2501_01951_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    from paper_2501_01951_b200 import build
    build.build()
    from paper_2501_01951_b200 import binding
    return binding


@pytest.mark.parametrize("dims", [(1, 3), (7, 16, 3), (127, 33, 5), (128, 20, 20, 4), (129, 64, 6), (301, 40, 12, 7)])
@pytest.mark.parametrize("announce", [False, True])
def test_host_iterations_are_the_device_ones(mg, dims, announce):
    from paper_2501_01951_b200.train import GcnTrainer
    n, L = 2003, len(dims) - 1
    s, d = synth.rmat_graph(n, 9000, 4)
    feats = [synth.uniform_tensor((n, dims[0]), 50 + i, -1, 1).pin_memory() for i in range(3)]
    y, m = synth.uniform_labels(n, dims[-1], 2), synth.bernoulli_mask(n, 0.3, 3)
    Ws = [synth.glorot_uniform(a, b, 500 + a) for a, b in zip(dims, dims[1:])]
    bs = [synth.uniform_tensor((b,), 600 + i, -0.1, 0.1) for i, b in enumerate(dims[1:])]
    ctx, host_ctx = mg.ctx_create(0), mg.ctx_create(0)
    tr = GcnTrainer(ctx, mg.graph_create(ctx, n, s, d), dims, mg.PREC_FP32)
    tr.set_params(Ws, bs)
    g = mg.graph_create(host_ctx, n, s, d)
    W, b = [w.clone() for w in Ws], [x.clone() for x in bs]
    z = lambda lst: [torch.zeros_like(x) for x in lst]
    mW, vW, mb, vb = z(W), z(W), z(b), z(b)
    pred = torch.zeros(n, dtype=torch.int32).pin_memory()
    for t, X in enumerate(feats, start=1):
        tr.set_inputs(padded(X), y.cuda(), m.cuda())
        tr.forward_and_loss(); tr.backward(); tr.step(t, **ADAM)
        if announce and t < len(feats):
            mg.train_step_host_prefetch(host_ctx, feats[t])
        loss = mg.train_step_host(host_ctx, g, dims, mg.PREC_FP32, X, y, m, W, b, mW, vW, mb, vb, t, pred=pred, **ADAM)
        assert loss == tr.loss.item() and torch.equal(pred, tr.pred.cpu())
        for l in range(L):
            assert torch.equal(W[l], tr.W[l].cpu()) and torch.equal(vW[l], tr.vW[l].cpu()) and torch.equal(mb[l], tr.mb[l].cpu())
    assert mg.ctx_poll_status(host_ctx, raise_on_error=False) == 0
