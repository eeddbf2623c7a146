"""Recorded iterations: what epoch() and forward() replay is bit for bit what the calls give, through every change that must
end a recording -- other buffers, options, profiling, scratch that moved -- and the refusals."""
import pytest
import torch

from helpers import padded
from paper_2501_01951_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    from paper_2501_01951_b200 import build
    build.build()
    from paper_2501_01951_b200 import binding
    return binding


def trainer(mg, precision, dims=(40, 24, 24, 9), **kw):
    from paper_2501_01951_b200.train import GcnTrainer
    n = 3000
    s, d = synth.rmat_graph(n, 20000, 5)
    ctx = mg.ctx_create(0)
    g = mg.graph_create(ctx, n, s, d)
    tr = GcnTrainer(ctx, g, dims, precision, **kw)
    tr.set_params([synth.glorot_uniform(a, b, 7 + a) for a, b in zip(dims, dims[1:])], [torch.zeros(b) for b in dims[1:]])
    tr.set_inputs(padded(synth.uniform_tensor((n, dims[0]), 3, -1, 1)), synth.uniform_labels(n, 9, 4).cuda(), synth.bernoulli_mask(n, kw.pop("mask", 0.3), 6).cuda())
    return ctx, g, tr


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("kw", [{}, dict(row_sparse=1), dict(row_sparse=2, row_plans=False), dict(train_rows_only=True), dict(cache_first_aggregation=True), dict(n_chunks=3)])
def test_replayed_iterations_are_the_calls(mg, precision, kw):
    a, b = trainer(mg, precision, **kw), trainer(mg, precision, **kw)
    for t in range(1, 9):
        if t == 5:                                    # other parameter buffers: the recording ends
            for _, _, tr in (a, b):
                tr.W[1] = tr.W[1].clone()
        if t == 7:                                    # scratch of the context moves
            for ctx, _, _ in (a, b):
                mg.ctx_reserve(ctx, 64 << 20)
        a[2].epoch(t)
        b[2]._iteration()
        b[2].step(t)
    assert a[2]._replays["iteration"].rec is not None
    for x, y in zip(a[2].W + a[2].b + a[2].dW + a[2].mW + [a[2].loss, a[2].pred], b[2].W + b[2].b + b[2].dW + b[2].mW + [b[2].loss, b[2].pred]):
        assert torch.equal(x, y)
    for _ in range(3):
        a[2].forward()
    b[2]._forward()
    assert torch.equal(a[2].X[-1], b[2].X[-1])
    for ctx, _, _ in (a, b):
        assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0


def replays_like_calls(a, b, ts):
    """Iterations of trainer `a` through epoch(), of its twin `b` call by call: the same bits."""
    for t in ts:
        a.epoch(t)
        b._iteration()
        b.step(t)
    for x, y in zip(a.W + a.b + a.dW + a.mW + [a.loss, a.pred], b.W + b.b + b.dW + b.mW + [b.loss, b.pred]):
        assert torch.equal(x, y)
    assert a._replays["iteration"].rec is not None


@pytest.mark.parametrize("dims", [(64, 24, 24, 9), (64, 24, 9), (16, 24, 9)])     # first layer updates first, or aggregates first
@pytest.mark.parametrize("change", ["inputs", "row_sparse"])
def test_recording_ends_with_the_row_plans_it_used(mg, dims, change):
    """Row plans made anew may lie where the old ones lay, under an equal key."""
    a, b = trainer(mg, mg.PREC_FP32, dims=dims, row_sparse=1)[2], trainer(mg, mg.PREC_FP32, dims=dims, row_sparse=1)[2]
    replays_like_calls(a, b, range(1, 5))
    perm = torch.randperm(a.n, generator=torch.Generator().manual_seed(8)).cuda()
    for k in range(3):
        for tr in (a, b):
            tr.train_mask.copy_(tr.train_mask[perm])              # other nodes, as many, in the same buffers
            if change == "inputs":
                tr.set_inputs(tr.X[0], tr.labels, tr.train_mask)
            else:
                tr.configure(row_sparse=1)
        replays_like_calls(a, b, range(5 + 4 * k, 9 + 4 * k))
    for tr in (a, b):
        assert mg.ctx_poll_status(tr.ctx, raise_on_error=False) == 0


def test_recording_ends_with_the_chunk_schedules_it_used(mg):
    """Two trainers share a graph and cut its rows into different numbers of chunks: each one's calls replace the other's schedules."""
    ctx, g, a = trainer(mg, mg.PREC_FP32, n_chunks=3)
    b, twin = trainer(mg, mg.PREC_FP32, n_chunks=3)[2], trainer(mg, mg.PREC_FP32, n_chunks=5)[2]
    other = type(a)(ctx, g, a.dims, mg.PREC_FP32, n_chunks=5)
    other.set_params(twin.W, twin.b)
    other.set_inputs(a.X[0], a.labels, a.train_mask)
    replays_like_calls(a, b, range(1, 5))
    rec = a._replays["iteration"].rec
    replays_like_calls(other, twin, range(1, 5))
    assert not rec.replay()
    replays_like_calls(a, b, range(5, 9))
    assert a._replays["iteration"].rec is not rec
    torch.cuda.synchronize()
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0


@pytest.mark.parametrize("gone", ["plan", "graph"])
def test_replay_is_refused_once_a_graph_or_plan_is_gone(mg, gone):
    ctx, g, tr = trainer(mg, mg.PREC_FP32)
    plan = mg.rowplan_create(ctx, g, tr.train_mask)
    Y, Z = torch.ones((plan.in_count, 8), device="cuda"), torch.zeros((g.n, 8), device="cuda")
    calls = (lambda: mg.spmm_rowplan(ctx, plan, Y, Z, 8)) if gone == "plan" else (lambda: mg.spmm(ctx, g, tr.X[0], tr.saved[0], 8))
    bits = torch.zeros((g.n, 1), dtype=torch.int32, device="cuda")
    calls()
    rec, other = mg.record(ctx, calls), mg.record(ctx, lambda: mg.mask_pack(ctx, 8, bits, X=Z))
    assert rec.replay() and other.replay()
    plan.close()
    if gone == "graph":
        g.close()
    assert not rec.replay() and other.replay()
    torch.cuda.synchronize()
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0


def test_launches_are_counted_and_profiling_sees_every_kernel(mg):
    ctx, g, tr = trainer(mg, mg.PREC_TF32)
    total = lambda: mg.ctx_profile_read(ctx)[2]
    counts = []
    for t in range(1, 6):
        before, paths = total(), mg.ctx_gemm_paths(ctx)["tc_tf32"]
        tr.epoch(t)
        counts.append((total() - before, mg.ctx_gemm_paths(ctx)["tc_tf32"] - paths))
    assert counts[-1] == counts[1] and counts[1][0] > 10 and tr._replays["iteration"].rec is not None
    mg.ctx_profile_enable(ctx, True)
    mg.ctx_profile_read(ctx)
    tr.epoch(6)
    ms, launches, _ = mg.ctx_profile_read(ctx)
    mg.ctx_profile_enable(ctx, False)
    assert launches["spmm"] > 0 and ms["spmm"] > 0
    tr.epoch(7)
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0


def test_recording_is_refused_where_calls_would_allocate(mg):
    ctx, g, tr = trainer(mg, mg.PREC_FP32)
    assert mg.record(ctx, lambda: mg.ctx_reserve(ctx, 1 << 28)) is None
    tr.epoch(1)                                       # the context goes on
    rec = mg.record(ctx, tr._iteration)
    assert rec is not None and rec.replay()
    mg.ctx_set_option(ctx, mg.OPT_SPMM_SLICE_COLS, 8)
    assert not rec.replay()
    mg.ctx_set_option(ctx, mg.OPT_SPMM_SLICE_COLS, 0)
    assert rec.replay()
    torch.cuda.synchronize()
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
