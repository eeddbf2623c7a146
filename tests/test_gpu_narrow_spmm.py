"""Narrow aggregations (one warp per unit, at most 64 columns), segment lengths of small graphs and the block-wide
combination of hub rows, against the oracle: rows on either side of every boundary (12 entries, the segment length,
2,048 entries), widths on either side of every lane split."""
import numpy as np
import pytest
import torch

from helpers import TOL_FP32, rel_fro
from oracle import gcn_oracle as orc
from paper_2501_01951_b200 import synth

pytestmark = pytest.mark.gpu

LENGTHS = (1, 2, 3, 11, 12, 13, 14, 31, 33, 63, 64, 65, 66, 127, 129, 511, 512, 513, 514, 2046, 2047, 2048, 2049, 4999)


@pytest.fixture(scope="module")
def mg():
    from paper_2501_01951_b200 import build
    build.build()
    from paper_2501_01951_b200 import binding
    return binding


@pytest.fixture(scope="module")
def problem(mg):
    """Directed graph whose first rows have exactly the LENGTHS (the diagonal among them)."""
    n = 5000
    rng = np.random.default_rng(3)
    s, d = [], []
    for u, k in enumerate(LENGTHS):
        others = np.setdiff1d(rng.permutation(n), [u], assume_unique=False)
        s.append(np.full(k - 1, u)); d.append(rng.permutation(others)[: k - 1])
    s, d = np.concatenate(s), np.concatenate(d)
    go = orc.graph_build(n, s, d, flags=orc.ADD_SELF_LOOPS)
    assert tuple(np.diff(go.rowptr)[: len(LENGTHS)]) == LENGTHS
    ctx = mg.ctx_create(0)
    g = mg.graph_create(ctx, n, torch.tensor(s, dtype=torch.int32), torch.tensor(d, dtype=torch.int32), mg.GRAPH_ADD_SELF_LOOPS)
    yield ctx, g, go
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
    g.close(); ctx.close()


@pytest.mark.parametrize("w", [1, 4, 5, 8, 9, 16, 17, 24, 25, 32, 33, 47, 48, 49, 64, 65, 200])
def test_narrow_aggregation(mg, problem, w):
    ctx, g, go = problem
    n, ld = go.n, (w + 3) // 4 * 4
    X = synth.uniform_tensor((n, w), 70 + w, -1, 1)
    b = synth.uniform_tensor((w,), 71 + w, -0.5, 0.5)
    Y = torch.zeros(n, ld, device="cuda"); Y[:, :w] = X.cuda()
    Z = torch.full((n, ld), 9.0, device="cuda")
    want = orc.aggregate(go, X.numpy())
    rows = slice(0, len(LENGTHS))
    for epi, f in ((None, lambda z: z), (dict(bias=b.cuda(), relu=True), lambda z: np.maximum(z + b.numpy(), 0.0)),
                   (dict(residual=Y, residual_scale=0.5, bias=b.cuda()), lambda z: z + 0.5 * X.numpy() + b.numpy())):
        mg.spmm(ctx, g, Y, Z, w, epi=None if epi is None else mg.make_epilogue(**epi))
        got = Z[:, :w].cpu().numpy().astype(np.float64)
        assert rel_fro(got, f(want)) <= TOL_FP32 and rel_fro(got[rows], f(want)[rows]) <= TOL_FP32
        assert torch.all(Z[:, w:] == 0)
    mg.spmm(ctx, g, Y, Z, w, transposed=True)
    assert rel_fro(Z[:, :w].cpu().numpy().astype(np.float64), orc.aggregate(go, X.numpy(), transposed=True)) <= TOL_FP32


@pytest.mark.parametrize("n", [1 << 20, (1 << 20) + 1])
def test_column_blocks_of_large_graphs(mg, n):
    """Either side of the size from which long rows are cut into more column blocks."""
    lengths = (127, 128, 129, 255, 256, 257, 513, 3000)
    gen = torch.Generator(device="cuda").manual_seed(5)
    dst = torch.cat([torch.randperm(n, generator=gen, device="cuda")[:k] for k in lengths]).int()
    src = torch.cat([torch.full((k,), 100 * u + 7, dtype=torch.int32, device="cuda") for u, k in enumerate(lengths)])
    ctx = mg.ctx_create(0)
    g = mg.graph_create(ctx, n, src, dst, mg.GRAPH_NORM_NONE)
    for w in (12, 100):
        Y, Z = torch.randn(n, w, generator=gen, device="cuda"), torch.full((n, w), 9.0, device="cuda")
        mg.spmm(ctx, g, Y, Z, w)
        want = torch.zeros(n, w, dtype=torch.float64, device="cuda").index_add_(0, src.long(), Y.double()[dst.long()])
        assert rel_fro(Z.double().cpu().numpy(), want.cpu().numpy()) <= TOL_FP32
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
    g.close(); ctx.close()


@pytest.mark.parametrize("w", [65, 68, 93, 96, 97, 129, 132, 157, 192, 193])
def test_three_float4_a_lane(w):
    """Widths on either side of where lanes hold three float4: every column is the one that a wider call (two or four float4 a lane, entries in
    the same order) computes, bit for bit, in every bucket of rows and for segments of long rows, with the lean and the general epilogue."""
    from paper_2501_01951_b200 import binding as mg, synth
    ctx = mg.ctx_create(0)
    try:
        n = 30011
        src, dst = synth.rmat_graph(n, 400_000, 17)
        g = mg.graph_create(ctx, n, src, dst)
        gen = torch.Generator(device="cuda").manual_seed(w)
        wide = 256 if w > 128 else 128
        Y = torch.randn((n, wide), generator=gen, device="cuda")
        bias, gate = torch.randn(wide, generator=gen, device="cuda"), torch.randn((n, wide), generator=gen, device="cuda")
        ld = (w + 3) // 4 * 4
        Yn = torch.full((n, ld), float("nan"), device="cuda")
        Yn[:, :w] = Y[:, :w]
        for epi in (lambda c: None, lambda c: mg.make_epilogue(bias=bias[:c].clone(), relu=True),
                    lambda c: mg.make_epilogue(gate=gate[:, :c].contiguous() if c % 4 == 0 else torch.nn.functional.pad(gate[:, :c], (0, ld - w)), gate_scale=2.0),
                    lambda c: mg.make_epilogue(residual=gate, residual_scale=0.5)):
            a, b = torch.full((n, wide), 3.0, device="cuda"), torch.full((n, ld), 3.0, device="cuda")
            ea, eb = epi(wide), epi(w)
            mg.spmm(ctx, g, Y, a, wide, epi=ea)
            mg.spmm(ctx, g, Yn, b, w, epi=eb)
            assert torch.equal(a[:, :w], b[:, :w])
        g.close()
        assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
    finally:
        ctx.close()
