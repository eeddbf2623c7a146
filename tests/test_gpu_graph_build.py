"""Graph construction where its key width and its segment tables change: node counts around 2^15 and 2^16 (one 32-bit key
holds two ids below), with and without dropped edges, directed and symmetrised, hub rows of several hundred segments."""
import numpy as np
import pytest
import torch

from helpers import TOL_FP32, rel_fro
from oracle import gcn_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    from paper_2501_01951_b200 import build
    build.build()
    from paper_2501_01951_b200 import binding
    return binding


@pytest.mark.parametrize("n", [1, 2, 32767, 32768, 65535, 65536, 65537])
@pytest.mark.parametrize("sym,dropped", [(True, True), (True, False), (False, True)])
def test_csr_and_schedule(mg, n, sym, dropped):
    rng = np.random.default_rng(n)
    m = 40 if n < 10 else 60000
    s, d = rng.integers(0, n, m), rng.integers(0, n, m)
    hub = np.arange(0, n, 3) if n > 10 else np.zeros(0, np.int64)      # node n-1 is a hub
    s, d = np.concatenate([s, np.full(len(hub), n - 1)]), np.concatenate([d, hub])
    if not dropped:
        keep = s != d
        s, d = s[keep], d[keep]
    flags = (mg.GRAPH_SYMMETRISE if sym else 0) | mg.GRAPH_ADD_SELF_LOOPS
    go = orc.graph_build(n, s, d, flags=(orc.SYMMETRISE if sym else 0) | orc.ADD_SELF_LOOPS)
    ctx = mg.ctx_create(0)
    g = mg.graph_create(ctx, n, torch.tensor(s, dtype=torch.int32).cuda(), torch.tensor(d, dtype=torch.int32).cuda(), flags)
    for t, (rp, col) in ((False, (go.rowptr, go.col)), (True, (go.rowptr_t, go.col_t))):
        ex = mg.graph_export(g, transposed=t)
        assert np.array_equal(ex["rowptr"].numpy(), rp) and np.array_equal(ex["col"].numpy(), col)
    deg = np.diff(go.rowptr)
    assert g.nnz == len(go.col) and g.max_deg == deg.max()
    perm = mg.graph_export_schedule(g).numpy()
    assert np.array_equal(perm, np.lexsort((np.arange(n), -deg)))
    X = rng.standard_normal((n, 20)).astype(np.float32)
    Y = torch.tensor(X).cuda(); Z = torch.zeros_like(Y)
    for t in (False, True):
        mg.spmm(ctx, g, Y, Z, 20, transposed=t)
        assert rel_fro(Z.cpu().numpy(), orc.aggregate(go, X, transposed=t)) <= TOL_FP32
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
    g.close(); ctx.close()


def pairs_with_rows(rng, n, rows):
    """Directed edges: row u has `count` entries, some of them twice, the columns from a range of `span` ids."""
    src, dst = [], []
    for u, count, span in rows:
        lo = rng.integers(0, n - span + 1)
        cols = lo + rng.choice(span, min(count, span), replace=False)
        cols = np.concatenate([cols, cols[: len(cols) // 3]])
        src.append(np.full(len(cols), u)), dst.append(cols)
    s, d = np.concatenate(src), np.concatenate(dst)
    order = rng.permutation(len(s))
    return s[order], d[order]


@pytest.mark.parametrize("n,rows", [
    # rows around a bin's eight entries, a warp's 32 and 128, and rows whose columns lie close together (large bins)
    (40_000, [(3 + 7 * i, c, sp) for i, (c, sp) in enumerate([(1, 1), (7, 9000), (8, 9), (9, 9000), (31, 31), (33, 40), (64, 40_000), (127, 128), (128, 128), (129, 200), (300, 40_000),
                                                              (1000, 1024), (1025, 40_000), (5000, 5000)])]),
    # more than a bucket has room for: one row, several, and more than are worth bitmaps (the radix sort)
    (300_000, [(17, 13_000, 300_000)]),
    (70_001, [(u, 9000 + u, 70_001) for u in range(12)]),
    (70_001, [(0, 65_000, 70_001), (1, 70_001, 70_001), (2, 12_288, 12_288), (3, 2048, 2048), (4, 2049, 70_001)]),
    # ids of more than 20 bits have no bitmap
    ((1 << 20) + 5, [(9, 20_000, 1 << 20), (10, 100, 1 << 20)]),
    (1 << 20, [(9, 20_000, 1 << 20), ((1 << 20) - 1, 15_000, 1 << 20)]),
])
@pytest.mark.parametrize("sym,loops", [(False, False), (True, True)])
def test_rows_of_every_length(mg, n, rows, sym, loops):
    """Rows, degrees and values as numpy's sorted sets and fp32 give them."""
    rng = np.random.default_rng(len(rows))
    s, d = pairs_with_rows(rng, n, rows)
    ctx = mg.ctx_create(0)
    g = mg.graph_create(ctx, n, torch.tensor(s, dtype=torch.int32).cuda(), torch.tensor(d, dtype=torch.int32).cuda(),
                        (mg.GRAPH_SYMMETRISE if sym else 0) | (mg.GRAPH_ADD_SELF_LOOPS if loops else 0))
    keep = s != d
    u, v = s[keep].astype(np.int64), d[keep].astype(np.int64)
    if sym:
        u, v = np.concatenate([u, v]), np.concatenate([v, u])
    if loops:
        u, v = np.concatenate([u, np.arange(n)]), np.concatenate([v, np.arange(n)])
    keys = np.unique(u * n + v)
    ex = mg.graph_export(g)
    deg = np.bincount(keys // n, minlength=n)
    assert np.array_equal(ex["col"].numpy(), keys % n) and np.array_equal(np.diff(ex["rowptr"].numpy()), deg)
    assert np.array_equal(ex["deg"].numpy(), deg)
    with np.errstate(divide="ignore"):
        dinv = np.where(deg > 0, np.float32(1) / np.sqrt(deg.astype(np.float32)), np.float32(0)).astype(np.float32)
    assert np.array_equal(ex["dinv"].numpy(), dinv) and np.array_equal(ex["val"].numpy(), dinv[keys // n] * dinv[keys % n])
    g.close(); ctx.close()
