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
