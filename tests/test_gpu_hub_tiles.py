"""Aggregation with the dense corner of the graph on the tensor cores (graph_prepare_tiles): widths either side of chunks, halves, lane
splits and slices, every normalisation and orientation, the epilogues, rows that lie in tiles only, values the tensor core cannot take.

Against fp64: a result is a sum of fp32 sums of at most 512 terms each, so its error stays below 512 units of rounding of the sum of the
terms' absolute values in the worst case, and near sqrt(512) units (1.3e-6 of it) where the terms' signs do not matter; 4e-7 of the 2-norm is
what rounding to nearest gives on average (0.29 units per addition, a third of it for sums that grow)."""
import pytest
import torch

from paper_2501_01951_b200 import synth

pytestmark = pytest.mark.gpu
N, CORE = 9001, 4099


@pytest.fixture(scope="module")
def mg():
    from paper_2501_01951_b200 import build
    build.build()
    from paper_2501_01951_b200 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(mg):
    c = mg.ctx_create(0)
    yield c
    assert mg.ctx_poll_status(c, raise_on_error=False) == 0
    c.close()


def edges(seed):
    """A dense core of CORE nodes, ids scattered over [0, N), the first 300 of them joined to one another only; a sparse rest that leaves some
    nodes without neighbours."""
    gen = torch.Generator().manual_seed(seed)
    ids = torch.randperm(N, generator=gen)
    core = torch.randint(0, CORE, (2, 6_000_000), generator=gen)
    clique = torch.combinations(torch.arange(300)).T
    core = core[:, (core >= 300).all(0)]
    rest = torch.randint(300, N - 50, (2, 60_000), generator=gen)
    e = ids[torch.cat([core, clique, rest], 1)].int()
    return e[0].contiguous(), e[1].contiguous()


def matrix(mg, g, transposed):
    ex = mg.graph_export(g, transposed)
    return torch.sparse_csr_tensor(ex["rowptr"], ex["col"].long(), ex["val"].double(), (g.n, g.n)).cuda()


def features(w, seed, positive=False):
    Y = torch.full((N, (w + 3) // 4 * 4), float("nan"), device="cuda")        # what lies beyond the columns is not read
    Y[:, :w] = synth.uniform_tensor((N, w), seed, 0 if positive else -1, 1).cuda()
    return Y


@pytest.fixture(scope="module")
def graphs(mg, ctx):
    """{(norm, symmetric): (plain graph, graph with tiles, its matrices)}"""
    out = {}
    for norm, flags in (("sym", 0), ("row", mg.GRAPH_NORM_ROW), ("none", mg.GRAPH_NORM_NONE)):
        for symmetric in (True, False):
            fl = flags | (mg.GRAPH_SYMMETRISE if symmetric else 0) | (mg.GRAPH_ADD_SELF_LOOPS if norm == "sym" else 0)
            src, dst = edges(1)
            plain, tiled = (mg.graph_create(ctx, N, src, dst, fl) for _ in range(2))
            tiles, entries = mg.graph_prepare_tiles(tiled)
            assert tiles > 100 and entries > tiled.nnz // 2
            assert mg.graph_prepare_tiles(tiled) == (tiles, entries)
            out[norm, symmetric] = plain, tiled, [matrix(mg, tiled, t) for t in (False, True)]
    yield out
    for plain, tiled, _ in out.values():
        plain.close(), tiled.close()


@pytest.mark.parametrize("w", [1, 5, 16, 33, 47, 64, 65, 100, 128, 129, 160, 253, 256, 257, 300, 600])
@pytest.mark.parametrize("norm,symmetric,transposed", [("sym", True, False), ("sym", False, True), ("row", True, False), ("row", False, False),
                                                       ("none", False, False), ("none", False, True)])
def test_sums_against_fp64(mg, ctx, graphs, norm, symmetric, transposed, w):
    plain, tiled, A = graphs[norm, symmetric]
    for positive in (False, True):
        Y = features(w, 7, positive)
        Z, Zp = (torch.full_like(Y, 3.0) for _ in range(2))
        mg.spmm(ctx, tiled, Y, Z, w, transposed)
        mg.spmm(ctx, plain, Y, Zp, w, transposed)
        assert not torch.equal(Z, Zp)                                        # the tiles' kernels ran: sums in another order
        want = A[transposed] @ Y[:, :w].double()
        bound = 512 * 2.0 ** -24 * (A[transposed] @ Y[:, :w].double().abs())
        assert torch.all((Z[:, :w].double() - want).abs() <= bound)
        err, err_plain = (((z[:, :w].double() - want).norm() / want.norm()).item() for z in (Z, Zp))
        print(f"{norm} {symmetric} {transposed} w {w} positive {positive}: {err:.2e} gathered {err_plain:.2e}")
        assert err < 4e-7
        assert torch.all(Z[:, w:] == 0)
        again = torch.empty_like(Z)
        mg.spmm(ctx, tiled, Y, again, w, transposed)
        assert torch.equal(Z, again)


@pytest.mark.parametrize("w", [41, 128, 256, 260])
def test_epilogues_and_slices(mg, ctx, graphs, w):
    plain, tiled, _ = graphs["sym", True]
    ld, words = (w + 3) // 4 * 4, (w + 31) // 32
    Y = features(w, 3)
    t = lambda seed: synth.uniform_tensor((N, ld), seed, -1, 1).cuda()
    bits = torch.randint(-2 ** 31, 2 ** 31 - 1, (N, words), dtype=torch.int32, device="cuda")
    drop = (t(5)[:, :w] > 0).to(torch.uint8).contiguous()
    for epi in (dict(bias=t(4)[0, :w].contiguous(), relu=True), dict(gate=t(6), gate_scale=2.0), dict(gate_bits=bits, gate_scale=1.5),
                dict(residual=t(8), residual_scale=0.5, relu=True), dict(drop_mask=drop, keep_scale=2.0, bias=t(4)[0, :w].contiguous())):
        Z, Zp = (torch.full_like(Y, 3.0) for _ in range(2))
        mg.spmm(ctx, tiled, Y, Z, w, epi=mg.make_epilogue(**epi))
        mg.spmm(ctx, plain, Y, Zp, w, epi=mg.make_epilogue(**epi))
        assert (Z - Zp).abs().max() <= 2e-6 * Zp.abs().max()                  # two fp32 sums of the same terms
    whole, sliced = torch.empty_like(Y), torch.empty_like(Y)
    mg.spmm(ctx, tiled, Y, whole, w)
    for cols in (16, 100, 512):
        mg.ctx_set_option(ctx, mg.OPT_SPMM_SLICE_COLS, cols)
        mg.spmm(ctx, tiled, Y, sliced, w)
        mg.ctx_set_option(ctx, mg.OPT_SPMM_SLICE_COLS, 0)
        assert (whole - sliced).abs().max() <= 2e-6 * whole.abs().max()


@pytest.mark.parametrize("w", [47, 256])
def test_values_that_the_parts_cannot_hold(mg, ctx, graphs, w):
    """Infinities, NaN and numbers near the largest reach the same outputs as on the gather kernels, and no call after it."""
    plain, tiled, _ = graphs["none", True]
    hubs = mg.graph_degrees(tiled).argsort(descending=True)
    for value in (float("inf"), float("nan"), 3e38, -2e30, None, None):
        Y = features(w, 9)
        if value is not None:
            Y[hubs[700], w // 2] = value
        Z, Zp = (torch.empty_like(Y) for _ in range(2))
        mg.spmm(ctx, tiled, Y, Z, w)
        mg.spmm(ctx, plain, Y, Zp, w)
        Z, Zp = Z[:, :w], Zp[:, :w]
        assert torch.equal(torch.isnan(Z), torch.isnan(Zp)) and torch.equal(torch.isinf(Z), torch.isinf(Zp))
        fine = torch.isfinite(Zp)
        assert ((Z - Zp)[fine].abs() <= 2e-6 * Zp[fine].abs().max()).all()


def test_numbers_of_every_size(mg, ctx, graphs):
    """Columns from 1e-30 to 1e30 come out to the same relative error; zeros and whole numbers exactly."""
    _, tiled, A = graphs["none", True]
    w = 64
    Y = features(w, 11, True) * 10.0 ** torch.linspace(-30, 26, w, device="cuda")
    Y[:, 0] = 0
    Y[:, 1:3] = (Y[:, 1:3] * 1e30 * 5).round()
    Z = torch.empty_like(Y)
    mg.spmm(ctx, tiled, Y, Z, w)
    want = A[0] @ Y.double()
    assert torch.all(((Z.double() - want).norm(dim=0) <= 4e-7 * want.norm(dim=0)))
    assert torch.equal(Z[:, :3].double(), want[:, :3])


@pytest.mark.parametrize("w", [1, 16, 33, 65, 100, 256, 300])
@pytest.mark.parametrize("binades", [6, 12, 20, 38, 44, 68, 80])
def test_numbers_far_apart(mg, ctx, graphs, w, binades):
    """One row in fifty `binades` above the others: one, two and three passes of four digits, and more than they reach.  A term loses half a unit
    of the last pass at most, 2^-31, 2^-62 or 2^-93 of the largest, used up to 9, 40 and 71 binades: 2^-22 of the others' size, inside the bound
    of the sums."""
    plain, tiled, A = graphs["none", False]
    Y = features(w, 13)
    Y *= torch.where(torch.rand((N, 1), generator=torch.Generator().manual_seed(w)) < 0.02, 2.0 ** binades, 1.0).cuda()
    Z = torch.empty_like(Y)
    mg.spmm(ctx, tiled, Y, Z, w)
    want = A[0] @ Y[:, :w].double()
    assert torch.all((Z[:, :w].double() - want).abs() <= 512 * 2.0 ** -24 * (A[0] @ Y[:, :w].double().abs()))
    assert ((Z[:, :w].double() - want).norm() / want.norm()).item() < 4e-7


def test_a_wait_that_runs_out_is_reported(mg, ctx, graphs):
    _, tiled, _ = graphs["sym", True]
    Y, Z = features(256, 3), torch.empty((N, 256), device="cuda")
    mg.ctx_set_option(ctx, mg.OPT_DEBUG_WAIT_LIMIT, 2000)
    mg.ctx_set_option(ctx, mg.OPT_DEBUG_DROP_LOAD, 1)
    try:
        mg.spmm(ctx, tiled, Y, Z, 256)
        assert mg.ctx_poll_status(ctx, raise_on_error=False) == 3
    finally:
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_DROP_LOAD, 0)
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_WAIT_LIMIT, 0)
    want = torch.empty_like(Z)
    mg.spmm(ctx, tiled, Y, Z, 256)
    mg.spmm(ctx, graphs["sym", True][0], Y, want, 256)
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0 and (Z - want).abs().max() <= 2e-6 * want.abs().max()


def test_row_means_transposed_stay_with_the_gather_kernels(mg, ctx, graphs):
    plain, tiled, _ = graphs["row", True]
    Y, Z, Zp = features(100, 3), torch.empty((N, 100), device="cuda"), torch.empty((N, 100), device="cuda")
    mg.spmm(ctx, tiled, Y, Z, 100, True)
    mg.spmm(ctx, plain, Y, Zp, 100, True)
    assert torch.equal(Z, Zp)


def test_small_and_sparse_graphs_have_no_tiles(mg, ctx):
    for n, m in ((2000, 30_000), (400_000, 1_500_000)):
        gen = torch.Generator().manual_seed(n)
        e = torch.randint(0, n, (2, m), generator=gen, dtype=torch.int32)
        g = mg.graph_create(ctx, n, e[0].contiguous(), e[1].contiguous())
        assert mg.graph_prepare_tiles(g) == (0, 0)
        g.close()


@pytest.mark.parametrize("products", [1, 3])
def test_a_value_that_the_parts_cannot_hold_leaves_nothing_to_later_replays(mg, ctx, graphs, products):
    """Recordings with one and with three products: a replay whose last input held an infinity, then replays of the finite inputs, which
    give the bits of the calls; calls after a recording as well."""
    _, tiled, _ = graphs["sym", True]
    hub = mg.graph_degrees(tiled).argsort(descending=True)[700]
    Ys = [features(256, 20 + k) for k in range(products)]
    Zs = [torch.empty_like(Y) for Y in Ys]

    def calls():
        for Y, Z in zip(Ys, Zs):
            mg.spmm(ctx, tiled, Y, Z, 256)

    calls()
    want = [Z.clone() for Z in Zs]
    rec = mg.record(ctx, calls)
    assert rec.replay()
    kept = Ys[-1][hub].clone()
    Ys[-1][hub, 9] = float("inf")
    assert rec.replay()
    Ys[-1][hub] = kept
    for again in (rec.replay, rec.replay, calls):
        for Z in Zs:
            Z.zero_()
        again()
        assert all(torch.equal(Z, w) for Z, w in zip(Zs, want))
    rec.close()


@pytest.mark.parametrize("norm", ["sym", "none"])
def test_the_smallest_numbers_keep_their_bits(mg, ctx, graphs, norm):
    """Columns from 1e-38, where terms fall below fp32's normal range, up to 1e22, the largest that the parts hold: no further from fp64
    than the gather kernels, a tenth for the noise of one draw."""
    plain, tiled, A = graphs[norm, True]
    w = 64
    Y = features(w, 12) * 10.0 ** torch.linspace(-38, 22, w, device="cuda")
    Z, Zp = (torch.empty_like(Y) for _ in range(2))
    mg.spmm(ctx, tiled, Y, Z, w)
    mg.spmm(ctx, plain, Y, Zp, w)
    want = A[0] @ Y.double()
    err, err_plain = ((z.double() - want).norm(dim=0) for z in (Z, Zp))
    assert torch.all(err <= 1.1 * err_plain), (err / err_plain)


def spreads(n, w, seed):
    """Signed, of one sign, half zeros as behind a ReLU, and the first two with a row in a thousand 2^15 times the others."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((n, w), generator=gen, device="cuda")
    few = 1 + 2.0 ** 15 * (torch.rand((n, 1), generator=gen, device="cuda") < 0.001)
    return dict(signed=x, positive=x.abs(), relu=x.relu(), signed_mixed=x * few, positive_mixed=x.abs() * few)


def compare_errors(mg, ctx, plain, tiled, A, w, transposed=False):
    """The 2-norm of the error against fp64 is no larger than the gather kernels', but for a tenth: summed over ten draws, since with a few
    large rows one draw's ratio lies anywhere between half and twice that."""
    err = {}
    for seed in range(10):
        for name, Y in spreads(tiled.n, w, seed).items():
            want = A @ Y.double()
            for g in (tiled, plain):
                Z = torch.empty_like(Y)
                mg.spmm(ctx, g, Y, Z, w, transposed)
                err[name, g is tiled] = err.get((name, g is tiled), 0.0) + ((Z.double() - want).norm() / want.norm()).item()
    for name in spreads(8, 1, 0):
        print(f"w {w} {name}: {err[name, True] / 10:.2e} gathered {err[name, False] / 10:.2e} ratio {err[name, True] / err[name, False]:.2f}")
        assert err[name, True] <= 1.1 * err[name, False], name


@pytest.mark.parametrize("w", [64, 128, 160, 256])
@pytest.mark.parametrize("norm,symmetric,transposed", [("sym", True, False), ("row", True, False), ("none", False, False), ("none", False, True)])
def test_error_no_larger_than_the_gather_kernels(mg, ctx, graphs, norm, symmetric, transposed, w):
    plain, tiled, A = graphs[norm, symmetric]
    compare_errors(mg, ctx, plain, tiled, A[transposed], w, transposed)


@pytest.mark.parametrize("n,edges,flag", [(300_000, 4_650_000, 0), (60_000, 12_000_000, 0), (60_000, 12_000_000, "GRAPH_NORM_NONE")])
def test_error_on_graphs_with_hubs(mg, ctx, n, edges, flag):
    """Rows whose sums are mostly the rest of the matrix; rows of tiles of many pieces, whose sums the hubs decide."""
    src, dst = synth.rmat_graph(n, edges, 3, device="cuda")
    flags = mg.GRAPH_SYMMETRISE | (getattr(mg, flag) if flag else mg.GRAPH_ADD_SELF_LOOPS)
    plain, tiled = (mg.graph_create(ctx, n, src, dst, flags) for _ in range(2))
    assert mg.graph_prepare_tiles(tiled)[0] > 500
    compare_errors(mg, ctx, plain, tiled, matrix(mg, tiled, False), 132)
    plain.close(), tiled.close()


def test_a_layout_that_runs_out_of_memory_leaves_the_graph_as_it_was(mg, ctx, graphs):
    """Each allocation of the layout made to fail in turn (what has been enqueued until then is still writing to the blocks it got), a
    fresh graph every time, both orientations."""
    plain, _, _ = graphs["sym", False]
    src, dst = edges(1)
    Y, Z, Zp = features(100, 3), torch.empty((N, 100), device="cuda"), torch.empty((N, 100), device="cuda")
    mg.spmm(ctx, plain, Y, Zp, 100)
    failed = 0
    for k in range(1, 100):
        g = mg.graph_create(ctx, N, src, dst, mg.GRAPH_ADD_SELF_LOOPS)
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_FAIL_ALLOC, k)
        tiles = mg.graph_prepare_tiles(g)[0]
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_FAIL_ALLOC, 0)
        other = mg.graph_create(ctx, N, src, dst, mg.GRAPH_ADD_SELF_LOOPS)        # takes the memory that came back
        mg.spmm(ctx, other, Y, Z, 100)
        assert torch.equal(Z, Zp)
        mg.spmm(ctx, g, Y, Z, 100)
        assert torch.equal(Z, Zp) == (tiles == 0)
        g.close(), other.close()
        if tiles:
            break
        failed += 1
    assert 20 < failed < 90


@pytest.mark.parametrize("kind", ["gcn", "sage", "gin"])
def test_trainers_do_without_tiles_where_there_is_no_memory_for_them(mg, ctx, kind):
    from paper_2501_01951_b200.sage_gin import GinTrainer, SageTrainer
    from paper_2501_01951_b200.train import GcnTrainer
    make = dict(gcn=GcnTrainer, sage=SageTrainer, gin=GinTrainer)[kind]
    src, dst = edges(1)
    flags = mg.GRAPH_SYMMETRISE | dict(gcn=mg.GRAPH_ADD_SELF_LOOPS, sage=mg.GRAPH_NORM_ROW, gin=mg.GRAPH_NORM_NONE)[kind]
    for k in (1, 9, 20):
        g = mg.graph_create(ctx, N, src, dst, flags)
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_FAIL_ALLOC, k)
        make(ctx, g, (64, 128, 16), *([128] if kind == "gin" else []), mg.PREC_TF32)
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_FAIL_ALLOC, 0)
        assert mg.graph_prepare_tiles(g) == (0, 0)
        g.close()


@pytest.mark.parametrize("w", [100, 300])
def test_an_aggregation_without_memory_for_its_tiles_gathers(mg, graphs, w):
    plain, tiled, _ = graphs["sym", False]
    ctx = mg.ctx_create(0)
    Y = features(w, 3)
    Z, Zp, Zt = (torch.empty_like(Y) for _ in range(3))
    mg.ctx_set_option(ctx, mg.OPT_DEBUG_FAIL_ALLOC, 1)
    mg.spmm(ctx, tiled, Y, Z, w)
    mg.spmm(ctx, plain, Y, Zp, w)
    assert torch.equal(Z, Zp)
    mg.spmm(ctx, tiled, Y, Zt, w)
    assert not torch.equal(Zt, Zp) and (Zt - Zp).abs().max() <= 2e-6 * Zp.abs().max()
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
    ctx.close()


def iteration(mg, ctx, g, kind, precision, dims=(64, 128, 16), **kwargs):
    """Forward, loss and backward of a new trainer: logits, loss, predictions, gradients."""
    from paper_2501_01951_b200.sage_gin import GinTrainer, SageTrainer
    from paper_2501_01951_b200.train import GcnTrainer
    u = lambda *shape: synth.uniform_tensor(shape, sum(shape), -0.3, 0.3)
    pairs = list(zip(dims, dims[1:]))
    Ws, bs = [u(*p) for p in pairs], [u(p[1]) for p in pairs]
    if kind == "gcn":
        tr = GcnTrainer(ctx, g, dims, precision, **kwargs)
        tr.set_params(Ws, bs)
    elif kind == "sage":
        tr = SageTrainer(ctx, g, dims, precision)
        tr.set_params(Ws, [w + 0.1 for w in Ws], bs)
    else:
        tr = GinTrainer(ctx, g, dims, 96, precision)
        tr.set_params([u(d, 96) for d in dims[:-1]], [u(96) for _ in pairs], [u(96, d) for d in dims[1:]], bs)
    gen = torch.Generator().manual_seed(5)
    labels = torch.randint(0, dims[-1], (N,), generator=gen, dtype=torch.int32)
    mask = (torch.rand(N, generator=gen) < 0.3).to(torch.uint8)
    tr.set_inputs(features(dims[0], 3), labels.cuda(), mask.cuda())
    tr.forward()
    logits = (tr.X[-1] if kind == "gcn" else tr.logits)[:, :dims[-1]].clone()
    tr.compute_loss(), tr.backward()
    return [logits, tr.loss.clone(), tr.pred.clone()] + [t.clone() for t in (tr.dW + tr.db if kind == "gcn" else tr.grads)]


@pytest.mark.parametrize("kind", ["gcn", "sage", "gin"])
def test_who_else_uses_a_graph_changes_no_sums(mg, ctx, kind):
    """fp32 trainers, trainers in chunks and plain aggregations give the same bits before and after a trainer that takes the tiles is made on
    their graph, and so do recordings and their calls; the other way round it keeps its own."""
    src, dst = edges(1)
    flags = mg.GRAPH_SYMMETRISE | dict(gcn=mg.GRAPH_ADD_SELF_LOOPS, sage=mg.GRAPH_NORM_ROW, gin=mg.GRAPH_NORM_NONE)[kind]
    g, alone = (mg.graph_create(ctx, N, src, dst, flags) for _ in range(2))
    Y, Z = features(128, 3), torch.empty((N, 128), device="cuda")

    def others():
        mg.spmm(ctx, g, Y, Z, 128)
        return [Z.clone(), *iteration(mg, ctx, g, kind, mg.PREC_FP32), *(iteration(mg, ctx, g, kind, mg.PREC_TF32, n_chunks=3) if kind == "gcn" else [])]

    low = iteration(mg, ctx, alone, kind, mg.PREC_TF32)
    before = others()
    rec = mg.record(ctx, lambda: mg.spmm(ctx, g, Y, Z, 128))
    assert all(torch.equal(a, b) for a, b in zip(low, iteration(mg, ctx, g, kind, mg.PREC_TF32)))
    assert mg.graph_layout_tiles(g)[0] > 100
    assert all(torch.equal(a, b) for a, b in zip(before, others()))
    assert rec.replay() and torch.equal(Z, before[0])
    assert all(torch.equal(a, b) for a, b in zip(low, iteration(mg, ctx, g, kind, mg.PREC_TF32)))
    # asked for on the graph itself, plain aggregations take the tiles, and their recordings end
    mg.graph_prepare_tiles(g)
    assert not rec.replay()
    mg.spmm(ctx, g, Y, Z, 128)
    assert not torch.equal(Z, before[0])
    for t, same in ((False, True), (True, False)):
        mg.spmm(ctx, g, Y, Z, 128, tiles=t)
        assert torch.equal(Z, before[0]) == same
    assert all(torch.equal(a, b) for a, b in zip(before[1:], iteration(mg, ctx, g, kind, mg.PREC_FP32)))
    rec.close(), g.close(), alone.close()


def test_tiles_are_laid_out_for_the_widths_that_will_be_used(mg):
    """A graph whose tiles pay at 132 columns and not at 64: a trainer of narrow layers has none built, a later one of wider layers has, with
    the scratch of its aggregations set aside (none of them allocates)."""
    ctx = mg.ctx_create(0)
    n = 300_000
    src, dst = synth.rmat_graph(n, 4_650_000, 3, device="cuda")
    g = mg.graph_create(ctx, n, src, dst)
    assert mg.graph_layout_tiles(g, [64, 3]) == (0, 0) and mg.graph_layout_tiles(g, [64], ctx) == (0, 0)
    tiles, entries = mg.graph_layout_tiles(g, [64, 132], ctx)
    assert tiles > 500 and mg.graph_layout_tiles(g) == (tiles, entries)
    Y, Z, Zp = (torch.randn((n, 132), device="cuda") for _ in range(3))
    mg.ctx_set_option(ctx, mg.OPT_DEBUG_FAIL_ALLOC, 1)
    mg.spmm(ctx, g, Y, Z, 132, tiles=True)
    mg.ctx_set_option(ctx, mg.OPT_DEBUG_FAIL_ALLOC, 0)
    mg.spmm(ctx, g, Y, Zp, 132, tiles=False)
    assert not torch.equal(Z, Zp) and (Z - Zp).abs().max() <= 4e-6 * Zp.abs().max()
    g.close(), ctx.close()


@pytest.mark.parametrize("w", [96, 100, 161, 260, 300])
def test_sums_do_not_depend_on_the_slices(mg, ctx, graphs, w):
    """Slices below, at and above the widths at which the kernels' lane splits and the product's accumulators change."""
    _, tiled, _ = graphs["sym", True]
    Y, want = features(w, 5), torch.empty((N, (w + 3) // 4 * 4), device="cuda")
    mg.spmm(ctx, tiled, Y, want, w)
    for cols in (32, 64, 100, 128, 1024):
        Z = torch.full_like(want, 7.0)
        mg.ctx_set_option(ctx, mg.OPT_SPMM_SLICE_COLS, cols)
        try:
            mg.spmm(ctx, tiled, Y, Z, w)
        finally:
            mg.ctx_set_option(ctx, mg.OPT_SPMM_SLICE_COLS, 0)
        assert torch.equal(Z, want), cols


def gcn(mg, ctx, g, dims, precision, **kwargs):
    from paper_2501_01951_b200.train import GcnTrainer
    u = lambda *shape: synth.uniform_tensor(shape, sum(shape), -0.3, 0.3)
    tr = GcnTrainer(ctx, g, dims, precision, **kwargs)
    tr.set_params([u(*p) for p in zip(dims, dims[1:])], [u(d) for d in dims[1:]])
    gen = torch.Generator().manual_seed(5)
    tr.set_inputs(features(dims[0], 3), torch.randint(0, dims[-1], (N,), generator=gen, dtype=torch.int32).cuda(),
                  (torch.rand(N, generator=gen) < 0.3).to(torch.uint8).cuda())
    return tr


@pytest.mark.parametrize("classes", [3, 16, 41, 65, 100, 128, 200, 256])
def test_the_loss_inside_an_aggregation_with_tiles(mg, ctx, graphs, classes):
    """Narrow, one, two and three float4 a lane: predictions, loss and gradient as from the logits of the separate calls; without tiles the
    same to rounding (a probability moves with its logit, by less than 2e-6 of the largest)."""
    tr = gcn(mg, ctx, graphs["sym", True][1], (64, 96, classes), mg.PREC_TF32, order=[mg.ORDER_AUTO, mg.ORDER_UPD_FIRST])
    tr.forward()
    tr.compute_loss()
    want = [t.clone() for t in (tr.pred, tr.loss, tr.X[-1])]
    tr.forward_and_loss()
    assert torch.equal(tr.pred, want[0])
    assert abs(tr.loss.item() - want[1].item()) <= 2e-6 * want[1].item()
    assert (tr.X[-1] - want[2]).abs().max() <= 2e-6 * want[2].abs().max()
    with_tiles = tr.X[-1].clone()
    tr.descs[-1].flags &= ~mg.LAYER_TILES
    tr.forward_and_loss()
    assert not torch.equal(tr.X[-1], with_tiles) and (tr.X[-1] - with_tiles).abs().max() <= 1e-5 * with_tiles.abs().max()


def test_bf16_copies_beside_tiles(mg, ctx, graphs):
    """Those of A_hat X (aggregate first) and of a layer's output (update first)."""
    tiled = graphs["sym", True][1]
    tr = gcn(mg, ctx, tiled, (64, 128, 100), mg.PREC_BF16, order=mg.ORDER_AGG_FIRST, saved_lp_only=False)
    tr.forward()
    for l in range(2):
        assert torch.equal(tr.saved_lp[l][:, :tr.dims[l]], tr.saved[l][:, :tr.dims[l]].bfloat16())
    tr = gcn(mg, ctx, tiled, (64, 128, 100), mg.PREC_BF16, order=mg.ORDER_UPD_FIRST)
    tr.forward()
    copy = next(t for t in tr.lp if t.data_ptr() == tr.descs[0].x_out_lp)
    assert torch.equal(copy[:, :128], tr.X[1][:, :128].bfloat16())


@pytest.mark.parametrize("precision", ["PREC_TF32", "PREC_BF16"])
def test_recorded_iterations_with_tiles(mg, ctx, graphs, precision):
    """Epochs, replayed from the third on, against the calls one by one: the same weights."""
    a, b = (gcn(mg, ctx, graphs["sym", True][1], (64, 128, 41), getattr(mg, precision)) for _ in range(2))
    for t in range(1, 6):
        a.epoch(t)
        b.forward_and_loss(), b.backward(), b.step(t)
    assert a._replays["iteration"].rec is not None
    assert all(torch.equal(x, y) for x, y in zip(a.W + a.b, b.W + b.b))
