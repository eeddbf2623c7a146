"""Large fp32 products on the tensor cores, operands in three bf16 parts: either side of the tile, stage, accumulator and split
boundaries, with the whole epilogue, against fp64 and against the FMA kernel (which takes operands that are not aligned)."""
import pytest
import torch

from helpers import TOL_FP32
from paper_2501_01951_b200 import synth

pytestmark = pytest.mark.gpu


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


def device(t, ld):
    out = torch.full((t.shape[0], ld), float("nan"), device="cuda")      # what lies beyond the matrix is not read
    out[:, : t.shape[1]] = t
    return out


def up(x, aligned=True):
    return (x + 3) // 4 * 4 if aligned else x + 1 + (x % 2 == 1)


def product(mg, ctx, A, B, ta, tb, aligned=True, **epi):
    M, K, N = (A.shape[1], A.shape[0], 0) if ta else (*A.shape, 0)
    N = B.shape[0] if tb else B.shape[1]
    C = torch.full((M, up(N)), 3.0, device="cuda")
    mg.gemm(ctx, mg.PREC_FP32, ta, tb, M, N, K, device(A, up(A.shape[1], aligned)), device(B, up(B.shape[1], aligned)), C,
            **({"epi": mg.make_epilogue(**epi)} if epi else {}))
    assert torch.all(C[:, N:] == 3.0)
    return C[:, :N]


def error(got, want):
    return ((got.double() - want).norm() / want.norm()).item()


def operands(M, N, K, ta, tb, positive=False):
    lo = 0 if positive else -1
    return synth.uniform_tensor((K, M) if ta else (M, K), 31, lo, 1).cuda(), synth.uniform_tensor((N, K) if tb else (K, N), 32, lo, 1).cuda()


@pytest.mark.parametrize("M,N,K,ta", [
    (200000, 4, 64, False), (5000, 128, 256, False), (60000, 5, 300, False), (40, 40, 200000, True), (300, 5, 200001, True), (128, 128, 20011, True),
    (200001, 16, 127, False), (30000, 17, 1000, False), (100000, 129, 32, False), (500, 1000, 1023, False), (80001, 161, 33, False),
    (13000, 64, 512, False), (18943, 128, 168, False), (18945, 65, 330, False), (1300000, 40, 8, False), (1000, 1003, 1024, False),
    (32, 16, 800001, True), (33, 63, 200003, True), (129, 65, 50031, True), (128, 128, 24577, True), (501, 303, 2700, True), (1003, 1001, 401, True)])
@pytest.mark.parametrize("positive", [False, True])
def test_split_products(mg, ctx, M, N, K, ta, positive):
    for tb in ((False,) if ta else (False, True)):
        A, B = operands(M, N, K, ta, tb, positive)
        want = (A.T if ta else A).double() @ (B.T if tb else B).double()
        got, fma = product(mg, ctx, A, B, ta, tb), product(mg, ctx, A, B, ta, tb, aligned=False)
        assert error(got, want) <= TOL_FP32
        assert error(got, want) <= max(1.4 * error(fma, want), 7e-8)     # 6e-8 = one rounding to fp32


@pytest.mark.parametrize("M,N,K", [(60001, 40, 200), (30001, 161, 97), (9000, 300, 256)])
def test_split_epilogue(mg, ctx, M, N, K):
    A, B = operands(M, N, K, False, False)
    bias, drop = synth.uniform_tensor((N,), 33, -1, 1).cuda(), synth.bernoulli_mask(M * N, 0.5, 34).cuda()
    gate = synth.uniform_tensor((M, N), 35, -1, 1).cuda()
    words = (N + 31) // 32
    bits = torch.full((M, words + 1), -1, dtype=torch.int32, device="cuda")
    for relu in (False, True):                                           # under a ReLU the FMA kernel takes the product
        got = product(mg, ctx, A, B, False, False, bias=bias, relu=relu, drop_mask=drop, keep_scale=2.0, gate=device(gate, up(N)), gate_scale=0.5, sign_bits=bits)
        want = A.double() @ B.double() + bias.double()
        want = (torch.relu(want) if relu else want) * drop.reshape(M, N) * (gate > 0)
        assert error(got, want) <= TOL_FP32
        j = torch.arange(N, device="cuda")
        assert torch.equal((bits[:, j // 32] >> (j % 32)) & 1, (got > 0).int()) and torch.all(bits[:, words] == -1)


@pytest.mark.parametrize("ta", [False, True])
@pytest.mark.parametrize("where", ["A", "B"])
@pytest.mark.parametrize("value", [float("inf"), float("nan"), -3.4e38])
def test_operands_that_cannot_be_split(mg, ctx, ta, where, value):
    M, N, K = (200, 100, 25000) if ta else (25000, 100, 200)
    A, B = operands(M, N, K, ta, False)
    (A if where == "A" else B)[17, 5] = value
    bits = torch.zeros(M, (N + 31) // 32, dtype=torch.int32, device="cuda")
    epi = {} if ta else {"sign_bits": bits}
    got, bits_got = product(mg, ctx, A, B, ta, False, **epi), bits.clone()
    want = product(mg, ctx, A, B, ta, False, aligned=False, **epi)
    assert torch.equal(bits_got, bits) and torch.equal(got.isnan(), want.isnan()) and torch.equal(got.isinf(), want.isinf())
    ok = want.isfinite()
    assert error(got[ok] / 2.0**64, want[ok].double() / 2.0**64) <= TOL_FP32
    clean = operands(M, N, K, ta, False)                                 # the note of one product does not reach the next
    assert error(product(mg, ctx, *clean, ta, False), (clean[0].T if ta else clean[0]).double() @ clean[1].double()) <= TOL_FP32


@pytest.mark.parametrize("M,N,K", [(33, 63, 200003), (300, 17, 80001), (128, 65, 50000), (385, 161, 8193)])
def test_column_sums(mg, ctx, M, N, K):
    A, B = operands(M, N, K, True, False)
    C, sums = torch.zeros(M, up(N), device="cuda"), torch.full((N + 1,), 5.0, device="cuda")
    mg.weight_grad(ctx, mg.PREC_FP32, M, N, K, device(A, up(M)), device(B, up(N)), C, sums)
    assert error(C[:, :N], A.double().T @ B.double()) <= TOL_FP32
    assert (sums[:N].double() - B.double().sum(0)).abs().max() <= 1e-6 * B.double().abs().sum(0).max() and sums[N] == 5.0


def test_products_under_a_later_relu_keep_the_order_of_sums(mg, ctx):
    """Where a ReLU follows the aggregation of a product, every way to that product gives the FMA kernel's bits: GraphSAGE and GIN
    layers, a GCN layer, and its form on some rows only.  (The size is one the tensor cores take otherwise.)"""
    from paper_2501_01951_b200.sage_gin import GinTrainer, SageTrainer
    n, d, h = 20003, 300, 60
    g = mg.graph_create(ctx, n, *synth.rmat_graph(n, 60000, 41), mg.GRAPH_SYMMETRISE | mg.GRAPH_NORM_ROW)
    X = device(synth.uniform_tensor((n, d), 42, -1, 1), up(d)).nan_to_num()
    W = synth.uniform_tensor((d, h), 43, -1, 1).cuda()
    wide = torch.cat([W, -0.5 * W], 1).contiguous()
    fma = [torch.zeros(n, k, device="cuda") for k in (h, 2 * h)]
    for B, C in zip((W, wide), fma):
        mg.gemm(ctx, mg.PREC_FP32_FMA, False, False, n, C.shape[1], d, X, B, C)
        assert torch.equal(C, product(mg, ctx, X, B, False, False, aligned=False))
        assert not torch.equal(C, product(mg, ctx, X, B, False, False))
    y, m = synth.uniform_labels(n, 5, 44).cuda(), synth.bernoulli_mask(n, 0.3, 45).cuda()
    zero = [torch.zeros(h), torch.zeros(5)]

    want = torch.zeros(n, h, device="cuda")
    mg.spmm(ctx, g, fma[1][:, h:], want, h, epi=mg.make_epilogue(residual=fma[1][:, :h], residual_scale=1.0, relu=True))
    tr = SageTrainer(ctx, g, (d, h, 5), mg.PREC_FP32)
    tr.set_params([W, torch.zeros(h, 5)], [-0.5 * W, torch.zeros(h, 5)], zero)
    tr.set_inputs(X, y, m)
    tr.forward()
    assert tr.upd[0] and torch.equal(tr.S[1][:, :h], want)

    mg.spmm(ctx, g, fma[0], want, h, epi=mg.make_epilogue(residual=fma[0], residual_scale=1.25, relu=True))
    tr = GinTrainer(ctx, g, (d, 5), h, mg.PREC_FP32, gin_eps=0.25)
    tr.set_params([W], zero[:1], [torch.zeros(h, 5)], zero[1:])
    tr.set_inputs(X, y, m)
    tr.forward()
    assert tr.upd[0] and torch.equal(tr.T[0], want)

    mg.spmm(ctx, g, fma[0], want, h, epi=mg.make_epilogue(relu=True))
    desc = mg.layer_desc(d, h, up(d), h, h, mg.ORDER_UPD_FIRST, mg.PREC_FP32, mg.LAYER_RELU | mg.LAYER_FIRST)
    saved, out = torch.zeros(n, h, device="cuda"), torch.zeros(n, h, device="cuda")
    mg.layer_fwd(ctx, g, desc, X, W, None, None, saved, out)
    assert torch.equal(out, want)
    desc.flags |= mg.LAYER_OUT_ROWS_ONLY
    desc.gout_row_mask, desc.gout_row_count = m.data_ptr(), int(m.sum())
    mg.layer_fwd(ctx, g, desc, X, W, None, None, saved, out.fill_(-1.0))
    rows = m.bool()
    assert torch.equal(out[rows], want[rows]) and torch.all(out[~rows] == -1.0)


@pytest.mark.parametrize("precision,M,N,K,ta", [(0, 30001, 161, 97, False), (0, 128, 65, 50000, True), (2, 30001, 161, 97, False)])
def test_a_wait_that_runs_out_is_reported(mg, precision, M, N, K, ta):
    """The kernels that cut or convert fp32 operands, with the first load of every CTA left out and a short limit: the wait gives
    up, the status says so, and the products after it on the same context are right."""
    ctx = mg.ctx_create(0)
    A, B = (t.bfloat16().float() if precision == 2 else t for t in operands(M, N, K, ta, False))
    want = (A.T if ta else A).double() @ B.double()
    C = torch.zeros(M, up(N), device="cuda")
    call = lambda: mg.gemm(ctx, precision, ta, False, M, N, K, device(A, up(A.shape[1])), device(B, up(B.shape[1])), C)
    for _ in range(2):
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_WAIT_LIMIT, 2000)
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_DROP_LOAD, 2)
        call()
        assert mg.ctx_poll_status(ctx, raise_on_error=False) == 3
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_DROP_LOAD, 0)
        mg.ctx_set_option(ctx, mg.OPT_DEBUG_WAIT_LIMIT, 0)
        for _ in range(2):
            C.fill_(7.0)
            call()
            assert error(C[:, :N], want) <= TOL_FP32
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
    assert mg.ctx_gemm_paths(ctx)["tc_bf16"] == (6 if precision == 2 else 0)
    ctx.close()


def training_operands(kind, K, M, N):
    """A (K x M) and B (K x N) of a weight gradient: activations or bag-of-words features, and the gradient of a softmax loss over
    N classes (scores of the given spread, a share of the rows labelled) or one gated by a ReLU above it."""
    gen = torch.Generator(device="cuda").manual_seed(51)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")
    uniform = lambda *s: torch.rand(s, generator=gen, device="cuda")
    what, spread, share = kind
    p = torch.softmax(normal(K, N) * spread, 1)
    p[torch.arange(K, device="cuda"), torch.randint(0, N, (K,), generator=gen, device="cuda")] -= 1
    G = p * (uniform(K, 1) < share)
    if what == "words":
        return (uniform(K, M) < 0.02).float(), G
    H = torch.relu(normal(K, M))
    if what == "dropout":
        H = H * (uniform(K, M) < 0.5) * 2
    if what == "hidden":
        G = (G @ normal(N, N)) * (normal(K, N) > 0)
    return H, G


@pytest.mark.parametrize("kind", [("relu", 0.3, 0.54), ("relu", 4.0, 0.54), ("dropout", 4.0, 0.54), ("hidden", 1.0, 0.54), ("words", 4.0, 0.54), ("relu", 1.0, 0.01)])
@pytest.mark.parametrize("M,N,K", [(256, 40, 170003), (64, 47, 400000), (300, 172, 50001), (128, 80, 524288)])
def test_weight_gradients_of_training_lose_nothing(mg, ctx, kind, M, N, K):
    """No further from fp64 than the FMA kernel, down to one rounding of the result (2^-24).  The operands cancel as those of
    training do: most entries of a column of the gradient are small and of one sign, a few are large and of the other."""
    A, B = training_operands(kind, K, M, N)
    want = A.double().T @ B.double()
    got = {}
    for precision in (mg.PREC_FP32, mg.PREC_FP32_FMA):
        C = torch.zeros(M, up(N), device="cuda")
        mg.gemm(ctx, precision, True, False, M, N, K, device(A, up(M)), device(B, up(N)), C)
        got[precision] = C[:, :N]
    assert not torch.equal(*got.values())                                # the tensor cores did take it
    assert error(got[mg.PREC_FP32], want) <= max(error(got[mg.PREC_FP32_FMA], want), 2.0**-24)


@pytest.mark.parametrize("binades", [4, 10, 20])
@pytest.mark.parametrize("positive", [False, True])
@pytest.mark.parametrize("M,N,K,ta", [(20003, 128, 256, False), (30000, 64, 602, False), (256, 256, 100003, True), (128, 40, 50001, True)])
def test_split_products_of_spread_magnitudes(mg, ctx, binades, positive, M, N, K, ta):
    """Magnitudes over 2^-b .. 2^b inside every row and column, each element held to its own bound: an instruction of 16 terms cuts
    its terms off 24 bits below the largest of them (two instructions per accumulator in the K-major form, one in the other),
    and the fp32 sums behind it round once per accumulator (K / 32; 32 between two of the weight gradient's carries).  Four
    more for the small products, the parts left out, the sum over splits and the result.  The FMA kernel's own bound is
    K roundings, or 1024."""
    gen = torch.Generator(device="cuda").manual_seed(52)
    draw = lambda *s: ((torch.rand(s, generator=gen, device="cuda") if positive else torch.randn(s, generator=gen, device="cuda"))
                       * torch.exp2((torch.rand(s, generator=gen, device="cuda") * 2 - 1) * binades))
    A, B = draw(*((K, M) if ta else (M, K))), draw(K, N)
    got = product(mg, ctx, A, B, ta, False).double()
    a, b = (A.T if ta else A).double(), B.double()
    cuts, sums = (16, 32) if ta else (32, K // 32 + 1)
    assert torch.all((got - a @ b).abs() <= (cuts + sums + 4) * 2.0**-24 * (a.abs() @ b.abs()))


@pytest.mark.parametrize("M,N,K,ta", [(25000, 100, 200, False), (25000, 17, 200, False), (200, 100, 25000, True), (200, 17, 200001, True)])
def test_sums_that_overflow(mg, ctx, M, N, K, ta):
    """Finite operands whose products or sums leave fp32's range: the infinities (and the NaN of opposite ones) of the FMA kernel."""
    A, B = operands(M, N, K, ta, False)
    rows = A.T if ta else A
    rows[3], rows[5], B[7] = 1e30, 3e37, 1e10                            # of one row of the result a product, of another the sum
    clean = operands(M, N, K, ta, False)
    bits = torch.zeros(M, (N + 31) // 32, dtype=torch.int32, device="cuda")
    epi = {} if ta else {"sign_bits": bits}
    got, bits_got = product(mg, ctx, A, B, ta, False, **epi), bits.clone()
    want = product(mg, ctx, A, B, ta, False, aligned=False, **epi)
    assert want.isinf().any()
    assert torch.equal(got.isnan(), want.isnan()) and torch.equal(got.isinf(), want.isinf()) and torch.equal(bits_got, bits)
    ok = want.isfinite()
    assert torch.equal(got[ok], want[ok])
    assert error(product(mg, ctx, *clean, ta, False), (clean[0].T if ta else clean[0]).double() @ clean[1].double()) <= TOL_FP32
