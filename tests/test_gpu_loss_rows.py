"""Loss of one row per 8, 16 or 32 lanes: widths on either side of every lane split and of the kernels' choice, pitches with and without room,
row counts that leave warps partly empty, few and many train rows; against fp64."""
import pytest
import torch

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


@pytest.mark.parametrize("C", [1, 3, 4, 8, 29, 32, 33, 61, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("n,share", [(1, 1.0), (33, 0.5), (5003, 0.02), (150003, 0.6)])
@pytest.mark.parametrize("room,in_place", [(0, True), (8, False)])
def test_rows(mg, ctx, C, n, share, room, in_place):
    gen = torch.Generator(device="cuda").manual_seed(C * 7 + n)
    ld = (C + 3) // 4 * 4 + room
    full = torch.full((n, ld), float("nan"), device="cuda")        # what lies beyond the columns and their pad is neither read nor written
    full[:, :(C + 3) // 4 * 4] = 0
    x = torch.randn((n, C), generator=gen, device="cuda") * 3
    x[:, C // 2] = x[:, 0]                                          # equal maxima: the lowest index counts
    full[:, :C] = x
    y = torch.randint(0, C, (n,), generator=gen, device="cuda", dtype=torch.int32)
    m = (torch.rand(n, generator=gen, device="cuda") < share).to(torch.uint8)
    m[0] = 1
    out = full if in_place else torch.full_like(full, 5.0)
    loss, pred, good = torch.zeros(1, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"), torch.full((1,), 9, dtype=torch.int64, device="cuda")
    mg.loss_softmax_xent(ctx, full, y, m, loss, dlogits=out, pred=pred, n_correct=good, C_=C)
    x64, rows = x.double(), m.bool()
    T = int(m.sum())
    want = (torch.softmax(x64, 1) - torch.nn.functional.one_hot(y.long(), C)) / T * rows[:, None]
    ref = -torch.log_softmax(x64, 1).gather(1, y.long()[:, None])[rows].mean()
    # exp(x - lse): lse lies below 16 and is rounded to 2^-21 of it or less (4.8e-7), the difference likewise, exp by two units (1.2e-7 each): a
    # softmax is off by 1.2e-6 of itself at most, and where one is subtracted from it by 6e-8 more
    p64 = torch.softmax(x64, 1) * rows[:, None] / T
    assert torch.linalg.norm(out[:, :C].double() - want) <= 1.3e-6 * torch.linalg.norm(p64)
    assert abs(loss.item() - ref.item()) <= 2e-6 * abs(ref.item()) + 1e-6
    best = (x == x.max(1, keepdim=True).values).int().argmax(1).int()
    assert torch.equal(pred, best) and good.item() == int(((best == y) & rows).sum())
    if room:
        assert torch.isnan(full[:, -room:]).all() and (out[:, -room:] == 5.0).all()


@pytest.mark.parametrize("C", [16, 17, 48, 49, 96, 97, 192, 193, 257, 300, 384, 385, 512, 513])
@pytest.mark.parametrize("n,share", [(1, 1.0), (9, 0.5), (5003, 0.02), (40_003, 0.6)])
def test_rows_at_the_lane_splits(mg, ctx, C, n, share):
    test_rows(mg, ctx, C, n, share, 0, True)
    test_rows(mg, ctx, C, n, share, 4, False)


@pytest.mark.parametrize("C", [5, 47, 100, 172, 300])
def test_rows_without_numbers(mg, ctx, C):
    """NaN among numbers, nothing but NaN, infinities: the prediction ignores NaN, is the lowest column where there is nothing else; loss and
    gradient of the other rows stay as they are."""
    n, ld = 64, (C + 3) // 4 * 4
    x = torch.randn((n, ld), device="cuda")
    y, m = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.ones(n, dtype=torch.uint8, device="cuda")
    m[:8] = 0
    outs = []
    for odd in (False, True):
        if odd:
            x[0, :] = float("nan")
            x[1, 0] = float("nan")
            x[2, C - 1] = float("inf")
            x[3, :] = float("-inf")
        full, loss, pred = x.clone(), torch.zeros(1, device="cuda"), torch.full((n,), 7, dtype=torch.int32, device="cuda")
        mg.loss_softmax_xent(ctx, full, y, m, loss, dlogits=full, pred=pred, C_=C)
        outs.append((full[:, :C].clone(), loss.clone(), pred.clone()))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1]) and torch.equal(outs[0][2][4:], outs[1][2][4:])
    assert outs[1][2][:4].tolist() == [0, 1 + int(x[1, 1:C].argmax()), C - 1, 0]
