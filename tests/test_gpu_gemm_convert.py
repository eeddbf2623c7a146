"""bf16 products of fp32 rows that come without a bf16 copy: converted inside the kernel, on either side of its tile, chunk and
stage boundaries, with the whole epilogue, against the fp64 product of the rounded operands."""
import pytest
import torch

from helpers import round4
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


def device(t):
    out = torch.full((t.shape[0], round4(t.shape[1])), float("nan"), device="cuda")
    out[:, : t.shape[1]] = t.cuda()
    return out


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (127, 16, 31), (128, 17, 32), (129, 32, 33), (20001, 33, 63), (19000, 65, 301), (40000, 130, 64),
                                   (300, 255, 512), (300, 255, 513), (50001, 256, 65), (300, 257, 65)])
@pytest.mark.parametrize("tb", [False, True])
def test_products_of_unconverted_rows(mg, ctx, M, N, K, tb):
    A, B = synth.uniform_tensor((M, K), 61, -1, 1), synth.uniform_tensor((N, K) if tb else (K, N), 62, -1, 1)
    bias, drop, gate = synth.uniform_tensor((N,), 63, -1, 1), synth.bernoulli_mask(M * N, 0.5, 64), synth.uniform_tensor((M, N), 65, -1, 1)
    words = (N + 31) // 32
    bits = torch.full((M, words + 1), -1, dtype=torch.int32, device="cuda")
    C = torch.zeros(M, round4(N), device="cuda")
    b16 = lambda t: t.to(torch.bfloat16).double().cuda()
    want = b16(A) @ (b16(B).T if tb else b16(B))
    before = mg.ctx_gemm_paths(ctx)["tc_bf16"]
    mg.gemm(ctx, mg.PREC_BF16, False, tb, M, N, K, device(A), device(B), C)
    assert mg.ctx_gemm_paths(ctx)["tc_bf16"] == before + 1
    assert (C[:, :N].double() - want).norm() <= 2e-5 * want.norm()
    mg.gemm(ctx, mg.PREC_BF16, False, tb, M, N, K, device(A), device(B), C,
            epi=mg.make_epilogue(bias=bias.cuda(), relu=True, drop_mask=drop.cuda(), keep_scale=2.0, gate=device(gate), gate_scale=0.5, sign_bits=bits))
    got = C[:, :N]
    y = torch.relu(want + bias.double().cuda()) * drop.cuda().reshape(M, N) * (gate.cuda() > 0)
    assert (got.double() - y).norm() <= 2e-5 * max(y.norm().item(), 1e-3)
    j = torch.arange(N, device="cuda")
    assert torch.equal((bits[:, j // 32] >> (j % 32)) & 1, (got > 0).int()) and torch.all(bits[:, words] == -1)
