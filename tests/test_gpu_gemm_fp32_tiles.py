"""fp32 FMA products on either side of the tile, k-step, split and flush boundaries, in every operand form, aligned and
not, with the whole epilogue, against fp64."""
import numpy as np
import pytest
import torch

from helpers import TOL_FP32, rel_fro
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
    out = torch.zeros(t.shape[0], ld, device="cuda")
    out[:, : t.shape[1]] = t.cuda()
    return out


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (63, 31, 15), (64, 32, 16), (65, 33, 17), (127, 64, 33), (129, 65, 128), (40000, 129, 48),
                                   (20001, 63, 70), (300, 200, 1023), (19000, 128, 1025), (257, 40, 2100), (9000, 7, 1300)])
@pytest.mark.parametrize("ta,tb", [(False, False), (False, True), (True, False), (True, True)])
@pytest.mark.parametrize("aligned", [True, False])
def test_tiles(mg, ctx, M, N, K, ta, tb, aligned):
    if M > 10000 and (ta or K > 1000) and not aligned:
        pytest.skip("the large shapes once")
    A = synth.uniform_tensor((K, M) if ta else (M, K), 21, -1, 1)
    B = synth.uniform_tensor((N, K) if tb else (K, N), 22, -1, 1)
    up = (lambda x: (x + 3) // 4 * 4) if aligned else (lambda x: x + 1 + (x % 2 == 1))     # odd leading dimensions
    Ad, Bd = device(A, up(A.shape[1])), device(B, up(B.shape[1]))
    a64, b64 = A.numpy().astype(np.float64), B.numpy().astype(np.float64)
    want = (a64.T if ta else a64) @ (b64.T if tb else b64)
    C = torch.full((M, up(N)), 3.0, device="cuda")
    mg.gemm(ctx, mg.PREC_FP32, ta, tb, M, N, K, Ad, Bd, C)
    assert rel_fro(C[:, :N].cpu().numpy(), want) <= TOL_FP32 and torch.all(C[:, N:] == 3.0)
    if ta:
        return
    bias, drop, gate = synth.uniform_tensor((N,), 23, -1, 1), synth.bernoulli_mask(M * N, 0.5, 24), synth.uniform_tensor((M, N), 25, -1, 1)
    words = (N + 31) // 32
    bits = torch.full((M, words + 1), -1, dtype=torch.int32, device="cuda")
    mg.gemm(ctx, mg.PREC_FP32, ta, tb, M, N, K, Ad, Bd, C,
            epi=mg.make_epilogue(bias=bias.cuda(), relu=True, drop_mask=drop.cuda(), keep_scale=2.0, gate=device(gate, up(N)), gate_scale=0.5, sign_bits=bits))
    y = np.maximum(want + bias.numpy(), 0.0) * drop.numpy().reshape(M, N) * 2.0 * (gate.numpy() > 0) * 0.5
    got = C[:, :N].cpu().numpy()
    assert rel_fro(got, y) <= TOL_FP32
    packed = np.zeros((M, words * 32), dtype=np.uint32)
    packed[:, :N] = got > 0
    packed = (packed.reshape(M, words, 32) << np.arange(32, dtype=np.uint32)).sum(axis=2, dtype=np.uint32)
    assert np.array_equal(bits[:, :words].cpu().numpy().view(np.uint32), packed) and torch.all(bits[:, words] == -1)


@pytest.mark.parametrize("M,N,K", [(1, 16, 1), (63, 32, 15), (65, 48, 17), (130, 40, 40), (129, 128, 33), (20001, 128, 70), (9000, 100, 20), (257, 256, 1100)])
@pytest.mark.parametrize("offset", [0, 4, 1])
def test_dropout_masks(mg, ctx, M, N, K, offset):
    """Masks that are copied 16 and 4 bytes at a time beside the k-steps, and those that are not: rows that start at multiples of 16, of 4 and at odd bytes."""
    A, B = synth.uniform_tensor((M, K), 31, -1, 1), synth.uniform_tensor((K, N), 32, -1, 1)
    drop = synth.bernoulli_mask(M * N, 0.5, 33)
    at = torch.full((M * N + 16,), 255, dtype=torch.uint8, device="cuda")
    at[offset:offset + M * N] = drop.cuda()
    up = (N + 3) // 4 * 4
    C = torch.full((M, up), 3.0, device="cuda")
    mg.gemm(ctx, mg.PREC_FP32, False, False, M, N, K, device(A, (K + 3) // 4 * 4), device(B, up), C,
            epi=mg.make_epilogue(relu=True, drop_mask=at[offset:offset + M * N], keep_scale=2.0))
    want = np.maximum(A.numpy().astype(np.float64) @ B.numpy().astype(np.float64), 0.0) * drop.numpy().reshape(M, N) * 2.0
    got = C[:, :N].cpu().numpy()
    assert rel_fro(got, want) <= TOL_FP32 and not np.any(got[drop.numpy().reshape(M, N) == 0])
