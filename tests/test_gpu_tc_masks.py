"""Dropout masks, fp32 gates and bit gates of the tensor-core products' epilogues: aligned and byte-ragged widths, tiles of
one to four 32-column blocks per warp, single CTAs and CTA pairs, against the operand-exact fp64 product."""
import numpy as np
import pytest
import torch

from helpers import rel_fro
from paper_2501_01951_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    from paper_2501_01951_b200 import build
    build.build()
    from paper_2501_01951_b200 import binding
    return binding


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("M,N,K", [(130, 4, 40), (300, 19, 52), (257, 33, 64), (129, 64, 100), (500, 130, 33), (200, 255, 64), (150, 300, 40), (4100, 520, 512), (4097, 513, 600)])
def test_masks(mg, prec, M, N, K):
    ctx = mg.ctx_create(0)
    r4 = lambda x: (x + 3) // 4 * 4
    A, B = synth.uniform_tensor((M, K), 31, -1, 1), synth.uniform_tensor((K, N), 32, -1, 1)
    cut = (lambda t: t.to(torch.bfloat16).double()) if prec == 2 else (lambda t: (t.contiguous().view(torch.int32) & -8192).view(torch.float32).double())
    P = (cut(A) @ cut(B)).numpy()
    pad = lambda t: torch.nn.functional.pad(t, (0, r4(t.shape[1]) - t.shape[1])).cuda().contiguous()
    bias, gate = synth.uniform_tensor((N,), 33, -1, 1), synth.uniform_tensor((M, N), 34, -1, 1)
    drop = synth.bernoulli_mask(M * N, 0.5, 35)
    words = (N + 31) // 32
    gb = torch.zeros(M, words, dtype=torch.int32, device="cuda")
    mg.mask_pack(ctx, N, gb, X=pad(gate))
    C = torch.full((M, r4(N)), 3.0, device="cuda")
    y = P + bias.numpy()
    dm, gm = drop.numpy().reshape(M, N) * 2.0, (gate.numpy() > 0) * 0.5
    base = dict(bias=bias.cuda())
    cases = [(dict(drop_mask=drop.cuda(), keep_scale=2.0, relu=True, **base), np.maximum(y, 0) * dm), (dict(gate=pad(gate), gate_scale=0.5, **base), y * gm),
             (dict(gate_bits=gb, gate_scale=0.5, **base), y * gm), (dict(gate=gate.cuda().contiguous(), gate_scale=0.5, drop_mask=drop.cuda(), keep_scale=2.0, **base), y * dm * gm)]
    for (epi, want), keep in zip(cases, (dm, gm, gm, dm * gm)):
        bits = torch.full((M, words + 1), -1, dtype=torch.int32, device="cuda")
        mg.gemm(ctx, prec, False, False, M, N, K, pad(A), pad(B), C, epi=mg.make_epilogue(sign_bits=bits, **epi))
        got = C[:, :N].cpu().numpy()
        assert rel_fro(got, want) <= 2e-5 and np.all(got[keep == 0] == 0)
        packed = np.zeros((M, words * 32), dtype=np.uint32); packed[:, :N] = got > 0
        packed = (packed.reshape(M, words, 32) << np.arange(32, dtype=np.uint32)).sum(axis=2, dtype=np.uint32)
        assert np.array_equal(bits[:, :words].cpu().numpy().view(np.uint32), packed) and torch.all(bits[:, words] == -1)
    paths = mg.ctx_gemm_paths(ctx)
    assert paths["simt"] == 0 and paths["cta_pairs"] == (4 if M > 4000 else 0)
    assert mg.ctx_poll_status(ctx, raise_on_error=False) == 0
    ctx.close()
