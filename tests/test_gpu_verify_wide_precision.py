"""Merge-verify at 17..32 columns keeps the precision of the exact integer path it replaced: the tensor core's accumulation
truncates, which shows as a bias, where roundings to nearest leave none.

Scores: a sequence of one token, whose log-sum-exp is its score.  Keys and queries of one sign make every partial sum grow, and
queries over nine binades leave no common grid, so truncation would take some 0.46 ulp in each of 8 steps: a bias of about
1.5e-7 of the score.  With exact sums what is left are some eight roundings to nearest, 8 * 2^-24 at most for one score; their
mean over 128 independent key rows stays within 8 * 2^-24 / sqrt(128) = 4.2e-8.  (The scores are some hundreds, so that the
approximate exponent and logarithm of the one weight, some 2e-6, do not show.)

Values: weights within a binade or two over equal value rows of +1 and -1, contexts of 12 units per accumulator for the FP16 weights (a
table of 113600 tokens and 4 heads) and of 14 for the integer ones (131072), whose sums are exact.  Sixteen truncating steps
between two drains, at half an ulp of a running sum that grows to its final size: 8.5 * 0.5 * 2^-23 = 5.1e-7 at most on the
mean; the FP32 copy's roundings are to nearest.  (64 steps between drains: 1.3e-6.)"""
import numpy as np
import pytest
import torch

import oracle
from util import bf16_bits, dequant

pytestmark = pytest.mark.gpu


def _verify(lynx, q, K, V, table, lens, Hkv, G, k):
    geo = lynx.Geometry(Hkv * G, Hkv, 16, K.anchor.shape[0], table.shape[1])
    B = lens.numel()
    ws = lynx.make_workspace(geo, B, k, "cuda")
    out, _, _ = lynx.merge_verify_attention(geo, q.cuda(), K, V, table.cuda(), lens.cuda(), ws, causal=False)
    lynx.check(ws)
    return out.cpu().numpy().astype(np.float64), lynx.workspace_lse(geo, B, k, ws).cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("G,k", [(4, 5), (8, 3), (4, 8)])          # 20, 24, 32 columns
def test_scores_have_no_bias(G, k):
    import paper_2607_01831_b200 as lynx
    g = torch.Generator().manual_seed(1)
    B, Hkv = 64, 2
    kx = (1.0 + 3.0 * torch.rand(B, Hkv, 16, 128, generator=g)).to(torch.bfloat16)
    ends = 4.0 + torch.rand(B, Hkv, 16, 2, generator=g)            # rows around zero, each with a scale of its own
    kx[..., 0], kx[..., 1] = (-ends[..., 0]).to(torch.bfloat16), ends[..., 1].to(torch.bfloat16)
    v = torch.randn(B, Hkv, 16, 128, generator=g).to(torch.bfloat16)
    q = torch.exp2(9.0 * torch.rand(B, k, Hkv * G, 128, generator=g) - 3.0).to(torch.bfloat16)
    K, V = lynx.split_quantize(kx.cuda()), lynx.split_quantize(v.cuda())
    table = torch.arange(B, dtype=torch.int32).view(B, 1)
    _, lse = _verify(lynx, q, K, V, table, torch.ones(B, dtype=torch.int32), Hkv, G, k)
    key = dequant(*oracle.split_quantize(bf16_bits(kx)), full=True)[:, :, 0]      # [B][Hkv][128]
    s = np.einsum("bkhgd,bhd->bkhg", q.double().numpy().reshape(B, k, Hkv, G, 128), key).reshape(B, k, Hkv * G)
    f32 = np.float32                                               # the constants as the library holds them
    s *= np.float64(f32(0.08838834764831845) * f32(1.4426950408889634)) * np.float64(f32(0.6931471805599453))
    err = lse / s - 1.0
    assert s.min() > 50 and np.abs(err).max() <= 8 * 2.0 ** -24 + 2e-6 / s.min(), np.abs(err).max()
    assert abs(err.mean()) <= 8 * 2.0 ** -24 / np.sqrt(128), err.mean()


@pytest.mark.parametrize("n", [113600, 131072])
@pytest.mark.parametrize("G,k", [(4, 5), (4, 8)])
def test_values_are_drained_often_enough(G, k, n):
    import paper_2607_01831_b200 as lynx
    Hkv = 4
    row = torch.ones(128)
    row[1::2] = -1.0
    g = torch.Generator().manual_seed(2)
    kx = torch.randn(n // 16, Hkv, 16, 128, generator=g, dtype=torch.float32).to(torch.bfloat16)
    v = row.expand(n // 16, Hkv, 16, 128).to(torch.bfloat16).contiguous()
    K, V = lynx.split_quantize(kx.cuda()), lynx.split_quantize(v.cuda())
    q = (0.3 * torch.randn(1, k, Hkv * G, 128, generator=g)).to(torch.bfloat16)    # weights with mantissas of all kinds
    table = torch.arange(n // 16, dtype=torch.int32).view(1, -1)
    out, _ = _verify(lynx, q, K, V, table, torch.tensor([n], dtype=torch.int32), Hkv, G, k)
    want = dequant(*oracle.split_quantize(bf16_bits(v[:1])), full=True)[0, 0, 0]
    err = out / want - 1.0
    assert abs(err.mean()) <= 5.1e-7, err.mean()
    assert np.abs(err).max() <= 2 * 8.5 * 2.0 ** -23, np.abs(err).max()      # a whole ulp a step, and as much for everything else
