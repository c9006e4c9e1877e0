"""Verification with 17..32 columns on a context where one token outweighs every other one by 2^x: what the others add together
is still there when a weight of theirs is below the last step of the kernel's number format.

Bound, relative to the 2-norm of the output.  Where values go through integer products (24 units per CTA and more), a weight is off by
up to a step of 2^-26 of the largest, without a bias: the sum over n tokens of an accumulator by sqrt(n) / 2 steps (standard deviation),
four of which are allowed, times the ratio r of the others' values (their distance to the middle of their range) to the output; the
FP16 weights' steps of 2^-33 are below that.  The 32-bit sum of the weights in the thread that has the dominating token may lose its
own n / 32 others.  The rest, scores and roundings, is what contexts without such a token have (4e-6 allowed)."""
import math

import pytest
import torch

import paper_2607_01831_b200 as lynx

pytestmark = pytest.mark.gpu


def _values(p):
    nib = lambda t: torch.stack((t & 15, t >> 4), -1).flatten(-2).double()  # noqa: E731
    return p.meta[..., 1:2].double() + p.meta[..., 0:1].double() * (nib(p.anchor) * 16 + nib(p.residual))


@pytest.mark.parametrize("tokens,G,k", [(131072, 4, 8), (131072, 3, 6), (7040, 4, 8)])   # 28 units of 128 tokens per CTA; 2
@pytest.mark.parametrize("x", [20, 26.6, 30, 33])
def test_the_rest_of_the_context_counts(tokens, G, k, x):
    H, bt, where = 4, 64, 1000
    nb = tokens // bt
    g = torch.Generator(device="cuda")
    g.manual_seed(tokens + k)
    q = (1 + 0.05 * torch.randn(1, k, H * G, 128, generator=g, device="cuda")).to(torch.bfloat16)
    kx = 0.1 * torch.randn(nb, H, bt, 128, generator=g, device="cuda")
    vx = 0.2 * torch.randn(nb, H, bt, 128, generator=g, device="cuda") - 0.5
    vx[..., 5] += 4.0                                     # a channel apart: the others' codes lie far from the middle
    kx[where // bt, :, where % bt] = x / (math.log2(math.e) * math.sqrt(128))
    vx[where // bt, :, where % bt] = torch.randn(H, 128, generator=g, device="cuda")
    K, V = (lynx.split_quantize(t.to(torch.bfloat16)) for t in (kx, vx))
    geo = lynx.Geometry(H * G, H, bt, nb, nb)
    ws = lynx.make_workspace(geo, 1, k, "cuda")
    table = torch.arange(nb, dtype=torch.int32, device="cuda").view(1, -1)
    out, _, _ = lynx.merge_verify_attention(geo, q, K, V, table, torch.tensor([tokens], dtype=torch.int32, device="cuda"), ws, causal=False)
    lynx.check(ws)
    kd, vd = (_values(p).permute(1, 0, 2, 3).reshape(H, tokens, 128) for p in (K, V))
    p = torch.softmax(q[0].double().permute(1, 0, 2).reshape(H, G * k, 128) @ kd.transpose(1, 2) / math.sqrt(128), 2)
    ref = (p @ vd).reshape(H * G, k, 128).permute(1, 0, 2)
    err = ((out[0].double() - ref).norm() / ref.norm()).item()
    n = tokens * H / 148 / 2                              # tokens of one accumulator
    span = V.meta[..., 0].double().mean().item() * 128 * math.sqrt(128)   # the others' distance to the middle of their range
    r = span / (ref.norm() / math.sqrt(H * G * k)).item()
    bound = 4 * math.sqrt(n) / 2 * 2.0 ** -26 * r + n / 32 * min(2.0 ** -x, 2.0 ** -24) * r + 4e-6
    assert err <= bound, (err, bound)
