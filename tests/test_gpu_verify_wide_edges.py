"""GPU parity of merge-verify attention at 17..64 columns where its kernels can go wrong: around the 128-token units, the
drains of their accumulators and the changes of their reference exponents.  Outputs, log-sum-exps and the decision on a draft.

Tolerances.  The scores of these cases stay below 128 in log2 units; a weight 2^(x - ref) formed in binary32 from four
roundings of x is off by at most 4 * 2^-24 * 128 * ln 2 = 2.1e-5 of itself, the weights' two FP16 terms add 2^-22, and the
products' sums lose at most an ulp of half their final size per step, over the 8 steps of at most 16 units between two drains
128 * 2^-24 = 8e-6: 3e-5 of the largest |V| (below 8 here).  Half as much again is allowed.  A log-sum-exp carries the same four
roundings, at 33..64 columns eight truncations of a score (half an ulp on average, 8 * 2^-24 * 128 * ln 2 = 4.2e-5), and the
rounding of its own sum (2^-24 * 128): 7e-5, again with half as much on top.  A deviation |f - d| / (atol + rtol |f|) moves by
the error of f over atol, and by rtol / atol of that times itself.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from util import bf16_bits, dequant

pytestmark = pytest.mark.gpu

TOL = 1.5 * 3e-5 * 8
TOL_LSE = 1.5 * 7e-5
A, R = 0.5, 0.1             # atol, rtol of the decision


@pytest.fixture(scope="module")
def lynx():
    import paper_2607_01831_b200 as m
    m.load()
    return m


def _run(lynx, G, k, lens, ramp, causal=True, Hkv=2, bt=16):
    B = len(lens)
    lens_t = torch.tensor(lens, dtype=torch.int32)
    table, nb = synth.block_table(torch.tensor([max(n, 1) for n in lens], dtype=torch.int32), bt, False, "we", G * k)
    kx = synth.kv_block_values("normal", nb, Hkv, bt, "cpu", "weK", G * k).float()
    v = synth.kv_block_values("normal", nb, Hkv, bt, "cpu", "weV", G * k)
    q = synth.queries(B, k, Hkv * G, "cpu", "weQ", G * k).float()
    if ramp:   # scores that climb along the sequence: the largest weight so far is exceeded again and again
        q = 1.0 + 0.05 * q
        t = torch.arange(nb * bt, dtype=torch.float32).view(nb, 1, bt, 1) / (nb * bt)
        kx = 0.3 * kx + 7.0 * t
    q, kx = q.to(torch.bfloat16), kx.to(torch.bfloat16)
    K, V = lynx.split_quantize(kx.cuda()), lynx.split_quantize(v.cuda())
    kp, vp = oracle.split_quantize(bf16_bits(kx)), oracle.split_quantize(bf16_bits(v))
    geo = lynx.Geometry(Hkv * G, Hkv, bt, nb, table.shape[1])
    ws = lynx.make_workspace(geo, B, k, "cuda")
    draft = lynx.anchor_attention(geo, q.cuda(), K, V, table.cuda(), lens_t.cuda(), ws, causal=causal)
    draft[0, k // 2, 0, 3] += 2.0                          # one position off by more than the margin
    out, first, dev = lynx.merge_verify_attention(geo, q.cuda(), K, V, table.cuda(), lens_t.cuda(), ws, draft_out=draft,
                                                  atol=A, rtol=R, causal=causal)
    lynx.check(ws)
    lse = lynx.workspace_lse(geo, B, k, ws).cpu().numpy().astype(np.float64)
    ref = oracle.attention(True, bf16_bits(q), kp, vp, table.numpy(), lens_t.numpy(), Hkv, bt, causal=causal)
    got = out.cpu().numpy().astype(np.float64)
    assert np.all(np.isfinite(got))
    assert float(np.abs(got - ref).max()) <= TOL, float(np.abs(got - ref).max())
    want = _lse(q, kp, table.numpy(), lens, Hkv, bt, causal)
    assert np.array_equal(np.isneginf(lse), np.isneginf(want))
    fin = np.isfinite(want)
    assert float(np.abs(lse[fin] - want[fin]).max()) <= TOL_LSE, float(np.abs(lse[fin] - want[fin]).max())
    ref_first, ref_dev = oracle.verify_decision(ref, draft.cpu().numpy(), A, R)
    tol_dev = TOL / A * (1.0 + R * ref_dev)
    assert np.all(np.abs(dev.cpu().numpy() - ref_dev) <= tol_dev)
    if np.all(np.abs(ref_dev - 1.0) > tol_dev):            # (no position within the margin's own error)
        assert np.array_equal(first.cpu().numpy(), ref_first)


def _lse(q, kp, table, lens, Hkv, bt, causal):
    """Natural-log log-sum-exp of every output row's scores, binary64."""
    q = q.double().numpy()
    B, k, Hq, _ = q.shape
    key = dequant(*kp, full=True)                          # [blocks][Hkv][bt][128]
    out = np.full((B, k, Hq), -np.inf)
    for b, n in enumerate(lens):
        rows = key[table[b, :(n + bt - 1) // bt]].transpose(1, 0, 2, 3).reshape(Hkv, -1, 128)[:, :n]
        for j in range(k):
            lim = max(n - k + j + 1, 0) if causal else n
            if lim:
                s = np.einsum("hgd,htd->hgt", q[b, j].reshape(Hkv, -1, 128), rows[:, :lim]).reshape(Hq, lim)
                s *= np.float64(np.float32(1.0 / np.sqrt(128.0)))
                m = s.max(1)
                out[b, j] = m + np.log(np.exp(s - m[:, None]).sum(1))
    return out


@pytest.mark.parametrize("G,k", [(1, 16), (3, 6), (4, 8), (3, 11), (8, 8)])     # 16 (integer path), 18, 32, 33, 64 columns
@pytest.mark.parametrize("lens", [(127, 128), (129, 1), (16, 15, 300), (1024, 1025), (2303,)])
def test_lengths_around_units_and_drains(lynx, G, k, lens):
    _run(lynx, G, k, lens, ramp=False)


@pytest.mark.parametrize("G,k", [(4, 5), (4, 8), (8, 8)])
@pytest.mark.parametrize("lens", [(700, 129), (2600,)])
@pytest.mark.parametrize("causal", [True, False])
def test_scores_that_keep_rising_raise_the_references(lynx, G, k, lens, causal):
    _run(lynx, G, k, lens, ramp=True, causal=causal)
