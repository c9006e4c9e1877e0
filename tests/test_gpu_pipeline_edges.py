"""Anchor and verification attention with up to 16 query columns where the pipeline of their kernel can go wrong: pieces of fewer
units than it has softmax groups, of as many as it has buffers and one more, CTAs with many pieces, more units than the rings hold
several times over, references that are raised in every stage of it, and integer sums that are drained before they could overflow.
Verification with 17..32 columns likewise where its values go through integer products (its rule goes by the table's width, so that
a wide table takes short sequences there).  Against a 64-bit evaluation with torch on the dequantised planes.

Tolerance: a weight 2^(x - ref) formed in binary32 from four roundings of a score below 128 (log2 units) is off by 2.1e-5 of itself,
its rounding to an integer by 2^-29 of the largest, independently from token to token; the integer sums are exact, and putting
them together adds some 2^-22.  An output row, a weighted mean of values, is then off by less than 3e-5 of its 2-norm; half as
much again is allowed.  A log-sum-exp carries the four roundings and that of its own sum: 7e-5, likewise."""
import math

import pytest
import torch

import paper_2607_01831_b200 as lynx

pytestmark = pytest.mark.gpu
REL, LSE = 4.5e-5, 1.05e-4


def _values(p, full):
    nib = lambda t: torch.stack((t & 15, t >> 4), -1).flatten(-2).double()  # noqa: E731
    return p.meta[..., 1:2].double() + p.meta[..., 0:1].double() * (nib(p.anchor) * 16 + (nib(p.residual) if full else 8))


def _run(lens, Hkv, G, n_q, ramp, bt=16, width=0, states=(False, True)):
    g = torch.Generator(device="cuda")
    g.manual_seed(sum(lens) + G * n_q)
    need = [(n + bt - 1) // bt for n in lens]
    nb, B = sum(need), len(lens)
    table = torch.zeros(B, max(max(need), width), dtype=torch.int32)
    perm, pos = torch.randperm(nb, generator=torch.Generator().manual_seed(nb)).to(torch.int32), 0
    for b, n in enumerate(need):
        table[b, :n] = perm[pos:pos + n]
        pos += n
    k, v = (torch.randn(nb, Hkv, bt, 128, generator=g, device="cuda") for _ in range(2))
    q = torch.randn(B, n_q, Hkv * G, 128, generator=g, device="cuda")
    if ramp:   # scores that climb along the sequence: the largest weight so far is exceeded again and again
        q = 1.0 + 0.05 * q
        climb = torch.zeros(nb, device="cuda")
        for b, n in enumerate(need):
            climb[table[b, :n].long().cuda()] = torch.arange(n, device="cuda", dtype=torch.float32) / n
        k = 0.3 * k + 7.0 * climb.view(-1, 1, 1, 1)
    q = q.to(torch.bfloat16)
    K, V = (lynx.split_quantize(x.to(torch.bfloat16)) for x in (k, v))
    geo = lynx.Geometry(Hkv * G, Hkv, bt, nb, table.shape[1])
    ws = lynx.make_workspace(geo, B, n_q, "cuda")
    tab, ln = table.cuda(), torch.tensor(lens, dtype=torch.int32, device="cuda")
    for full in states:
        call = lynx.merge_verify_attention if full else lynx.anchor_attention
        outs = []
        for _ in range(2):   # (a second time on the workspace as the first left it)
            o = call(geo, q, K, V, tab, ln, ws, causal=True)
            outs.append(o[0] if full else o)
        lynx.check(ws)
        assert torch.equal(outs[0], outs[1])
        lse = lynx.workspace_lse(geo, B, n_q, ws)
        kd, vd = _values(K, full), _values(V, full)
        for b in range(B):
            n = lens[b]
            kk, vv = (x[tab[b, :need[b]].long()].permute(1, 0, 2, 3).reshape(Hkv, -1, 128)[:, :n] for x in (kd, vd))
            s = q[b].double().permute(1, 0, 2).reshape(Hkv, G * n_q, 128) @ kk.transpose(1, 2) / math.sqrt(128)
            last = n - n_q + torch.arange(n_q, device="cuda").repeat(G)
            s.masked_fill_(torch.arange(n, device="cuda") > last[:, None], -math.inf)
            ref = (torch.softmax(s, 2).nan_to_num(0.0) @ vv).reshape(Hkv * G, n_q, 128).permute(1, 0, 2)
            got = outs[0][b].double()
            assert torch.isfinite(got).all()
            assert (got - ref).norm() <= REL * ref.norm(), (full, b, ((got - ref).norm() / ref.norm()).item())
            want = torch.logsumexp(s, 2).reshape(Hkv * G, n_q).permute(1, 0)
            fin = torch.isfinite(want)
            assert torch.equal(fin, torch.isfinite(lse[b])) and (lse[b].double() - want)[fin].abs().max() <= LSE


@pytest.mark.parametrize("G,n_q", [(3, 1), (4, 1), (7, 1), (4, 2), (3, 3), (4, 4), (16, 1)])   # 3, 4, 7, 8, 9, 16, 16 columns
@pytest.mark.parametrize("lens", [
    [1, 16, 127, 128, 129],                                   # pieces of one unit and of two
    [128 * n for n in range(1, 18)] + [128 * 17 + 1],         # around every depth of the buffers, CTAs with several pieces
    [60 + 70 * (i % 5) for i in range(400)],                  # many pieces per CTA
])
def test_pieces(G, n_q, lens):
    _run(lens, 1, G, n_q, ramp=False)


@pytest.mark.parametrize("G,n_q", [(4, 1), (8, 1), (4, 4)])
@pytest.mark.parametrize("ramp", [False, True])
def test_rings_that_come_round(G, n_q, ramp):
    _run([148 * 128 * 19 + 77], 1, G, n_q, ramp)              # 19 and 20 units per CTA


@pytest.mark.parametrize("G,n_q", [(4, 1), (8, 1), (4, 4)])
@pytest.mark.parametrize("lens", [[700, 129], [2600], [128 * 9] * 40])
def test_references_that_are_raised(G, n_q, lens):
    _run(lens, 2, G, n_q, ramp=True)


def _wide(Hkv, B):
    """Blocks of a table that gives 148 CTAs 24 units of 128 tokens each, and some more."""
    return 24 * 148 * 8 // (Hkv * B) + 1


@pytest.mark.parametrize("G,n_q", [(3, 6), (3, 7), (4, 8)])   # 18, 21, 32 columns
@pytest.mark.parametrize("lens", [[1, 16, 127, 128, 129], [128 * n for n in range(1, 7)], [60 + 70 * (i % 5) for i in range(100)]])
def test_values_on_integers(G, n_q, lens):
    _run(lens, 1, G, n_q, ramp=False, width=_wide(1, len(lens)), states=(True,))


@pytest.mark.parametrize("lens", [[700, 129], [2600], [128 * 9] * 40])
def test_values_on_integers_when_references_are_raised(lens):
    _run(lens, 2, 4, 8, ramp=True, width=_wide(2, len(lens)), states=(True,))


def test_sums_are_drained_before_they_could_overflow():
    """148 heads of 1032 units: a CTA has a head, and each of up to four softmax groups more than the 256 units between drains."""
    heads, tokens, bt = 148, 1032 * 128, 64
    nb = tokens // bt
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    K, V = (lynx.alloc_planes((nb, heads, bt), "cuda") for _ in range(2))
    for P in (K, V):
        for i in range(0, nb, 129):
            x = torch.randn(129, heads, bt, 128, generator=g, device="cuda")
            lynx.split_quantize(x.to(torch.bfloat16), out=lynx.Planes(P.anchor[i:i + 129], P.residual[i:i + 129], P.meta[i:i + 129]))
    tab = torch.arange(nb, dtype=torch.int32, device="cuda").view(1, -1)
    ln = torch.tensor([tokens], dtype=torch.int32, device="cuda")
    for G, n_q in ((1, 4), (1, 8), (1, 16), (2, 16)):
        geo = lynx.Geometry(heads * G, heads, bt, nb, nb)
        ws = lynx.make_workspace(geo, 1, n_q, "cuda")
        q = torch.randn(1, n_q, heads * G, 128, generator=g, device="cuda").to(torch.bfloat16)
        for full in (False, True):
            call = lynx.merge_verify_attention if full else lynx.anchor_attention
            o = call(geo, q, K, V, tab, ln, ws, causal=False)
            o = o[0] if full else o
            lynx.check(ws)
            for h in (0, 77, 147):
                kd, vd = (_values(lynx.Planes(*(t[:, h] for t in (P.anchor, P.residual, P.meta))), full).reshape(tokens, 128) for P in (K, V))
                sl = slice(h * G, h * G + G)
                ref = torch.softmax(q[0, :, sl].double().reshape(-1, 128) @ kd.T / math.sqrt(128), 1) @ vd
                got = o[0, :, sl].double().reshape(-1, 128)
                # (a mean of 132096 values is 1 / 360 of one.  Anchor levels count from the zero point: the mean is the difference of two
                # sums of its size, here up to 5.5, with some four roundings.  Full codes count from the middle of their row, half a unit
                # away from zero at most where rows are 128 normal values)
                bound = REL * ref.norm() + 4 * 2.0 ** -24 * (0.5 if full else 5.5) * ref.numel() ** 0.5
                assert (got - ref).norm() <= bound, (G, n_q, full, h, ((got - ref).norm() / bound).item())


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("G,n_q", [(1, 4), (1, 8), (1, 16), (2, 16)])
def test_sums_that_would_overflow(G, n_q, full):
    """A CTA for each head and 2120 units for each CTA: 530 for each of four softmax groups, 706 of three, 1060 of two.  Every unit has one
    token whose weight is 2^-12 over the others', so that these are 255 in a byte plane, and values at the ends of their rows: without drains
    a sum of full codes passes 2^31 at 514 units, of an Anchor's odd dims at 274 (kDrainUnits).  All units are the same two blocks, so that the
    result is one unit's.  Bound: the sums of weights in 32 bits, at most half an ulp for each of a thread's additions and either sum; a sum
    that wraps around is off by more than the result."""
    heads, units, bt = 148, 2120, 64
    v = torch.empty(2, heads, bt, 128)
    v[..., :64], v[..., 64:] = 2.0, -1.0                  # codes 255 and 0, Anchor levels 15 and 0
    k = torch.zeros(2, heads, bt, 128)
    k[..., 1] = 1.0                                       # (a scale for every row)
    k[0, :, 0, 0] = 1.0
    q = torch.zeros(1, n_q, heads * G, 128)
    q[..., 0] = 0.0015                                    # 0.0015 / sqrt(128) log2(e) = 1.9e-4
    K, V = (lynx.split_quantize(x.to(torch.bfloat16).cuda()) for x in (k, v))
    q = q.to(torch.bfloat16).cuda()
    nb = units * 2
    table = torch.arange(2, dtype=torch.int32, device="cuda").repeat(units).view(1, nb)
    geo = lynx.Geometry(heads * G, heads, bt, 2, nb)
    ws = lynx.make_workspace(geo, 1, n_q, "cuda")
    call = lynx.merge_verify_attention if full else lynx.anchor_attention
    o = call(geo, q, K, V, table, torch.tensor([units * 128], dtype=torch.int32, device="cuda"), ws, causal=False)
    o = (o[0] if full else o)[0].double()
    lynx.check(ws)
    kd, vd = (_values(p, full).permute(1, 0, 2, 3).reshape(heads, 128, 128) for p in (K, V))
    s = q[0].double().permute(1, 0, 2).reshape(heads, G * n_q, 128) @ kd.transpose(1, 2) / math.sqrt(128)
    ref = (torch.softmax(s, 2) @ vd).reshape(heads * G, n_q, 128).permute(1, 0, 2)
    adds = units // 2 * 4                                 # (two groups, four tokens of a unit to a thread)
    assert (o - ref).abs().max() <= 2 * adds * 2.0 ** -24 * ref.abs().max(), (o - ref).abs().max().item()
