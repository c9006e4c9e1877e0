"""A draft that is a view at any element offset of a larger buffer gives the decision of the same draft at an aligned address,
bit for bit: its rows are read four values at a time where it is 16-byte aligned, one by one where it is not.  At 4, 16, 32
and 64 columns (and a window that runs as slices), where a CTA writes the final outputs itself, where the partial results of
several CTAs are merged, and for a sequence without tokens."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,k", [(4, 1), (4, 4), (4, 8), (8, 8), (8, 11)])
@pytest.mark.parametrize("lens", [(100, 0, 37), (6000, 300)])     # one CTA per head; several
def test_draft_at_any_element_offset(G, k, lens):
    import paper_2607_01831_b200 as lynx
    B, Hkv, bt = len(lens), 2, 16
    lens_t = torch.tensor(lens, dtype=torch.int32)
    table, nb = synth.block_table(torch.clamp(lens_t, min=1), bt, True, "da", G * k)
    K = lynx.split_quantize(synth.kv_block_values("normal", nb, Hkv, bt, "cpu", "daK", G).cuda())
    V = lynx.split_quantize(synth.kv_block_values("normal", nb, Hkv, bt, "cpu", "daV", G).cuda())
    q = synth.queries(B, k, Hkv * G, "cpu", "daQ", G).cuda()
    geo = lynx.Geometry(Hkv * G, Hkv, bt, nb, table.shape[1])
    ws = lynx.make_workspace(geo, B, k, "cuda")
    td, ld = table.cuda(), lens_t.cuda()
    draft = lynx.anchor_attention(geo, q, K, V, td, ld, lynx.make_workspace(geo, B, k, "cuda"), causal=True)
    draft[0, k - 1, 1, 5] += 3.0                                   # a rejected position
    if 0 in lens:
        draft[lens.index(0), 0, 0, 127] = 0.3                      # a deviation against the zeros of an empty sequence

    def run(offset):
        buf = torch.full((draft.numel() + 8,), float("nan"), device="cuda")
        view = buf[offset:offset + draft.numel()].view(draft.shape)
        view.copy_(draft)
        assert view.data_ptr() % 16 == 4 * offset % 16
        got = lynx.merge_verify_attention(geo, q, K, V, td, ld, ws, draft_out=view, atol=0.5, rtol=0.1)
        lynx.check(ws)
        return got

    want = run(0)
    # the decision itself, from the outputs
    dev = ((want[0] - draft).abs() / (0.5 + 0.1 * want[0].abs())).amax((2, 3))
    assert torch.allclose(want[2], dev, rtol=1e-6, atol=0.0)       # three roundings: subtraction, denominator, quotient
    rejected = want[2] > 1.0
    first = torch.where(rejected.any(1), rejected.int().argmax(1), torch.full((B,), k, device="cuda"))
    assert torch.equal(want[1], first.int()) and int(want[1][0]) <= k - 1
    for offset in (1, 2, 3, 4):
        for w, g in zip(want, run(offset)):
            assert torch.equal(w, g)
