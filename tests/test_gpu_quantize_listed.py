"""Quantisation of listed blocks against that of all rows: blocks of a multiple of four rows, whose rows are looked up four at a time,
and others, with ids that no block has among them and lists around the rows that a CTA takes at a time."""
import pytest
import torch

import paper_2607_01831_b200 as lynx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 4, 6, 12, 48, 128])
@pytest.mark.parametrize("n_ids", [1, 3, 11, 33, 200])
def test_listed_blocks(rows, n_ids):
    g = torch.Generator(device="cuda")
    g.manual_seed(rows + n_ids)
    blocks = 240
    src = torch.randn(blocks, 1, rows, 128, generator=g, device="cuda").to(torch.bfloat16)
    want = lynx.split_quantize(src)
    ids = torch.randperm(blocks, generator=torch.Generator().manual_seed(n_ids))[:n_ids].to(torch.int32)
    if n_ids > 3:
        ids[1], ids[n_ids // 2] = -1, blocks   # (not of this pool: left out)
    out = lynx.Planes(*(torch.full_like(t, 77) for t in (want.anchor, want.residual, want.meta)))
    lynx.split_quantize(src, out=out, block_ids=ids.cuda(), rows_per_block=rows)
    listed = torch.zeros(blocks, dtype=torch.bool)
    listed[ids[(ids >= 0) & (ids < blocks)].long()] = True
    for a, b in zip((out.anchor, out.residual, out.meta), (want.anchor, want.residual, want.meta)):
        assert torch.equal(a[listed], b[listed]) and (a[~listed] == 77).all()
