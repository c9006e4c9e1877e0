"""Split-quantise takes its source rows with 256-bit loads where the source is 32-byte aligned and with two 128-bit loads
where it is 16-byte aligned only: both give the oracle's planes and metadata bit for bit, dense and through a block list,
for row counts around the rows a warp has in flight."""
import numpy as np
import pytest
import torch

import oracle
import synth
from util import bf16_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 8])          # elements: 8 = 16 bytes
@pytest.mark.parametrize("rows", [1, 3, 4, 5, 127, 2049])
def test_dense_rows(offset, rows):
    import paper_2607_01831_b200 as lynx
    n = (rows + 15) // 16
    x = synth.kv_block_values("student_t4", n, 1, 16, "cpu", "al", rows).reshape(-1, 128)[:rows]
    buf = torch.zeros(offset + rows * 128, dtype=torch.bfloat16, device="cuda")
    src = buf[offset:].view(rows, 128)
    src.copy_(x)
    assert src.data_ptr() % 32 == 2 * offset % 32
    got = lynx.split_quantize(src)
    for g, w in zip((got.anchor, got.residual), oracle.split_quantize(bf16_bits(x))[:2]):
        assert np.array_equal(g.cpu().numpy(), w)
    assert np.array_equal(got.meta.cpu().numpy().view(np.uint32), oracle.split_quantize(bf16_bits(x))[2].view(np.uint32))


@pytest.mark.parametrize("offset", [0, 8])
def test_listed_blocks(offset):
    import paper_2607_01831_b200 as lynx
    nb, rpb = 9, 2 * 16
    x = synth.kv_block_values("lognormal_channels", nb, 2, 16, "cpu", "alb", 1).reshape(nb * rpb, 128)
    buf = torch.zeros(offset + x.numel(), dtype=torch.bfloat16, device="cuda")
    src = buf[offset:].view(nb * rpb, 128)
    src.copy_(x)
    ids = torch.tensor([7, 0, 4], dtype=torch.int32, device="cuda")
    out = lynx.Planes(torch.full((nb * rpb, 64), 0xAA, dtype=torch.uint8, device="cuda"),
                      torch.full((nb * rpb, 64), 0xAA, dtype=torch.uint8, device="cuda"),
                      torch.full((nb * rpb, 2), -7.0, device="cuda"))
    lynx.split_quantize(src, out=out, block_ids=ids, rows_per_block=rpb)
    wa, wr, wm = oracle.split_quantize(bf16_bits(x))
    listed = np.isin(np.arange(nb * rpb) // rpb, [7, 0, 4])
    a, r, m = out.anchor.cpu().numpy(), out.residual.cpu().numpy(), out.meta.cpu().numpy()
    assert np.array_equal(a[listed], wa[listed]) and np.array_equal(r[listed], wr[listed])
    assert np.array_equal(m[listed].view(np.uint32), wm[listed].view(np.uint32))
    assert np.all(a[~listed] == 0xAA) and np.all(r[~listed] == 0xAA) and np.all(m[~listed] == -7.0)
