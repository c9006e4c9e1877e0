"""Joining the partial results of the CTAs that share a head: the kernel behind every verification and behind anchor calls with
few heads (four warps per row, or one), and the last CTA of a head where there are many.  At the edges of its rules: heads with
one CTA, with as many as the grid has, rows that do not fill a CTA, query heads per KV head that divide nothing, sequences
without tokens among others.  Against the float64 oracle at the tolerance of test_gpu_parity.py; the decision as there."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_parity import _case, _close, lynx  # noqa: F401
from util import bf16_bits

pytestmark = pytest.mark.gpu


# (sequences, KV heads, query heads per KV head, positions, lengths)
SHAPES = [
    (1, 1, 1, 1, [1]),                                    # one unit, one row
    (1, 1, 3, 2, [148 * 256 + 5]),                        # one head has the whole grid: 148 slots and more than one round
    (3, 1, 5, 1, [700, 0, 129]),                          # an empty sequence; 15 rows
    (2, 2, 16, 3, [300, 4000]),                           # 48 columns
    (37, 1, 4, 1, [64 + 40 * i for i in range(37)]),      # just enough heads for the last CTA to join them
    (36, 1, 4, 1, [64 + 40 * i for i in range(36)]),      # and one fewer
    (40, 1, 2, 1, [20000] + [17] * 39),                   # many heads, one of them with nearly all CTAs
    (40, 1, 4, 4, [32768] + [64] * 39),                   # and 16 columns: long segments among those of one CTA
    (39, 1, 4, 8, [64] * 20 + [9000] + [100] * 17 + [15000]),   # two of them, 32 columns, in the middle and at the end
    (21, 2, 8, 8, [64] * 20 + [7000]),                    # 64 columns, two heads
    (41, 1, 4, 2, [3000] + [1] * 40),                     # 24 CTAs, where a segment begins to be long
    (42, 1, 4, 2, [2900, 3100] + [1] * 40),               # 23 and 25, where two levels begin
    (2, 8, 4, 4, [1, 128]),                               # heads of one unit
    (5, 3, 1, 7, [257, 1, 0, 900, 128]),
]


@pytest.mark.parametrize("B,Hkv,G,n_q,lens", SHAPES)
def test_joined_results(lynx, B, Hkv, G, n_q, lens):
    c = _case(lynx, B * 100 + G, B, Hkv, G, n_q, lens)
    dev = [t.cuda() for t in (c["q"], c["table"], c["lens"])]
    ref = {f: oracle.attention(f, bf16_bits(c["q"]), c["kp"], c["vp"], c["table"].numpy(), c["lens"].numpy(), Hkv, c["bt"], causal=True)
           for f in (False, True)}
    for _ in range(2):   # (a second time on the workspace as the first left it)
        draft = lynx.anchor_attention(c["geo"], dev[0], c["K"], c["V"], dev[1], dev[2], c["ws"], causal=True)
        out, first, devs = lynx.merge_verify_attention(c["geo"], dev[0], c["K"], c["V"], dev[1], dev[2], c["ws"], draft_out=draft,
                                                       atol=0.5, rtol=0.1)
        lynx.check(c["ws"])
        _close(draft.cpu().numpy().astype(np.float64), ref[False], "anchor")
        _close(out.cpu().numpy().astype(np.float64), ref[True], "verify")
        want, want_dev = oracle.verify_decision(ref[True], draft.cpu().numpy(), 0.5, 0.1)
        assert np.allclose(devs.cpu().numpy(), want_dev, rtol=2e-2, atol=1e-2)
        clear = np.all(np.abs(want_dev - 1.0) > 0.05, axis=1)
        assert np.array_equal(first.cpu().numpy()[clear], want[clear])
        plain = lynx.merge_verify_attention(c["geo"], dev[0], c["K"], c["V"], dev[1], dev[2], c["ws"])[0]
        assert torch.equal(plain, out)
