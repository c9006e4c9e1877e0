"""BF16-page attention where a chunk of 2048 tokens is shared by a cluster of 1 to 8 CTAs: around the tiles of 16 tokens, the chunk,
the cluster sizes that the number of heads leads to, and calls whose sequences are one chunk (no second kernel).  Outputs against
the float64 oracle at the tolerance of test_gpu_parity.py, log-sum-exps at that of test_gpu_tail.py."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_parity import _case, _close, lynx  # noqa: F401
from util import bf16_bits, bits_to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hkv,G,n_q,lens,bt", [
    (1, 1, 1, [1], 16), (2, 4, 1, [15, 16, 17], 16), (2, 4, 1, [63, 64, 65, 0], 16), (2, 8, 1, [2047], 16), (2, 4, 1, [2048], 16),
    (2, 4, 1, [2049, 130], 16), (1, 4, 2, [4097, 2048, 3], 32), (1, 2, 1, [1000], 48), (3, 1, 5, [900, 257], 64),
    (8, 4, 1, [300 + 7 * i for i in range(10)], 16),      # 80 pieces: clusters of two
    (8, 4, 1, [40] * 40, 16),                             # 320 pieces: no clusters
])
def test_shared_chunks(lynx, Hkv, G, n_q, lens, bt):
    c = _case(lynx, 700 + Hkv + len(lens), len(lens), Hkv, G, n_q, lens, bt)
    _, k = lynx.recombine(c["K"], want_codes=False, want_bf16=True)
    _, v = lynx.recombine(c["V"], want_codes=False, want_bf16=True)
    B = len(lens)
    n = int(lynx.load().lynx_bf16_workspace_bytes(c["geo"]._c(), B, n_q))
    ws = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")   # (nothing is expected of the workspace's contents)
    q, table, lens_d = (t.cuda() for t in (c["q"], c["table"], c["lens"]))
    kb, vb = bf16_bits(k), bf16_bits(v)
    for causal in (False, True):
        got = [lynx.bf16_attention(c["geo"], q, k, v, table, lens_d, ws, causal=causal) for _ in range(2)]
        assert torch.equal(got[0], got[1])
        ref = oracle.attention_bf16_pages(bf16_bits(c["q"]), kb, vb, c["table"].numpy(), c["lens"].numpy(), causal=causal)
        _close(got[0].cpu().numpy().astype(np.float64), ref, f"causal={causal}")
        lse = lynx.bf16_workspace_lse(c["geo"], B, n_q, ws).cpu().numpy()
        kf, qf = bits_to_f64(kb), bits_to_f64(bf16_bits(c["q"]))
        for b in range(B):
            for j in range(n_q):
                see = lens[b] - n_q + j + 1 if causal else lens[b]
                for h in range(Hkv * G):
                    if see <= 0:
                        assert lse[b, j, h] == -np.inf
                        continue
                    t = np.arange(see)
                    rows = kf[c["table"].numpy()[b][t // bt], h // G, t % bt]
                    s = rows @ qf[b, j, h] * np.float64(np.float32(1.0 / np.sqrt(128.0)))
                    want = s.max() + np.log(np.exp(s - s.max()).sum())
                    assert abs(lse[b, j, h] - want) < 2e-4, (b, j, h)
