"""The block of a token by multiplication: the rule itself, compiled for the host, and the attention kernels with block sizes that
are no power of two."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01831_b200", "csrc")

CHECK = r"""
#include <cstdio>
#include <initializer_list>
#include "block_division.cuh"
int main() {
  long long bad = 0;
  auto check = [&](int32_t n) {
    const lynx::BlockDiv d = lynx::block_div(n);
    const int64_t top = 2147483647ll, last = top / n, step = last / 1000 + 1;
    for (int64_t k = 0; k <= last; k += step)
      for (int64_t q : {k, last - k})
        for (int64_t t = q * n - 1; t <= q * n + 1; ++t)
          if (t >= 0 && t <= top && lynx::quotient((int32_t)t, d) != (int32_t)(t / n)) ++bad;
    for (int64_t t : {top, top - 1}) if (lynx::quotient((int32_t)t, d) != (int32_t)(t / n)) ++bad;
  };
  for (int32_t n = 2; n <= 4096; ++n) check(n);
  for (int64_t n = 4096; n < (1 << 30); n = n / 3 * 4 + 16) check((int32_t)n);
  check(1 << 30);
  printf("%lld", bad);
}
"""


def test_quotients_are_exact(tmp_path):
    """Every block size up to 4096 and some up to 2^30, at the multiples of the size around which a quotient could be off."""
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(CHECK)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout == "0"


@pytest.mark.gpu
@pytest.mark.parametrize("bt", [16, 48, 80, 128, 1008])
@pytest.mark.parametrize("G,n_q", [(4, 1), (4, 4), (4, 8), (8, 8)])
def test_block_sizes(bt, G, n_q):
    import oracle
    import paper_2607_01831_b200 as lynx
    from test_gpu_parity import _case, _close
    from util import bf16_bits
    c = _case(lynx, 40 + bt + G, 2, 2, G, n_q, [1500, 333], bt)
    q, table, lens = (t.cuda() for t in (c["q"], c["table"], c["lens"]))
    for full, call in ((False, lynx.anchor_attention), (True, lambda *a, **k: lynx.merge_verify_attention(*a, **k)[0])):
        got = call(c["geo"], q, c["K"], c["V"], table, lens, c["ws"], causal=True)
        lynx.check(c["ws"])
        ref = oracle.attention(full, bf16_bits(c["q"]), c["kp"], c["vp"], c["table"].numpy(), c["lens"].numpy(), 2, bt, causal=True)
        _close(got.cpu().numpy().astype(np.float64), ref, f"full={full}")
