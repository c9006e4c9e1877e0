"""One workspace for calls of different batches, heads and positions: what outlives a call (the status word, the tickets) is where no
other call puts its results.  The layout is compiled for the host; on the GPU, calls of two batches take turns on one workspace."""
import os
import random
import re
import subprocess

import pytest
import torch

import paper_2607_01831_b200 as lynx

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01831_b200", "csrc")

CHECK = r"""
#include <cstdio>
#include <initializer_list>
#include "workspace_layout.cuh"
int main() {
  const int sms = 148;
  size_t kept = 0, end = 0, bad = 0, n = 0;
  for (int B : {1, 2, 16, 37, 256, 1000})
    for (int Hkv : {1, 8, 32})
      for (int G : {1, 4, 16})
        for (int nq : {1, 4, 64})
          for (int cols : {8, 16, 32, 64}) {
            const lynx::WsLayout w = lynx::ws_layout(sms, B, nq, Hkv * G, Hkv, cols);
            if (n++ == 0) { kept = w.off_tickets; end = w.end_kept; }
            bad += w.off_tickets != kept || w.end_kept != end;                                   // the same for every call
            const size_t at[] = {4, w.off_tickets, w.off_groups, w.end_kept, w.off_long, w.off_seq_ctr, w.off_dev, w.off_lse, w.off_part, w.bytes};
            const size_t need[] = {0, sms * 4, 2 * sms * 4, 0, (sms + 7) / 8 * 4, (size_t)B * 4, (size_t)B * Hkv * 64, (size_t)B * nq * Hkv * G * 4,
                                   (size_t)(B * Hkv + sms) * cols * 528};
            for (int i = 0; i < 9; ++i) bad += at[i] + need[i] > at[i + 1] || at[i + 1] % (i > 4 ? 16 : 4) != 0;
          }
  std::printf("%zu %zu", bad, n);
}
"""


def test_no_results_on_what_is_kept(tmp_path):
    src, exe = tmp_path / "l.cpp", tmp_path / "l"
    src.write_text(CHECK)
    subprocess.run(["g++", "-std=c++17", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    bad, n = (int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert n == 648 and bad == 0


def test_counts_are_either_kept_or_zeroed_by_the_call():
    """Tickets are taken at places that do not depend on the batch; everything else that is counted is zeroed by the kernel before."""
    text = "".join(re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, n)).read()) for n in ("attention.cu", "attention_i8.cuh", "attention_f16.cuh", "attention_pipe.cuh"))
    counted = set(re.findall(r"atomic(?:Inc|Add|Max|Or)\((?:reinterpret_cast<int\*>\()?(?:p\.)?(\w+)", text))
    assert counted == {"ticket", "ws_seq_ctr", "ws_dev", "ws_flags"}
    group = re.search(r"SlotGroup slot_group\(.*?\n\}", text, re.S).group(0)
    assert set(re.findall(r"p\.(ws_\w+)", group)) == {"ws_tickets", "ws_groups"}
    assert set(re.findall(r"\blast_of\(([^,]+),", text)) == {"uint32_t* ticket", "g.ticket", "p.ws_tickets + item.first_cta"}
    # (deviations: by the publishing producer of the kernels that verify, which share plane_producer)
    assert len(re.findall(r"p\.ws_dev\[[^;]*\] = 0\.0f;", text)) == 1 and "p.ws_seq_ctr[b] = 0u;" in text
    assert len(re.findall(r"\bplane_producer<C>\(", text)) == 2
    assert len(re.findall(r"\bper_sequence<\w+, C::kPartCols>\(", text)) == 4, "at every end of a producer"


def test_no_cta_is_first_of_two_shared_segments():
    """The cut of the work in CTAs (the rule of sk_range), played through: the index of a ticket is one segment's."""
    rng = random.Random(5)
    for _ in range(300):
        n_cta, units = rng.choice([1, 7, 148]), [rng.choice([0, 1, 3, 50, 900]) for _ in range(rng.randint(1, 60))]
        if rng.random() < 0.3:
            units = [rng.randint(1, 900)] * rng.randint(1, n_cta)
        segs, total = [u for u in units], sum(units)
        if not total:
            continue
        c = n_cta // len(segs)
        if len(set(segs)) == 1 and c >= 1 and c * len(segs) * 100 >= 85 * n_cta:
            q = -(-segs[0] // c)
            spans = [(s * c * q, s * c * q + u) for s, u in enumerate(segs)]
        else:
            q = -(-total // n_cta)
            spans = [(sum(segs[:s]), sum(segs[:s + 1])) for s in range(len(segs)) if segs[s]]
        first = [lo // q for lo, hi in spans if (hi - 1) // q > lo // q]
        assert len(first) == len(set(first)) and all(0 <= f < n_cta for f in first)


def _problem(lens, Hkv, G, n_q, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    need = [(n + 15) // 16 for n in lens]
    nb, table, pos = max(1, sum(need)), torch.zeros(len(lens), max(need), dtype=torch.int32), 0
    for b, n in enumerate(need):
        table[b, :n] = torch.arange(pos, pos + n, dtype=torch.int32)
        pos += n
    K, V = (lynx.split_quantize(torch.randn(nb, Hkv, 16, 128, generator=g, device="cuda").to(torch.bfloat16)) for _ in range(2))
    q = torch.randn(len(lens), n_q, Hkv * G, 128, generator=g, device="cuda").to(torch.bfloat16)
    geo = lynx.Geometry(Hkv * G, Hkv, 16, nb, max(need))
    args = (geo, q, K, V, table.cuda(), torch.tensor(lens, dtype=torch.int32, device="cuda"))
    return lambda ws: _calls(args, ws, geo, len(lens), n_q)


def _calls(args, ws, geo, B, n_q):
    draft = lynx.anchor_attention(*args, ws, causal=True)
    out, first, dev = (t.fill_(7) for t in (torch.empty_like(draft), torch.empty(B, dtype=torch.int32, device="cuda"), torch.empty(B, n_q, device="cuda")))
    lynx.merge_verify_attention(*args, ws, draft_out=draft, atol=0.5, rtol=0.1, out_full=out, first_reject=first, dev=dev)
    lse = lynx.workspace_lse(geo, B, n_q, ws).clone()
    lynx.check(ws)
    return [draft, out, first, dev, lse]


@pytest.mark.gpu
def test_batches_take_turns_on_one_workspace():
    """A large batch whose heads are shared between neighbouring CTAs, one long sequence, and windows in between, on one workspace:
    the same bits as on a workspace of its own, every time."""
    probs = [_problem([200 + 3 * (i % 50) for i in range(256)], 8, 4, 1, 1), _problem([20000], 8, 4, 4, 2),
             _problem([0 if i % 7 == 0 else 130 + i for i in range(60)], 2, 8, 8, 3), _problem([9000, 131], 1, 4, 8, 4)]
    geo = lynx.Geometry(64, 8, 16, 1 << 16, 2000)
    size = lynx.workspace_bytes(geo, 256, 16)
    fresh = lambda: torch.zeros(size, dtype=torch.uint8, device="cuda")  # noqa: E731
    want = [f(fresh()) for f in probs]
    ws = fresh()
    for i in (0, 1, 0, 2, 0, 3, 1, 2, 0, 3, 2, 1, 0):
        for a, b in zip(probs[i](ws), want[i]):
            assert torch.equal(a, b)
