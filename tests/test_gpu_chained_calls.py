"""Chains of calls on one stream, with no host synchronisation between them, against the same calls with a synchronisation
after each, bit for bit: every kernel sees what the kernels before it on the stream wrote -- also where its launch may begin
before they have ended, where buffers are reused with other contents from one round to the next, and on a stream other than
the default one."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

ROUNDS = 6


def _inputs(B, Hkv, G, n_q, bt, blocks):
    nb = B * blocks
    x = [synth.kv_block_values("student_t4", nb, Hkv, bt, "cuda", "ch", i).to(torch.bfloat16) for i in range(2 * ROUNDS)]
    q = [synth.queries(B, n_q, Hkv * G, "cuda", "chq", i) for i in range(ROUNDS)]
    g = torch.Generator().manual_seed(3)
    table = [torch.randperm(nb, generator=g).to(torch.int32).view(B, blocks).cuda() for _ in range(ROUNDS)]
    lens = [torch.randint(n_q, blocks * bt + 1, (B,), generator=g).to(torch.int32).cuda() for _ in range(ROUNDS)]
    return x, q, table, lens


def _chain(lynx, inputs, B, Hkv, G, n_q, bt, blocks, after):
    """ROUNDS rounds over the same buffers; `after` is called behind every step."""
    x, q, table, lens = inputs
    nb = B * blocks
    geo = lynx.Geometry(Hkv * G, Hkv, bt, nb, blocks)
    src = [torch.zeros_like(x[0]) for _ in range(2)]
    qq, tt, ll = torch.zeros_like(q[0]), torch.zeros_like(table[0]), torch.zeros_like(lens[0])
    K, V = (lynx.alloc_planes((nb, Hkv, bt), "cuda") for _ in range(2))
    ws = lynx.make_workspace(geo, B, n_q, "cuda")
    pages = [torch.zeros(nb, Hkv, bt, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    n = int(lynx.load().lynx_bf16_workspace_bytes(geo._c(), B, n_q))
    bf_ws = torch.zeros(n, dtype=torch.uint8, device="cuda")
    draft, full = (torch.zeros(B, n_q, Hkv * G, 128, device="cuda") for _ in range(2))
    out = []

    def rec(p, dst):
        lynx._ok(lynx.load().lynx_recombine(lynx._ptr(p.anchor), lynx._ptr(p.residual), lynx._ptr(p.meta), nb * Hkv * bt, None,
                                            lynx._ptr(dst), lynx._stream()), "recombine")
    for i in range(ROUNDS):
        for step in (lambda: src[0].copy_(x[2 * i]), lambda: src[1].copy_(x[2 * i + 1]), lambda: qq.copy_(q[i]),
                     lambda: tt.copy_(table[i]), lambda: ll.copy_(lens[i]),
                     lambda: lynx.split_quantize(src[0], out=K), lambda: lynx.split_quantize(src[1], out=V),
                     lambda: lynx.anchor_attention(geo, qq, K, V, tt, ll, ws, causal=True, out=draft),
                     lambda: lynx.merge_verify_attention(geo, qq, K, V, tt, ll, ws, draft_out=draft, atol=0.05, rtol=0.05, out_full=full),
                     lambda: rec(K, pages[0]), lambda: rec(V, pages[1]),
                     lambda: lynx.bf16_attention(geo, qq, pages[0], pages[1], tt, ll, bf_ws, causal=True),
                     lambda: lynx.lse_merge(full, lynx.workspace_lse(geo, B, n_q, ws), draft, lynx.bf16_workspace_lse(geo, B, n_q, bf_ws)),
                     lambda: lynx.hier_dequantize(lynx.hier_quantize(src[0].view(-1, 256, 128))),
                     lambda: [t.clone() for t in (K.anchor, V.residual, V.meta, draft, full, *pages)]):
            got = step()
            after()
            if got is not None and not isinstance(got, lynx.Planes):
                out += [t for t in (got if isinstance(got, (list, tuple)) else [got])]
    lynx.check(ws)
    return [t.clone() for t in out]


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("G,n_q,blocks", [(4, 1, 24), (4, 4, 40), (4, 8, 200), (8, 8, 72)])
def test_chained_calls_equal_synchronised_ones(G, n_q, blocks, side_stream):
    import paper_2607_01831_b200 as lynx
    shape = (2, 2, G, n_q, 16, blocks)
    inputs = _inputs(*shape)
    torch.cuda.synchronize()
    want = _chain(lynx, inputs, *shape, torch.cuda.synchronize)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if side_stream else torch.cuda.current_stream()
    with torch.cuda.stream(stream):
        got = _chain(lynx, inputs, *shape, lambda: None)
    torch.cuda.synchronize()
    assert len(got) == len(want)
    for i, (a, b) in enumerate(zip(got, want)):
        assert torch.equal(a, b), i
