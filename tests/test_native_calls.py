"""The extension behind the per-step calls does what their Python bodies do: the same bits, objects and errors on the GPU, and it
leaves alone (returns None for) whatever is not a plain GPU tensor."""
import threading
import warnings

import pytest
import torch

import paper_2607_01831_b200 as lynx

D = 128


def _native():
    lynx.load()
    from paper_2607_01831_b200 import _native as n
    return n


def test_what_is_not_plain_is_left_alone():
    n = _native()
    geo = lynx.Geometry(8, 2, 16, 4, 4)
    q = torch.zeros(1, 1, 8, D, dtype=torch.bfloat16)
    planes = lynx.alloc_planes((4, 2, 16), "cpu")
    i = torch.zeros(1, 4, dtype=torch.int32)
    ws = torch.zeros(64, dtype=torch.uint8)
    assert n.anchor_attention(geo, q, planes, planes, i, i, ws, False, 0.0, None) is None
    assert n.anchor_attention(geo, None, planes, planes, i, i, ws, False, 0.0, None) is None
    assert n.anchor_attention(object(), q, planes, planes, i, i, ws, False, 0.0, None) is None
    assert n.anchor_attention(geo, q) is None
    assert n.merge_verify_attention(geo, q, planes, planes, i, i, ws, None, 0.0, 0.0, True, 0.0, None, None, None) is None
    assert n.bf16_attention(geo, q, q, q, i, i, ws, False, 0.0, None) is None
    assert n.split_quantize(q, planes, None, 0) is None
    assert n.recombine(planes, True, False) is None
    assert n.lse_view(geo, 1, 1, ws, False) is None
    assert n.lse_merge(q.float(), q.float(), q.float(), q.float(), None, False) is None
    assert n.hier_quantize(torch.zeros(1, 256, D, dtype=torch.bfloat16)) is None
    assert n.hier_dequantize(ws, None, ws, ws, ws, ws, None) is None
    with pytest.raises(lynx.LynxError, match="device tensors"):
        lynx.anchor_attention(geo, q, planes, planes, i, i, ws)
    with pytest.raises(lynx.LynxError, match="q must be"):
        lynx.anchor_attention(geo, q.float(), planes, planes, i, i, ws)


@pytest.fixture
def unresolved(monkeypatch):
    """The module as before its first call."""
    lynx.load()
    for v in [v for v in vars(lynx) if v.startswith("_fast_")]:
        monkeypatch.setattr(lynx, v, lynx._fast(v, "recombine"))
    lynx._extension.cache_clear()
    yield monkeypatch
    lynx._extension.cache_clear()


def test_an_extension_for_another_torch_is_not_used(unresolved):
    assert _native().torch_version == torch.__version__ and lynx._extension() is _native()
    lynx._extension.cache_clear()
    unresolved.setattr(torch, "__version__", "2.12.0+cu130")
    with pytest.warns(RuntimeWarning, match="built for torch"):
        assert lynx._fast_recombine(None, True, False) is None
    assert lynx._fast_recombine is lynx._python_only
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        assert lynx._fast_anchor() is None        # said once


def test_an_extension_that_does_not_load_is_said(unresolved):
    import sys
    unresolved.setitem(sys.modules, "paper_2607_01831_b200._native", None)
    unresolved.delattr(lynx, "_native", raising=False)
    with pytest.warns(RuntimeWarning, match="not used"):
        assert lynx._fast_recombine(None, True, False) is None


def test_the_library_is_built_without_its_extension(monkeypatch, tmp_path):
    from paper_2607_01831_b200 import build as b
    assert not b._native_stale()
    monkeypatch.setattr(torch, "__version__", "2.12.0+cu130")
    assert b._native_stale() and not b._stale()
    monkeypatch.setattr(b, "_native_cmd", lambda out: ["false"])
    monkeypatch.setattr(b, "_build_library", lambda verbose: pytest.fail("the library is there"))
    with pytest.warns(UserWarning, match="was not built"):
        assert b.build() == b.LIB


def _everything(seed, stream=None):
    """Every call with an extension function, on inputs of a seed."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    with torch.cuda.stream(stream or torch.cuda.current_stream()):
        nb, Hkv, G, B, k = 9, 2, 4, 2, 3
        src = [torch.randn(nb, Hkv, 16, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
        K, V = lynx.split_quantize(src[0]), lynx.split_quantize(src[1], out=lynx.alloc_planes((nb, Hkv, 16), "cuda"))
        part = lynx.Planes(*(torch.zeros_like(t) for t in (K.anchor, K.residual, K.meta)))
        lynx.split_quantize(src[0], out=part, block_ids=torch.tensor([1, 5], dtype=torch.int32, device="cuda"), rows_per_block=Hkv * 16)
        geo = lynx.Geometry(Hkv * G, Hkv, 16, nb, 4)
        table = torch.tensor([[0, 1, 2, 3], [4, 5, 6, 7]], dtype=torch.int32, device="cuda")
        lens = torch.tensor([50, 64], dtype=torch.int32, device="cuda")
        q = torch.randn(B, k, Hkv * G, D, generator=g, device="cuda").to(torch.bfloat16)
        ws = lynx.make_workspace(geo, B, k, "cuda")
        draft = lynx.anchor_attention(geo, q, K, V, table, lens, ws, causal=True)
        lse = lynx.workspace_lse(geo, B, k, ws).clone()
        given = torch.empty_like(draft)
        assert lynx.anchor_attention(geo, q, K, V, table, lens, ws, causal=True, softmax_scale=0.1, out=given) is given
        full, first, dev = lynx.merge_verify_attention(geo, q, K, V, table, lens, ws, draft_out=draft, atol=0.5, rtol=0.1)
        alone = lynx.merge_verify_attention(geo, q, K, V, table, lens, ws)
        assert alone[1] is None and alone[2] is None
        codes, none = lynx.recombine(K)
        assert none is None
        _, kp = lynx.recombine(K, want_codes=False, want_bf16=True)
        _, vp = lynx.recombine(V, want_codes=False, want_bf16=True)
        n = int(lynx.load().lynx_bf16_workspace_bytes(geo._c(), B, k))
        ws2 = torch.zeros(n, dtype=torch.uint8, device="cuda")
        pages = lynx.bf16_attention(geo, q, kp, vp, table, lens, ws2, causal=True)
        lse2 = lynx.bf16_workspace_lse(geo, B, k, ws2).clone()
        joined, jl = lynx.lse_merge(draft, lse, pages, lse2, want_lse=True)
        h = lynx.hier_quantize(torch.randn(3, 256, D, generator=g, device="cuda").to(torch.bfloat16))
        back = [lynx.hier_dequantize(h), lynx.hier_dequantize(h, anchor_only=True)]
        out = [K.anchor, K.residual, K.meta, V.anchor, part.anchor, part.meta, draft, lse, given, full, first, dev, alone[0], codes, kp, vp, pages,
               lse2, joined, jl, lynx.lse_merge(draft, lse, pages, lse2), h.q_anc, h.q_res, h.gamma_min, h.gamma_scale, h.mu, h.sigma, *back]
    return out


def _python(monkeypatch):
    for v in [v for v in vars(lynx) if v.startswith("_fast_")]:
        monkeypatch.setattr(lynx, v, lynx._python_only)


@pytest.mark.gpu
def test_same_as_the_python_bodies(monkeypatch):
    got = _everything(3)
    assert lynx._fast_anchor is _native().anchor_attention
    _python(monkeypatch)
    want = _everything(3)
    for i, (a, b) in enumerate(zip(got, want)):
        assert a.dtype == b.dtype and a.shape == b.shape and a.stride() == b.stride() and a.device == b.device, i
        assert torch.equal(a.view(torch.uint8) if a.is_floating_point() else a, b.view(torch.uint8) if b.is_floating_point() else b), i


@pytest.mark.gpu
@pytest.mark.parametrize("python", [False, True])
def test_same_errors(monkeypatch, python):
    if python:
        _python(monkeypatch)
    K = lynx.split_quantize(torch.zeros(4, 2, 16, D, dtype=torch.bfloat16, device="cuda"))
    geo = lynx.Geometry(8, 2, 16, 4, 4)
    table, lens = torch.zeros(1, 4, dtype=torch.int32, device="cuda"), torch.full((1,), 20, dtype=torch.int32, device="cuda")
    q = torch.zeros(1, 1, 8, D, dtype=torch.bfloat16, device="cuda")
    ws = lynx.make_workspace(geo, 1, 1, "cuda")
    ok = lambda **k: lynx.anchor_attention(**{**dict(geo=geo, q=q, K=K, V=K, block_table=table, seq_lens=lens, workspace=ws), **k})  # noqa: E731
    ok()
    for match, kw in (("contiguous", dict(q=torch.zeros(1, 8, 1, D, dtype=torch.bfloat16, device="cuda").transpose(1, 2).expand(1, 1, 8, D)[:, :, ::1].as_strided((1, 1, 8, D), (8 * D, 8 * D, 0, 1)))),
                      ("q must be", dict(q=q.float())), ("status 5", dict(workspace=ws[:256])), ("status 3", dict(workspace=ws[4:])),
                      ("device tensors", dict(seq_lens=lens.cpu())), ("status 4", dict(geo=lynx.Geometry(8, 2, 24, 4, 4))),
                      ("contiguous", dict(out=torch.empty(1, 1, D, 8, device="cuda").transpose(2, 3)))):
        with pytest.raises(lynx.LynxError, match=match):
            ok(**kw)
    with pytest.raises(lynx.LynxError, match="draft_out must be"):
        lynx.merge_verify_attention(geo, q, K, K, table, lens, ws, draft_out=torch.zeros(1, 2, 8, D, device="cuda"), atol=1.0)
    with pytest.raises(lynx.LynxError, match="status 2"):
        lynx.merge_verify_attention(geo, q, K, K, table, lens, ws, draft_out=torch.zeros(1, 1, 8, D, device="cuda"), atol=0.0)
    with pytest.raises(lynx.LynxError, match="smaller"):
        lynx.workspace_lse(geo, 1, 1, ws[:256])


@pytest.mark.gpu
def test_threads_on_their_own_streams():
    want = [_everything(s) for s in range(4)]
    torch.cuda.synchronize()
    got = [None] * 4

    def work(i):
        for _ in range(3):
            s = torch.cuda.Stream()
            got[i] = _everything(i, s)
            s.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w, g in zip(want, got):
        assert g is not None and all(torch.equal(a, b) for a, b in zip(w, g))
