"""bench.py's count of kernels per attention call is what the calls launch: the kernel nodes of a captured call, over the conditions
that the dispatch has (few and many heads, sequences of one unit and of more, slices of positions, with and without a draft)."""
import ctypes

import pytest
import torch

import bench
import paper_2607_01831_b200 as lynx

pytestmark = pytest.mark.gpu


def _nodes(call):
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    n = ctypes.c_size_t(0)
    assert ctypes.CDLL("libcudart.so.12").cudaGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("n_q", [1, 4, 8, 17, 64])
@pytest.mark.parametrize("B,Hkv,G,tokens", [(1, 2, 4, 100), (1, 2, 4, 300), (40, 1, 4, 100), (40, 1, 4, 300), (36, 1, 1, 129), (37, 1, 8, 128)])
def test_counts(B, Hkv, G, tokens, n_q):
    blocks = (tokens + 15) // 16
    K, V = (lynx.split_quantize(torch.zeros(blocks, Hkv, 16, 128, dtype=torch.bfloat16, device="cuda")) for _ in range(2))
    geo = lynx.Geometry(Hkv * G, Hkv, 16, blocks, blocks)
    table = torch.arange(blocks, dtype=torch.int32, device="cuda").repeat(B, 1)
    lens = torch.full((B,), tokens, dtype=torch.int32, device="cuda")
    q = torch.zeros(B, n_q, Hkv * G, 128, dtype=torch.bfloat16, device="cuda")
    ws = lynx.make_workspace(geo, B, n_q, "cuda")
    out, first, dev = torch.empty(q.shape, device="cuda"), torch.empty(B, dtype=torch.int32, device="cuda"), torch.empty(B, n_q, device="cuda")
    draft = torch.zeros_like(out)
    sms, cap = torch.cuda.get_device_properties(0).multi_processor_count, blocks * 16
    count = lambda full, d: bench.attention_kernels(B, Hkv, G, n_q, cap, sms, full, d)  # noqa: E731
    assert _nodes(lambda: lynx.anchor_attention(geo, q, K, V, table, lens, ws, out=out)) == count(False, False)
    verify = lambda **kw: lynx.merge_verify_attention(geo, q, K, V, table, lens, ws, out_full=out, first_reject=first, dev=dev, **kw)  # noqa: E731
    assert _nodes(lambda: verify()) == count(True, False)
    assert _nodes(lambda: verify(draft_out=draft, atol=0.5, rtol=0.1)) == count(True, True)
