"""Verification with 17..32 columns goes through integer products for the values where a table gives CTAs 24 units of 128 tokens and
has room for five in a sequence: many short sequences in a table of their own width do not (they would lose by it), few long ones do.
By the names of the kernels of a captured call."""
import ctypes

import pytest
import torch

import paper_2607_01831_b200 as lynx

pytestmark = pytest.mark.gpu


class _KernelNode(ctypes.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("dims", ctypes.c_uint * 7), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def _kernels(call):
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    cu = ctypes.CDLL("libcuda.so.1")
    graph, n = ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    names = []
    for node in nodes:
        p, name = _KernelNode(), ctypes.c_char_p()
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
        assert (cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)) if p.func else cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kern))) == 0
        names.append(name.value.decode())
    return names


@pytest.mark.parametrize("B,H,blocks,ints", [(200, 8, 32, False), (1200, 2, 32, False), (1200, 2, 33, True), (1, 4, 7103, False), (1, 4, 7104, True),
                                            (1, 4, 113600 // 16, False), (1, 4, 131072 // 16, True)])   # (tables of test_gpu_verify_wide_precision.py)
def test_variant(B, H, blocks, ints):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 148:
        pytest.skip("sizes for 148 SMs")
    K, V = (lynx.split_quantize(torch.zeros(1, H, 16, 128, dtype=torch.bfloat16, device="cuda")) for _ in range(2))
    geo = lynx.Geometry(H * 4, H, 16, 1, blocks)
    table = torch.zeros(B, blocks, dtype=torch.int32, device="cuda")
    lens = torch.full((B,), 16, dtype=torch.int32, device="cuda")
    q = torch.zeros(B, 8, H * 4, 128, dtype=torch.bfloat16, device="cuda")
    ws = lynx.make_workspace(geo, B, 8, "cuda")
    out = torch.empty(q.shape, device="cuda")
    names = _kernels(lambda: lynx.merge_verify_attention(geo, q, K, V, table, lens, ws, out_full=out))
    assert any(f"attn_f16_kernelILi32ELb{int(ints)}E" in n for n in names), names
