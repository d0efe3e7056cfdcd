"""The form in which the intra-chunk kernel is launched, read from a captured call: a grid of chunks x heads up to two items an SM, a
row of items (the CTAs without a chunk behind all others) from there to where the pipeline's one CTA per SM begins: five items an SM
by the host's bound, which counts a ragged chunk for each sequence, or four where the sequences would have fewer at equal lengths."""
import ctypes

import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I

pytestmark = pytest.mark.gpu


class KernelNode(ctypes.Structure):      # CUDA_KERNEL_NODE_PARAMS
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3), ("smem", ctypes.c_uint),
                ("args", ctypes.c_void_p), ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def grids(graph):
    """(threads a block, grid) of the graph's kernels."""
    cu = ctypes.CDLL("libcuda.so.1")
    n = ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(ctypes.c_void_p(graph), None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(ctypes.c_void_p(graph), nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        kn = KernelNode()
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(kn)) == 0
        out.append((kn.block[0], tuple(kn.grid)))
    return out


@pytest.mark.parametrize("lens, hv, form", [
    ([64 * 9], 8, "grid"),
    ([64] * 32, 8, "row"),               # 32 chunks of the 64 that T and N allow
    ([64 * 9], 32, "row"), ([64 * 20], 32, "row"),
    ([64] * 13, 32, "row"), ([48] * 16, 32, "row"), ([128] * 8, 32, "row"),      # more than five an SM by the bound, fewer than four in fact
    ([130] * 8, 32, "pipeline"), ([65] * 17, 32, "pipeline"), ([64 * 60], 32, "pipeline"),
])
def test_form(lens, hv, form):
    from paper_2607_17979_b200 import api
    p = I.prefill_inputs(lens, hv, hv, seed=61, init="zero")
    final = torch.empty((p["N"], hv, 128, 128), device="cuda")
    o = torch.empty((p["T"], hv, 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(api.gdn_prefill_workspace_bytes(p["T"], p["N"], hv, hv), dtype=torch.uint8, device="cuda")
    args = (U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), U.dev_bf16(p["v"]), U.dev(p["g"]), U.dev(p["beta"]),
            U.dev(p["cu_seqlens"]), None, final, None, o, p["scale"], ws)
    api.gdn_prefill(*args, route="stream")
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
        api.gdn_prefill(*args, route="stream")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    chunks = p["T"] // 64 + p["N"]
    want = {"grid": (256, (chunks, hv, 1)), "row": (256, (chunks * hv, 1, 1)), "pipeline": (800, (sms, 1, 1))}[form]
    assert want in grids(graph.raw_cuda_graph())
