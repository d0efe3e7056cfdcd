"""gdn_prefill_route names the route that gdn_prefill takes: the launches of a captured call are that route's."""
import ctypes

import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I

pytestmark = pytest.mark.gpu


def launches(graph):
    n = ctypes.c_size_t(0)
    rt = ctypes.CDLL("libcudart.so.12")
    assert rt.cudaGraphGetNodes(ctypes.c_void_p(graph), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("lens, hv, hint, route, nodes", [
    ([12], 4, 0, "recurrent", 1), ([48], 8, 0, "blocks", 1),
    ([130], 32, 0, "stream", 2), ([2495], 32, 0, "stream", 2), ([40] * 40, 4, 40, "stream", 3),     # with a table launch
    ([2496], 32, 0, "overlap", 5), ([6100, 2000], 32, 6100, "overlap", 5),
    ([4096, 4096], 32, 4096, "stream", 2), ([6100, 2000], 32, 0, "stream", 2),
    ([512, 1024, 2048, 4096], 32, 4096, "stream", 2),               # the benchmark's
])
def test_route_is_what_runs(lens, hv, hint, route, nodes):
    from paper_2607_17979_b200 import api
    p = I.prefill_inputs(lens, hv, hv, seed=31, init="zero")
    assert api.gdn_prefill_route(p["T"], p["N"], hint, hv, torch.cuda.get_device_properties(0).multi_processor_count) == route
    final = torch.empty((p["N"], hv, 128, 128), device="cuda")
    o = torch.empty((p["T"], hv, 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(api.gdn_prefill_workspace_bytes(p["T"], p["N"], hv, hv), dtype=torch.uint8, device="cuda")
    args = (U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), U.dev_bf16(p["v"]), U.dev(p["g"]), U.dev(p["beta"]),
            U.dev(p["cu_seqlens"]), None, final, None, o, p["scale"], ws)
    api.gdn_prefill(*args, max_seqlen_hint=hint)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
        api.gdn_prefill(*args, max_seqlen_hint=hint)
    assert launches(graph.raw_cuda_graph()) == nodes
    if lens == [512, 1024, 2048, 4096]:
        assert nodes == api.LAUNCHES_PER_PREFILL
