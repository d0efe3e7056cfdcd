"""Two parts whose launches do not run side by side: what that costs."""
import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens, hv", [([2560], 32), ([16384], 8)])
def test_serialised_launches_lose_less_than_a_millisecond_beyond_the_work_done_twice(lens, hv):
    """Serialised on purpose (split_permille = -2): the chains give up soon after their first missing record, the other launches
    take at most what the three launches take, and the chains' work so far is lost."""
    from paper_2607_17979_b200 import api
    p = I.prefill_inputs(lens, hv // 2, hv, seed=55, init="zero")
    final = torch.empty((p["N"], hv, 128, 128), device="cuda")
    o = torch.empty((p["T"], hv, 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(api.gdn_prefill_workspace_bytes(p["T"], p["N"], hv // 2, hv), dtype=torch.uint8, device="cuda")
    args = (U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), U.dev_bf16(p["v"]), U.dev(p["g"]), U.dev(p["beta"]),
            U.dev(p["cu_seqlens"]), None, final, None, o, p["scale"], ws)

    def ms(route, split):
        best = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            api.gdn_prefill(*args, route=route, split_permille=split)
            b.record()
            torch.cuda.synchronize()
            best.append(a.elapsed_time(b))
        return min(best)

    three = ms("stream", -1)
    out = (o.clone(), final.clone())
    assert ms("overlap", -2) < 2 * three + 1.0
    assert torch.equal(o, out[0]) and torch.equal(final, out[1])
