"""Chunks with fewer than 64 tokens: only the 16-token blocks that hold tokens are written, copied and read, so whatever an
earlier chunk has left in shared memory must not reach the result, not even an infinity or a NaN."""
import numpy as np
import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I
from test_gpu_prefill import oracle_prefill

pytestmark = pytest.mark.gpu

TAILS = [1, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64]


def run(p, poison, route, hint):
    from paper_2607_17979_b200 import api
    v = U.dev_bf16(p["v"])
    if poison:
        v[:p["cu_seqlens"][1]:3] = float("nan")
        v[1:p["cu_seqlens"][1]:3] = float("inf")
    final = torch.empty((p["N"], p["Hv"], 128, 128), device="cuda")
    o = torch.empty((p["T"], p["Hv"], 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.full((api.gdn_prefill_workspace_bytes(p["T"], p["N"], p["Hqk"], p["Hv"]),), 0xff, dtype=torch.uint8, device="cuda")
    api.gdn_prefill(U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), v, U.dev(p["g"]), U.dev(p["beta"]), U.dev(p["cu_seqlens"]), None,
                    final, None, o, p["scale"], ws, max_seqlen_hint=hint, route=route)
    torch.cuda.synchronize()
    return o, final


@pytest.mark.parametrize("route, hv, hinted", [
    ("stream", 4, False),       # 52 units: half units, one each
    ("stream", 16, True),       # 208 units, one chain of eight chunks: half units, several a CTA
    ("stream", 32, False),      # 416 units: whole units, several a CTA
    ("overlap", 4, False), ("fused", 4, False),
])
def test_tails_behind_a_poisoned_sequence(route, hv, hinted):
    lens = [512 if hinted else 130] + TAILS
    p = I.prefill_inputs(lens, hv // 2, hv, seed=9990 + hv, alpha_lo=0.5, init="zero")
    o_ref, S_ref, _ = oracle_prefill(p, init=None)
    o, S = run(p, False, route, 512 if hinted else 0)
    U.check_o(U.host_f64_from_bf16(o), o_ref, U.O_REL_L2_PREFILL)
    U.check_state(S.cpu().numpy().astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
    o_p, S_p = run(p, True, route, 512 if hinted else 0)
    assert not torch.isfinite(S_p[0]).all()
    assert torch.equal(o[lens[0]:], o_p[lens[0]:]) and torch.equal(S[1:], S_p[1:])
