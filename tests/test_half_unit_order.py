"""In the half-unit state pass the hand-over of a state may be overtaken by the next one while output warps still wait for it, by
one and no more: a wait by parity cannot tell a phase from the one after the next, so the hand-overs have two barriers in turn."""
import os
import re

import numpy as np
import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I
from test_gpu_prefill import oracle_prefill

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")


def test_hand_overs_of_the_state_alternate_between_two_barriers():
    s = open(os.path.join(CSRC, "gdn_prefill_half.cuh")).read()
    for wait in ("warp_wait(&bar_s[g & 1][0], (g >> 1) & 1u", "warp_wait(&bar_s[g & 1][1], (g >> 1) & 1u",
                 "await(&bar_s[(g + 1) & 1][1], ((g + 1) >> 1) & 1u)"):
        assert s.count(wait) == 1
    assert len(re.findall(r"(?:wait|await)\(&bar_s\[", s)) == 3
    arrivals = re.findall(r"hand_over\(&bar_s(.+)\);", s)
    assert arrivals == ["[gc & 1][ch]", "[(g + 1) & 1][ch]"]
    # what bounds the lead: the next U~ is put in place by the warps that wait, behind their rows
    out = s[s.index("===================== output warps"):]
    assert out.index("preload(g + k)") < out.index("await(&bar_s[")


@pytest.mark.gpu
def test_ragged_tails_between_units_many_times():
    """Several half units a CTA with ragged tails, whose rows the output warps write slowly: no call runs into a wait's limit."""
    from paper_2607_17979_b200 import api
    p = I.prefill_inputs([1337, 512, 199], 16, 32, seed=77, init="normal")
    pool = U.dev(p["init_state"])
    o = torch.empty((p["T"], 32, 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(api.gdn_prefill_workspace_bytes(p["T"], p["N"], 16, 32), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    args = (U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), U.dev_bf16(p["v"]), U.dev(p["g"]), U.dev(p["beta"]), U.dev(p["cu_seqlens"]))
    final = torch.empty_like(pool)
    for _ in range(4000):
        api.gdn_prefill(*args, pool, final, None, o, p["scale"], ws, max_seqlen_hint=1337, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    o_ref, S_ref, _ = oracle_prefill(p)
    U.check_o(U.host_f64_from_bf16(o), o_ref, U.O_REL_L2_PREFILL)
    U.check_state(final.cpu().numpy().astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
