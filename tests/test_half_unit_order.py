"""In the half-unit state pass the state product of a chunk waits for the output warps to be through with the chunk before: they
have then seen that chunk's successor's state handed over, which the one after must not overtake (a wait by parity cannot tell a
phase from the one after the next)."""
import os
import re

import numpy as np
import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I
from test_gpu_prefill import oracle_prefill

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")


def test_state_product_waits_for_the_rows_before():
    s = open(os.path.join(CSRC, "gdn_prefill_half.cuh")).read()
    issuers = s[s.index("===================== issuers"):s.index("===================== chain warps")]
    rows = issuers.index("warp_wait(&bar_y_read, (g - 1) & 1u")
    u = issuers.index("warp_wait(&bar_u, g & 1u")
    product = issuers.index("mma_ts_c<false>(tD4")
    assert rows < u < product and issuers.count("&bar_y_read") == 1
    out = s[s.index("===================== output warps"):]
    assert out.index("await(&bar_s[1], (g + 1) & 1u)") < out.index("mbar_arrive(&bar_y_read)")
    assert not re.search(r"bar_s\[0\]", out)


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
