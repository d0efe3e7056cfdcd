"""The intra-chunk kernel's items run as a grid of chunks x heads up to two items an SM and as a row of items, last chunks first,
beyond: both against the oracle on either side of the line, with and without a table launch and with CTAs that have no chunk."""
import numpy as np
import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I
from test_gpu_prefill import oracle_prefill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens, hqk, hv", [
    ([64 * 70], 1, 4),                  # below the line, one sequence
    ([64 * 80 + 1], 1, 4),              # above it
    ([64 * 297], 1, 1),                 # one head: a row whatever the number
    ([1, 0, 65, 3] * 8, 4, 8),          # above it, 24 chunks of the 40 that T and N allow
    ([5, 130, 0] * 11, 2, 4),           # 33 sequences: table launch; below it
    ([5, 130, 0] * 11, 5, 10),          # above it, a number of heads that is no power of two
])
def test_item_order(lens, hqk, hv):
    from paper_2607_17979_b200 import api
    p = I.prefill_inputs(lens, hqk, hv, seed=7700 + hv, alpha_lo=0.5, init="zero")
    o_ref, S_ref, _ = oracle_prefill(p, init=None)
    final = torch.empty((p["N"], p["Hv"], 128, 128), device="cuda")
    o = torch.empty((p["T"], p["Hv"], 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.full((api.gdn_prefill_workspace_bytes(p["T"], p["N"], hqk, hv),), 0xff, dtype=torch.uint8, device="cuda")
    api.gdn_prefill(U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), U.dev_bf16(p["v"]), U.dev(p["g"]), U.dev(p["beta"]),
                    U.dev(p["cu_seqlens"]), None, final, None, o, p["scale"], ws, route="stream")
    torch.cuda.synchronize()
    U.check_o(U.host_f64_from_bf16(o), o_ref, U.O_REL_L2_PREFILL)
    U.check_state(final.cpu().numpy().astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
