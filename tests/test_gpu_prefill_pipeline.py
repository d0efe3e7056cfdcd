"""The intra-chunk kernel as a pipeline (more than five items an SM) against the oracle, at chunk lengths on either side of its 16-
and 32-token steps, with and without a table launch; and against the CTA-per-item form, whose results it repeats bit for bit: the
same sequences in a batch small enough for that one."""
import numpy as np
import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I
from test_gpu_prefill import oracle_prefill

pytestmark = pytest.mark.gpu


def run(p, lo, hi):
    """Sequences lo .. hi - 1 of the batch by themselves."""
    from paper_2607_17979_b200 import api
    cu = p["cu_seqlens"].astype(np.int64)
    t0, t1, n = int(cu[lo]), int(cu[hi]), hi - lo
    sub = {k: np.ascontiguousarray(p[k][t0:t1]) for k in ("q", "k", "v", "g", "beta")}
    Hqk, Hv = p["q"].shape[1], p["v"].shape[1]
    final = torch.empty((n, Hv, 128, 128), device="cuda")
    o = torch.empty((t1 - t0, Hv, 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.full((api.gdn_prefill_workspace_bytes(t1 - t0, n, Hqk, Hv),), 0xff, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.gdn_prefill(U.dev_bf16(sub["q"]), U.dev_bf16(sub["k"]), U.dev_bf16(sub["v"]), U.dev(sub["g"]), U.dev(sub["beta"]),
                    U.dev((cu[lo:hi + 1] - t0).astype(np.int32)), U.dev(np.ascontiguousarray(p["init_state"][lo:hi])), final, None, o,
                    p["scale"], ws, route="stream", dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return U.host_f64_from_bf16(o), final.cpu().numpy()


@pytest.mark.parametrize("lens, hqk, hv", [
    ([64 * 33 + t for t in (1, 15, 16, 17, 31, 32)], 1, 4),          # 816 items, no table launch
    ([33, 47, 48, 49, 63, 64, 65, 96, 97, 112, 113, 128] * 3, 8, 24),    # 36 sequences: table launch
    ([5] * 40 + [640], 3, 18),                                       # chunks of one block before full ones
])
def test_against_the_oracle_and_the_form_for_few_items(lens, hqk, hv):
    p = I.prefill_inputs(lens, hqk, hv, seed=8100 + hv, alpha_lo=0.5, init="normal")
    assert sum((n + 63) // 64 for n in lens) * hv > 740
    o, S = run(p, 0, len(lens))
    o_ref, S_ref, _ = oracle_prefill(p)
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
    cu = p["cu_seqlens"]
    for lo in (0, len(lens) - 1):       # a sequence by itself is few items
        o1, S1 = run(p, lo, lo + 1)
        U.check_o(o1, o_ref[cu[lo]:cu[lo + 1]], U.O_REL_L2_PREFILL)
        # (the state pass may run in the other form, whole units or half ones, which round alike in the state only)
        assert np.linalg.norm(S1[0] - S[lo]) <= 1e-6 * np.linalg.norm(S[lo])
