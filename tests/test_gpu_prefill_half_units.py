"""The state pass with two CTAs per (sequence, v-head) unit, on either side of the lines where it is taken (148 SMs) and with more
half units than SMs, so that a CTA goes from one to the next: unequal lengths, empty sequences and padding slots in
between, states in place."""
import numpy as np
import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I
from test_gpu_prefill import oracle_prefill

pytestmark = pytest.mark.gpu


def run(p, slots, num_slots, alias, hint, split=None):
    from paper_2607_17979_b200 import api
    pool = U.dev(p["init_state"])
    final = pool if alias else torch.full((num_slots, p["Hv"], 128, 128), 7.0, device="cuda")
    o = torch.full((p["T"], p["Hv"], 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(api.gdn_prefill_workspace_bytes(p["T"], p["N"], p["Hqk"], p["Hv"]), dtype=torch.uint8, device="cuda")
    api.gdn_prefill(U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), U.dev_bf16(p["v"]), U.dev(p["g"]), U.dev(p["beta"]),
                    U.dev(p["cu_seqlens"]), pool, final, U.dev(slots), o, p["scale"], ws, max_seqlen_hint=hint,
                    dev_status=status, route="stream" if split is None else "overlap",
                    split_permille=-1 if split is None else split)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return U.host_f64_from_bf16(o), final.cpu().numpy()


@pytest.mark.parametrize("alias", [False, True])
@pytest.mark.parametrize("lens, hv", [
    ([1000, 64, 65, 0, 129, 7, 63, 1] * 3, 8),         # 192 units, hint 1000: half units, several a CTA, ragged unit changes
    ([640] + [1, 64, 0] * 12, 4),                      # 148 units, one long chain among single tokens
    ([130 - i % 67 for i in range(37)], 2),            # 74 units: one half unit per SM
    ([700, 650], 32),                                  # 64 units, equal chains
    ([4096 // 64] * 2 + [300], 2),                     # a handful
])
def test_half_units(lens, hv, alias):
    n = len(lens)
    p = I.prefill_inputs(lens, max(hv // 2, 1), hv, seed=9900 + n + hv, alpha_lo=0.5, init="normal")
    slots = np.arange(n, dtype=np.int32)[::-1].copy()
    slots[3::7] = -1
    o, S = run(p, slots, n, alias, max(lens))
    o_ref, S_ref, _ = oracle_prefill(p, slot_idx=slots, num_slots=n)
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    used = np.sort(slots[slots >= 0])
    unused = np.setdiff1d(np.arange(n), used)
    for s in used:
        U.check_state(S[s:s + 1].astype(np.float64), S_ref[s:s + 1], U.STATE_REL_L2_PREFILL)
    assert np.array_equal(S[unused], p["init_state"][unused] if alias else np.full_like(S[unused], 7.0))


@pytest.mark.parametrize("hv, n", [(70, 1), (35, 2), (71, 1)])
def test_two_parts_at_the_last_unit_count_that_has_them(hv, n):
    """70 units leave eight of 148 SMs to the producers; with 71 the three launches run."""
    p = I.prefill_inputs([400 - 90 * i for i in range(n)], hv, hv, seed=9950 + hv, alpha_lo=0.5, init="normal")
    slots = np.arange(n, dtype=np.int32)
    o, S = run(p, slots, n, False, 400, split=200)
    o2, S2 = run(p, slots, n, False, 400)
    o_ref, S_ref, _ = oracle_prefill(p, slot_idx=slots, num_slots=n)
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
    assert np.array_equal(o, o2) and np.array_equal(S, S2)
