"""Chunked prefill with more (sequence, v-head) units than SMs, so that a CTA goes from one unit's final state
to the next one's initial state: unequal lengths, empty sequences and padding slots in between, states in place."""
import numpy as np
import pytest

import gpu_util as U
from paper_2607_17979_b200 import inputs as I
from test_gpu_prefill import oracle_prefill, run_prefill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("route", ["stream", "fused", "overlap"])
@pytest.mark.parametrize("alias", [False, True])
@pytest.mark.parametrize("lens", [[1] * 20, [64, 65, 0, 129, 7] * 8, [200] + [1, 63, 0] * 12])
def test_unit_changes(lens, alias, route):
    n = len(lens)
    p = I.prefill_inputs(lens, 4, 16, seed=9700 + n, alpha_lo=0.5, init="normal")
    slots = np.arange(n, dtype=np.int32)[::-1].copy()
    slots[3::7] = -1
    o, S, status = run_prefill(p, route, slot_idx=slots, num_slots=n, alias=alias, pool_fill=7.0)
    o_ref, S_ref, _ = oracle_prefill(p, slot_idx=slots, num_slots=n)
    assert status == 0
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    used = np.sort(slots[slots >= 0])
    unused = np.setdiff1d(np.arange(n), used)
    for s in used:
        U.check_state(S[s:s + 1].astype(np.float64), S_ref[s:s + 1], U.STATE_REL_L2_PREFILL)
    assert np.array_equal(S[unused], p["init_state"][unused] if alias else np.full_like(S[unused], 7.0))


@pytest.mark.parametrize("n, hv", [(37, 2), (75, 1), (37, 4), (149, 1)])
def test_record_forms(n, hv):
    """Half as many units as SMs and one more, as many and one more (148 SMs), where the state pass takes two CTAs
    per unit and one: the two-part entry point, which runs the three launches for such batches, gives the same bits."""
    p = I.prefill_inputs([130 - i % 67 for i in range(n)], 1, hv, seed=9800 + n + hv, alpha_lo=0.5, init="normal")
    o, S, status = run_prefill(p, "stream")
    o2, S2, status2 = run_prefill(p, "overlap", split_permille=300)
    o_ref, S_ref, _ = oracle_prefill(p)
    assert status == 0 and status2 == 0
    assert np.array_equal(o, o2) and np.array_equal(S, S2)
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
