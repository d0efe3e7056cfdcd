"""GPU parity of the token-block kernels (multi-token decode, short-prompt prefill) at the edges of
their blocks: every token count around the 4-, 8- and 16-token variants, both tile orientations, with
few tiles and with enough for the other launch shape, and prompts of one block, of several, and of
none, against the fp64 oracle."""
import numpy as np
import pytest

from paper_2607_17979_b200 import inputs as I
import gpu_util as U
from test_gpu_decode_multi import KV, VK, oracle_multi, run_multi
from test_gpu_prefill import oracle_prefill, run_prefill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", [VK, KV])
@pytest.mark.parametrize("B,Hv", [(2, 2), (40, 4)])
@pytest.mark.parametrize("L", [1, 3, 4, 5, 8, 9, 15, 16])
def test_decode_block_edges(layout, B, Hv, L):
    d = I.decode_multi_inputs(B, L, 1, Hv, 128, B + 2, seed=9000 + 10 * L + B, slots="perm", alpha_lo=0.5)
    o, pool, status = run_multi(d, layout)
    o_ref, pool_ref, _ = oracle_multi(d)
    assert status == 0
    U.check_o(o, o_ref, U.O_REL_L2_DECODE)
    touched = d["slot_idx"]
    assert U.rel_l2(pool[touched].astype(np.float64), pool_ref[touched]) < 1e-5
    untouched = np.setdiff1d(np.arange(B + 2), touched)
    assert np.array_equal(pool[untouched], d["state"][untouched])


@pytest.mark.parametrize("lens", [[1], [4, 3], [5], [8, 1, 0], [9], [16, 7], [17], [32, 33, 0, 15], [64], [48, 16, 1]])
@pytest.mark.parametrize("init", ["zero", "normal"])
@pytest.mark.parametrize("route", ["recurrent", "auto"])
def test_short_prompt_block_edges(lens, init, route):
    p = I.prefill_inputs(lens, 2, 4, seed=9500 + sum(lens), alpha_lo=0.5, init=init)
    o, S, status = run_prefill(p, route)
    o_ref, S_ref, _ = oracle_prefill(p)
    assert status == 0
    U.check_o(o, o_ref, U.O_REL_L2_DECODE)
    # (gdn_prefill sends more than 64 tokens, whose lengths it is not told, to the chunked kernels)
    blocks = route == "recurrent" or sum(lens) <= 64
    assert U.rel_l2(S.astype(np.float64), S_ref) < (1e-5 if blocks else U.STATE_REL_L2_PREFILL)
