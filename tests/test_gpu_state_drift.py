"""The recurrent state over hundreds of consecutive calls on one pool, with no decay that would forget
an earlier call's error: roundings to nearest walk at random, a one-sided error adds up call by call."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2607_17979_b200 import inputs as I
import gpu_util as U

pytestmark = pytest.mark.gpu

CALLS = 400
# One rounding to nearest per element and call: relative error uniform within half an ulp, 2^-24 / sqrt(3) for a
# significand of 1 and less above it, 2.5e-8 on average.  Independent roundings: 2.5e-8 sqrt(400) = 5e-7.
# Four times that; an error of the same size but of one sign would reach 1e-5.
BOUND = 4 * 2.5e-8 * CALLS ** 0.5


def drift(L, step, transposed=False):
    """Relative state error after CALLS calls of L tokens; step(pool, inputs) makes one call."""
    first = I.decode_multi_inputs(1, L, 1, 2, 128, 1, seed=400)
    tiles = lambda x: np.ascontiguousarray(x.transpose(0, 1, 3, 2)) if transposed else x
    pool, ref = U.dev(tiles(first["state"])), first["state"].astype(np.float64)
    for c in range(CALLS):
        d = I.decode_multi_inputs(1, L, 1, 2, 128, 1, seed=10000 + c)
        d["g"] = np.zeros_like(d["g"])              # alpha = 1
        d["beta"] = (d["beta"] * 1e-3).astype(np.float32)
        step(pool, d)
        for t in range(L):
            row = lambda a: np.ascontiguousarray(a[:, t])
            oracle.decode(row(d["q"]), row(d["k"]), row(d["v"]), row(d["g"]), row(d["beta"]), ref, None, d["scale"])
    torch.cuda.synchronize()
    return U.rel_l2(tiles(pool.cpu().numpy()).astype(np.float64), ref)


@pytest.mark.parametrize("L", [1, 4, 8, 16])
@pytest.mark.parametrize("layout", [0, 1])
def test_multi_token_decode(layout, L):
    from paper_2607_17979_b200 import api

    def step(pool, d):
        o = torch.empty((1, L, 2, 128), dtype=torch.bfloat16, device="cuda")
        api.gdn_decode_multi(U.dev_bf16(d["q"]), U.dev_bf16(d["k"]), U.dev_bf16(d["v"]), U.dev(d["g"]), U.dev(d["beta"]),
                             pool, None, o, d["scale"], layout)

    assert drift(L, step, transposed=layout == api.STATE_KV) < BOUND


@pytest.mark.parametrize("L", [3, 7, 16, 40])
def test_short_prompts_that_continue(L):
    """(40 tokens are three blocks, so three roundings per element and call)"""
    from paper_2607_17979_b200 import api
    ws = torch.empty(api.gdn_prefill_workspace_bytes(L, 1, 1, 2), dtype=torch.uint8, device="cuda")
    cu = torch.tensor([0, L], dtype=torch.int32, device="cuda")

    def step(pool, d):
        o = torch.empty((L, 2, 128), dtype=torch.bfloat16, device="cuda")
        api.gdn_prefill(U.dev_bf16(d["q"][0]), U.dev_bf16(d["k"][0]), U.dev_bf16(d["v"][0]), U.dev(d["g"][0]),
                        U.dev(d["beta"][0]), cu, pool, pool, None, o, d["scale"], ws)

    assert drift(L, step) < BOUND * math.ceil(L / 16) ** 0.5
