"""The intra-chunk kernel's two forms, a persistent pipeline and a CTA per item: the pipeline on batches with empty sequences, one head
and far fewer chunks than the host's bound, against the oracle; and the same sequences in both, whose results are equal bit for bit
where the state pass runs in one form."""
import numpy as np
import pytest
import torch

import gpu_util as U
from paper_2607_17979_b200 import inputs as I
from test_gpu_prefill import oracle_prefill

pytestmark = pytest.mark.gpu


def form(lens, hv):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T, n = sum(lens), len(lens)
    return "few" if (T // 64 + n) * hv <= 5 * sms or n * -(-T // (64 * n)) * hv <= 4 * sms else "pipeline"


def run(p, lo, hi):
    """Sequences lo .. hi - 1 of the batch by themselves."""
    from paper_2607_17979_b200 import api
    cu = p["cu_seqlens"].astype(np.int64)
    t0, t1, n, hv = int(cu[lo]), int(cu[hi]), hi - lo, p["Hv"]
    sub = {k: np.ascontiguousarray(p[k][t0:t1]) for k in ("q", "k", "v", "g", "beta")}
    final = torch.empty((n, hv, 128, 128), device="cuda")
    o = torch.empty((t1 - t0, hv, 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.full((api.gdn_prefill_workspace_bytes(t1 - t0, n, p["Hqk"], hv),), 0xff, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.gdn_prefill(U.dev_bf16(sub["q"]), U.dev_bf16(sub["k"]), U.dev_bf16(sub["v"]), U.dev(sub["g"]), U.dev(sub["beta"]),
                    U.dev((cu[lo:hi + 1] - t0).astype(np.int32)), U.dev(np.ascontiguousarray(p["init_state"][lo:hi])), final, None, o,
                    p["scale"], ws, route="stream", dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return o.cpu(), final.cpu()


@pytest.mark.parametrize("lens, hqk, hv", [
    ([64 * 741], 1, 1),                  # one head
    ([1, 0, 65, 3] * 8, 8, 24),          # 32 chunks of the 40 that T and N allow, empty sequences, no table launch
    ([5, 130, 0] * 11, 5, 20),           # 33 sequences: table launch
    ([0, 0, 3000, 0], 4, 16),
])
def test_pipeline_against_the_oracle(lens, hqk, hv):
    assert form(lens, hv) == "pipeline"
    p = I.prefill_inputs(lens, hqk, hv, seed=8300 + hv, alpha_lo=0.5, init="normal")
    o, S = run(p, 0, len(lens))
    o_ref, S_ref, _ = oracle_prefill(p)
    U.check_o(U.host_f64_from_bf16(o.cuda()), o_ref, U.O_REL_L2_PREFILL)
    U.check_state(S.numpy().astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("lens, hqk, hv, parts", [
    ([64 * 33 + t for t in (1, 15, 16, 17, 31, 32)], 1, 4, [(i, i + 1) for i in range(6)]),               # half units on either side
    ([64, 50, 33, 17, 16, 1, 48, 49, 63, 31, 32, 15], 40, 80, [(0, 4), (4, 8), (8, 12)]),                 # whole units
])
def test_either_form_gives_the_same_bits(lens, hqk, hv, parts):
    assert form(lens, hv) == "pipeline"
    p = I.prefill_inputs(lens, hqk, hv, seed=8400 + hv, alpha_lo=0.5, init="normal")
    o, S = run(p, 0, len(lens))
    cu = p["cu_seqlens"]
    for lo, hi in parts:
        assert form(lens[lo:hi], hv) == "few"
        o1, S1 = run(p, lo, hi)
        assert torch.equal(o1, o[cu[lo]:cu[hi]]) and torch.equal(S1, S[lo:hi])
