"""The decay between two tokens of a chunk is ONE exponential, 2^(b_r - b_i) of the gates' prefix sums, wherever the pair lies.

With orthogonal keys, beta = v = 1 and a zero state nothing else is left of an output: every query asks for one earlier token's key,
so o is that pair's decay, rounded to bf16 once.  The prefix sums are exact (gates are multiples of 2^-10), and the exponential is
the one torch's exp2 takes on the device, so the values are equal, not close: a decay put together from two exponentials is off by
a last bit of fp32, and of half a million values some round the other way."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunks, heads", [(16, 4), (512, 32)])      # few items; the pipeline, 524288 pairs below the diagonal blocks
def test_outputs_are_the_rounded_decay(chunks, heads):
    from paper_2607_17979_b200 import api
    T, N = 64 * chunks, chunks
    gen = torch.Generator().manual_seed(chunks)
    token = torch.arange(T) % 64
    asked = torch.where(token < 32, token, torch.randint(0, 32, (T,), generator=gen))       # of the same chunk; its own key below 32
    eye = torch.eye(128, dtype=torch.bfloat16)
    q, k = eye[asked][:, None].cuda(), eye[token][:, None].cuda()
    v = torch.ones(T, heads, 128, dtype=torch.bfloat16, device="cuda")
    g = (-torch.randint(1, 103, (T, heads), generator=gen) / 1024.0).cuda()
    beta = torch.ones(T, heads, device="cuda")
    cu = torch.arange(0, T + 1, 64, dtype=torch.int32, device="cuda")
    final = torch.empty(N, heads, 128, 128, device="cuda")
    o = torch.empty_like(v)
    ws = torch.empty(api.gdn_prefill_workspace_bytes(T, N, 1, heads), dtype=torch.uint8, device="cuda")
    api.gdn_prefill(q.contiguous(), k.contiguous(), v, g, beta, cu, None, final, None, o, 1.0, ws, route="stream")
    torch.cuda.synchronize()
    b2 = g.view(N, 64, heads).double().cumsum(1).float() * torch.tensor(math.log2(math.e), dtype=torch.float32, device="cuda")
    of = b2.gather(1, asked.view(N, 64, 1).expand(-1, -1, heads).cuda())
    want = torch.exp2(b2 - of).to(torch.bfloat16).view(T, heads, 1).expand_as(o)
    assert torch.equal(o, want), int((o != want)[..., 0].sum())
