"""The calls a serving program makes of this library, as cases with seeded inputs.

A case is a dict of plain values.  `listed()` names twelve; `draw(rng)` gives another of the same
ranges.  `prepare` makes what the program holds before the call (inputs, state pool, workspace),
`run` makes the call through the binding and hands back everything it wrote, `work` counts the
bytes and operations the operator cannot do without, `tolerance` says how far two correct
implementations may lie apart.

  op "decode"    one new token for each of B sequences, state pool updated in place
  op "verify"    L new tokens for each of B sequences (draft verification), either tile orientation
  op "prefill"   packed variable-length prompts, outputs and final states

Options: `paged` = the pool has more slots than the batch has sequences and a slot table maps them;
`gate` = the call starts from the raw per-token projections, as a layer does, and goes through
gdn_gate first; `resume` = the prompts continue states already in the pool (read and written in
place through the slot table); `hint` = the program tells the length of the longest prompt.
"""
import math

import torch

from paper_2607_17979_b200 import api

D = 128
SCALE = D ** -0.5
# (q/k heads, v heads): the library's benchmark layer, and what one GPU holds of it when its heads
# are shared out over two and four GPUs
HEADS = ((16, 32), (8, 16), (4, 8))


def listed():
    return [
        # a single interactive stream: nothing but latency
        dict(name="decode_b1", op="decode", B=1, Hqk=4, Hv=8, slots=1, paged=False, gate=False),
        # a lightly loaded server, the layer's whole step from the raw projections on, odd batch
        dict(name="decode_step_b7", op="decode", B=7, Hqk=16, Hv=32, slots=16, paged=True, gate=True),
        # a busy server; the state pool is larger than L2
        dict(name="decode_b64", op="decode", B=64, Hqk=16, Hv=32, slots=64, paged=False, gate=False),
        # a full server on a paged 1 GiB pool: the largest decode
        dict(name="decode_b256_paged", op="decode", B=256, Hqk=16, Hv=32, slots=512, paged=True, gate=False),
        # draft verification: four tokens a sequence on a busy server
        dict(name="verify_b64_l4", op="verify", B=64, L=4, Hqk=16, Hv=32, slots=64, paged=False, layout="vk"),
        # draft verification with long drafts, odd sizes, a pool of transposed tiles
        dict(name="verify_b23_l7_kv", op="verify", B=23, L=7, Hqk=16, Hv=32, slots=48, paged=True, layout="kv"),
        # the shortest prompts
        dict(name="prefill_6", op="prefill", lens="6", Hqk=4, Hv=8, alpha_lo=0.9, gate=False, resume=False, hint=True),
        # one short chat turn, its length not passed on
        dict(name="prefill_100", op="prefill", lens="100", Hqk=16, Hv=32, alpha_lo=0.9, gate=False, resume=False, hint=False),
        # a scheduler's slice of 2048 tokens of three prompts that continue, from the raw projections on
        dict(name="prefill_resume_2048", op="prefill", lens="1337,512,199", Hqk=16, Hv=32, alpha_lo=0.9, gate=True, resume=True, hint=True),
        # an ordinary packed batch of unequal prompts
        dict(name="prefill_varlen_7680", op="prefill", lens="512,1024,2048,4096", Hqk=16, Hv=32, alpha_lo=0.9, gate=False, resume=False, hint=True),
        # many short prompts, every one with a ragged tail or two chunks exactly
        dict(name="prefill_57seqs_8192", op="prefill", lens="144x56,128", Hqk=16, Hv=32, alpha_lo=0.9, gate=False, resume=False, hint=True),
        # one long document: the largest prefill
        dict(name="prefill_long_32768", op="prefill", lens="32768", Hqk=16, Hv=32, alpha_lo=0.95, gate=False, resume=True, hint=True),
    ]


def draw(rng):
    def spread(lo, hi):         # evenly over the logarithm
        return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))

    Hqk, Hv = rng.choice(HEADS)
    op = rng.choice(("decode", "verify", "prefill", "prefill"))
    if op == "decode":
        B, paged = spread(1, 256), rng.random() < 0.5
        return dict(op=op, B=B, Hqk=Hqk, Hv=Hv, slots=B + rng.randint(1, B) if paged else B, paged=paged,
                    gate=rng.random() < 0.5)
    if op == "verify":
        B, paged = spread(1, 64), rng.random() < 0.5
        return dict(op=op, B=B, L=rng.randint(2, 16), Hqk=Hqk, Hv=Hv, slots=B + rng.randint(1, B) if paged else B,
                    paged=paged, layout=rng.choice(("vk", "vk", "kv")))
    T = spread(2, 32768)
    N = spread(1, min(64, T))
    share = [rng.expovariate(1.0) + 0.02 for _ in range(N)]
    lens = [max(1, int(T * s / sum(share))) for s in share]
    return dict(op=op, lens=",".join(map(str, lens)), Hqk=Hqk, Hv=Hv, alpha_lo=rng.choice((0.9, 0.95)),
                gate=rng.random() < 0.3, resume=rng.random() < 0.5, hint=rng.random() < 0.7)


def _lens(text):
    out = []
    for part in text.split(","):
        n, _, count = part.partition("x")
        out += [int(n)] * int(count or 1)
    return out


def prepare(case, seed):
    dev = "cuda"
    gen = torch.Generator(device=dev).manual_seed(seed)
    host = torch.Generator().manual_seed(seed)
    Hqk, Hv = case["Hqk"], case["Hv"]

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=dev)

    def unit(*shape):
        return torch.nn.functional.normalize(normal(*shape), dim=-1).to(torch.bfloat16)

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=gen, device=dev)

    def states(n):              # tiles of the recurrent cache
        return normal(n, Hv, D, D).mul_(0.02)

    if case["op"] == "prefill":
        lens = _lens(case["lens"])
        rows, entries = (sum(lens),), len(lens)
    else:
        rows, entries = ((case["B"], case["L"]) if case["op"] == "verify" else (case["B"],)), case["B"]

    s = dict(op=case["op"])
    s["q"], s["k"] = unit(*rows, Hqk, D), unit(*rows, Hqk, D)
    s["v"] = normal(*rows, Hv, D).to(torch.bfloat16)
    s["o"] = torch.empty((*rows, Hv, D), dtype=torch.bfloat16, device=dev)
    if case.get("gate"):
        # raw projections and the layer's two vectors, initialised as such layers are: decay rates
        # U[1, 16), step sizes log-uniform in [0.001, 0.1)
        s["a"], s["b"] = normal(*rows, Hv).to(torch.bfloat16), normal(*rows, Hv).to(torch.bfloat16)
        s["A_log"] = uniform(1.0, 16.0, Hv).log()
        dt = uniform(math.log(1e-3), math.log(1e-1), Hv).exp()
        s["dt_bias"] = dt + torch.log(-torch.expm1(-dt))
        s["g"], s["beta"] = torch.empty((*rows, Hv), device=dev), torch.empty((*rows, Hv), device=dev)
    else:
        s["g"] = uniform(case.get("alpha_lo", 0.9), 1.0, *rows, Hv).clamp_(max=1.0).log()
        s["beta"] = torch.sigmoid(normal(*rows, Hv))

    if case["op"] == "prefill":
        cu = [0]
        for n in lens:
            cu.append(cu[-1] + n)
        s["cu"] = torch.tensor(cu, dtype=torch.int32, device=dev)
        slots = entries + 1 if case["resume"] else entries
        s["final"] = states(slots) if case["resume"] else torch.empty((slots, Hv, D, D), device=dev)
        s["init"] = s["final"] if case["resume"] else None
        s["slot_idx"] = torch.randperm(slots, generator=host)[:entries].to(torch.int32).to(dev) if case["resume"] else None
        s["ws"] = torch.empty(api.gdn_prefill_workspace_bytes(cu[-1], entries, Hqk, Hv), dtype=torch.uint8, device=dev)
        s["hint"] = max(lens) if case["hint"] else 0
        return s
    s["pool"] = states(case["slots"])
    s["slot_idx"] = torch.randperm(case["slots"], generator=host)[:entries].to(torch.int32).to(dev) if case["paged"] else None
    s["layout"] = api.STATE_KV if case.get("layout") == "kv" else api.STATE_VK
    return s


def run(s):
    if "a" in s:
        api.gdn_gate(s["a"], s["b"], s["A_log"], s["dt_bias"], s["g"], s["beta"])
    if s["op"] == "prefill":
        api.gdn_prefill(s["q"], s["k"], s["v"], s["g"], s["beta"], s["cu"], s["init"], s["final"], s["slot_idx"], s["o"],
                        SCALE, s["ws"], max_seqlen_hint=s["hint"])
        return {"o": s["o"], "state": s["final"]}
    if s["op"] == "verify":
        api.gdn_decode_multi(s["q"], s["k"], s["v"], s["g"], s["beta"], s["pool"], s["slot_idx"], s["o"], SCALE, s["layout"])
    else:
        api.gdn_decode(s["q"], s["k"], s["v"], s["g"], s["beta"], s["pool"], s["slot_idx"], s["o"], SCALE)
    return {"o": s["o"], "state": s["pool"]}


def work(case):
    """q, k, v, gates read once, o written once, every touched state tile read (unless it starts at
    zero) and written once; per token and v-head the recurrence's two matrix-vector products, decay
    and rank-one update over a 128 x 128 tile."""
    Hqk, Hv = case["Hqk"], case["Hv"]
    if case["op"] == "prefill":
        lens = _lens(case["lens"])
        rows, entries, passes = sum(lens), len(lens), 2 if case["resume"] else 1
    else:
        rows, entries, passes = case["B"] * case.get("L", 1), case["B"], 2
    gates = 12 if case.get("gate") else 8     # a, b in and g, beta out, or g, beta in
    return {"bytes": rows * (2 * Hqk * D * 2 + 2 * Hv * D * 2 + gates * Hv) + entries * passes * Hv * D * D * 4,
            "flops": rows * Hv * 8 * D * D}


def tolerance(case):
    # decode: fp32 throughout, o rounded to bf16 (a differing last bit of some values).  prefill: bf16
    # operands with fp32 accumulation; o carries 3e-3 of operand and output rounding on either side
    return {"rel": 2e-3} if case["op"] != "prefill" else {"rel": 1e-2}
