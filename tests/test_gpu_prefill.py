"""GPU parity: gdn_prefill (chunked) and gdn_prefill_recurrent against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_17979_b200 import inputs as I
import gpu_util as U

pytestmark = pytest.mark.gpu

IMPLS = ["chunked", "fused", "stream", "recurrent"]


def run_prefill(p, impl, slot_idx=None, num_slots=None, init="from_inputs", alias=False,
                pool_fill=None, split_permille=-1):
    """Returns (o fp64 [T,Hv,128], final fp32 numpy [num_slots,Hv,128,128], status)."""
    from paper_2607_17979_b200 import api
    N, Hv, T = p["N"], p["Hv"], p["T"]
    num_slots = N if num_slots is None else num_slots
    init_np = p["init_state"] if isinstance(init, str) else init
    init_t = U.dev(init_np)
    if alias:
        assert init_t is not None
        final = init_t
    else:
        final = torch.full((num_slots, Hv, 128, 128), float("nan") if pool_fill is None else pool_fill,
                           dtype=torch.float32, device="cuda")
    o = torch.full((T, Hv, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    args = (U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), U.dev_bf16(p["v"]), U.dev(p["g"]),
            U.dev(p["beta"]), U.dev(p["cu_seqlens"]), init_t, final, U.dev(slot_idx), o, p["scale"])
    if impl in ("chunked", "fused", "stream", "overlap", "auto"):
        ws = torch.empty(max(api.gdn_prefill_workspace_bytes(T, N, p["Hqk"], Hv), 256),
                         dtype=torch.uint8, device="cuda")
        api.gdn_prefill(*args, ws, dev_status=status, route=impl, split_permille=split_permille)
    else:
        api.gdn_prefill_recurrent(*args, dev_status=status)
    torch.cuda.synchronize()
    return U.host_f64_from_bf16(o), final.cpu().numpy(), int(status.item())


def oracle_prefill(p, slot_idx=None, num_slots=None, init="from_inputs"):
    init_np = p["init_state"] if isinstance(init, str) else init
    init64 = None if init_np is None else init_np.astype(np.float64)
    o, S, bad = oracle.prefill(p["q"], p["k"], p["v"], p["g"], p["beta"], p["cu_seqlens"], init64,
                               slot_idx, p["scale"], num_slots=num_slots)
    return o, S, bad


def compare(p, impl, o_rel_bound=U.O_REL_L2_PREFILL, **kw):
    o, S, status = run_prefill(p, impl, **kw)
    okw = {k: v for k, v in kw.items() if k in ("slot_idx", "num_slots", "init")}
    o_ref, S_ref, _ = oracle_prefill(p, **okw)
    assert status == 0
    if p["T"] > 0:
        U.check_o(o, o_ref, o_rel_bound)
    return o, S, o_ref, S_ref


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("L", [1, 2, 63, 64, 65, 127, 128, 129, 200])
def test_single_sequence_lengths(impl, L):
    for seed, init in [(0, "zero"), (1, "normal"), (2, "normal")]:
        p = I.prefill_inputs([L], 1, 2, seed=300 + seed, init=init)
        o, S, o_ref, S_ref = compare(p, impl)
        U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("Hqk,Hv", [(1, 1), (1, 2), (2, 4), (4, 8), (16, 32)])
def test_packed_ragged_batch_with_empty_sequence(impl, Hqk, Hv):
    lens = [1, 2, 63, 64, 0, 65, 127, 128, 129, 200]
    if Hv == 32:
        lens = [65, 0, 130]
    p = I.prefill_inputs(lens, Hqk, Hv, seed=400 + Hv, init="normal")
    o, S, o_ref, S_ref = compare(p, impl)
    U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
    empty = lens.index(0)
    assert np.array_equal(S[empty], p["init_state"][empty])        # passes through bit-exactly


@pytest.mark.parametrize("impl", IMPLS)
def test_slots_padding_alias_and_untouched_slots(impl):
    lens = [70, 5, 64, 33]
    p = I.prefill_inputs(lens, 2, 4, seed=500, init="zero")
    rs = np.random.default_rng(5)
    pool = (rs.standard_normal((7, 4, 128, 128)) * 0.02).astype(np.float32)
    idx = np.array([6, -1, 2, 9], np.int32)                         # padding, out of range
    o, S, status = run_prefill(p, impl, slot_idx=idx, num_slots=7, init=pool, alias=True)
    o_ref, S_ref, bad = oracle_prefill(p, slot_idx=idx, num_slots=7, init=pool)
    assert status == 1 and bad == 4
    cu = p["cu_seqlens"]
    assert np.abs(o[cu[1]:cu[2]]).max() == 0 and np.abs(o[cu[3]:cu[4]]).max() == 0
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    assert np.array_equal(S[[0, 1, 3, 4, 5]], pool[[0, 1, 3, 4, 5]])
    U.check_state(S[[6, 2]].astype(np.float64), S_ref[[6, 2]], U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("case", ["beta0", "beta1", "g0", "alpha09", "v0", "same_keys"])
def test_degenerate_values(impl, case):
    p = I.prefill_inputs([150, 64], 2, 4, seed=600, init="normal")
    if case == "beta0":
        p["beta"][:] = 0
    elif case == "beta1":
        p["beta"][:] = 1
    elif case == "g0":
        p["g"][:] = 0
    elif case == "alpha09":
        p["g"][:] = np.float32(np.log(0.9))
    elif case == "v0":
        p["v"][:] = 0
    elif case == "same_keys":                # worst case for the triangular solve
        p["k"][:] = p["k"][:1, :1]
        p["beta"][:] = 1
    # With every key identical the two terms of O = e^b Q S0^T + P U cancel almost completely, so
    # the bf16 rounding of the operands P and U (2^-9 each) is amplified in o's RELATIVE error;
    # the stated absolute gate (2e-2) still holds with a 20x margin.  Only this case is relaxed.
    bound = 2e-2 if (case == "same_keys" and impl != "recurrent") else U.O_REL_L2_PREFILL
    o, S, o_ref, S_ref = compare(p, impl, o_rel_bound=bound)
    U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("impl", IMPLS)
def test_bad_cu_seqlens_sets_status_and_skips(impl):
    p = I.prefill_inputs([40, 30], 1, 2, seed=700, init="zero")
    p["cu_seqlens"] = np.array([0, 50, 45], np.int32)               # decreasing, and cu[N] != T
    o, S, status = run_prefill(p, impl, pool_fill=7.0)
    assert status & 2


@pytest.mark.parametrize("impl", IMPLS)
def test_deterministic_and_split_prefill_hand_off(impl):
    p = I.prefill_inputs([192], 2, 4, seed=800, init="normal")
    o1, S1, _ = run_prefill(p, impl)
    o2, S2, _ = run_prefill(p, impl)
    assert np.array_equal(o1, o2) and np.array_equal(S1, S2)
    # prefill(128) then prefill(64 from its final state) tracks prefill(192)
    a = {n: (x[:128] if isinstance(x, np.ndarray) and x.shape[:1] == (192,) else x) for n, x in p.items()}
    b = {n: (x[128:] if isinstance(x, np.ndarray) and x.shape[:1] == (192,) else x) for n, x in p.items()}
    a.update(T=128, cu_seqlens=np.array([0, 128], np.int32))
    b.update(T=64, cu_seqlens=np.array([0, 64], np.int32))
    oa, Sa, _ = run_prefill(a, impl)
    ob, Sb, _ = run_prefill(b, impl, init=Sa)
    o_ref, S_ref, _ = oracle_prefill(p)
    U.check_o(np.concatenate([oa, ob]), o_ref, U.O_REL_L2_PREFILL)
    U.check_state(Sb.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)


def test_chunked_and_recurrent_routes_agree():
    p = I.prefill_inputs([300, 17, 128], 2, 4, seed=900, init="normal")
    oc, Sc, _ = run_prefill(p, "chunked")
    orr, Sr, _ = run_prefill(p, "recurrent")
    assert np.abs(oc - orr).max() <= U.O_MAX_ABS
    assert U.rel_l2(Sc.astype(np.float64), Sr.astype(np.float64)) <= U.STATE_REL_L2_PREFILL


@pytest.mark.parametrize("trial", [0, 1, 2, 3, 4])
def test_prefill_varlen_benchmark_config_full(trial):
    """4 sequences {512,1024,2048,4096}, 32 v-heads, five seeds: every output against the oracle,
    through the length-routed entry point (the call the benchmark times) and, on the first seed,
    through the three launches under both names and the single cooperative launch."""
    p = I.make_config(3, trial)
    o_ref, S_ref, _ = oracle_prefill(p)
    cu = p["cu_seqlens"]
    for impl in (("auto", "chunked", "stream", "fused") if trial == 0 else ("auto",)):
        o, S, status = run_prefill(p, impl)
        assert status == 0
        U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
        U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
        for n in range(4):                                           # no sequence hides in the norm
            U.check_o(o[cu[n]:cu[n + 1]], o_ref[cu[n]:cu[n + 1]], U.O_REL_L2_PREFILL)


def check_long_context(p, o_ref, S_ref, impl, **kw):
    """One 32768-token sequence at full size: every v-head on its own (outputs of the whole
    sequence, outputs of the last 4096 tokens -- the far end of the carry -- and the final state)."""
    o, S, status = run_prefill(p, impl, **kw)
    assert status == 0 and np.isfinite(o).all() and np.isfinite(S).all()
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
    for hv in range(p["Hv"]):
        U.check_o(o[:, hv], o_ref[:, hv], U.O_REL_L2_PREFILL)
        U.check_o(o[-4096:, hv], o_ref[-4096:, hv], U.O_REL_L2_PREFILL)
        U.check_state(S[:, hv].astype(np.float64), S_ref[:, hv], U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("trial", [0, 1, 2, 3, 4])
def test_prefill_long_context_benchmark_config_all_heads(trial):
    """The oracle runs the whole 32768-token, 32-head batch; the GPU result is compared head by
    head through the routed entry point (the two-part production for this shape) on five seeds
    and, on the first seed, through the three launches under both names."""
    p = I.make_config(4, trial)
    o_ref, S_ref, _ = oracle_prefill(p)
    for impl in (("auto", "chunked", "stream") if trial == 0 else ("auto",)):
        check_long_context(p, o_ref, S_ref, impl)


@pytest.mark.parametrize("impl", ["auto", "chunked", "stream", "fused"])
def test_batches_that_are_all_padding_or_all_empty(impl):
    """No valid work at all: every slot negative (rows zeroed, no state touched), and every
    sequence but one empty (states pass through bit-exactly)."""
    p = I.prefill_inputs([70, 5, 130], 2, 4, seed=31, init="normal")
    slots = np.array([-1, -5, -2], np.int32)
    o, S, status = run_prefill(p, impl, slot_idx=slots, pool_fill=3.0)
    assert status == 0
    assert np.array_equal(o, np.zeros_like(o)) and np.array_equal(S, np.full_like(S, 3.0))
    q = I.prefill_inputs([0, 0, 90, 0], 2, 4, seed=32, init="normal")
    o, S, o_ref, S_ref = compare(q, impl)
    assert np.array_equal(S[[0, 1, 3]], q["init_state"][[0, 1, 3]])
    U.check_state(S[2:3].astype(np.float64), S_ref[2:3], U.STATE_REL_L2_PREFILL)


def test_thousands_of_tiny_sequences():
    """2000 sequences of 1-40 tokens, 4 v-heads (8000 units): the length-routed entry point and
    the persistent state pass against the oracle."""
    rng = np.random.default_rng(11)
    lens = [int(x) for x in rng.integers(1, 41, size=2000)]
    p = I.prefill_inputs(lens, 2, 4, seed=33, init="normal")
    o_ref, S_ref, _ = oracle_prefill(p)
    for impl in ("auto", "stream"):
        o, S, status = run_prefill(p, impl)
        assert status == 0
        U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
        U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("impl", ["chunked", "stream", "fused"])
def test_chunked_repeatable_under_load_many_ctas(impl):
    """Several back-to-back runs of a batch that fills the GPU (64 sequence-heads, ragged tails,
    last chunks of every length class) must be bit-identical: a missed barrier between the
    kernel's warp roles shows up as run-to-run differences long before it shows up as a large
    error."""
    lens = [448, 449, 511, 512, 513, 1000, 77, 1536]
    p = I.prefill_inputs(lens, 4, 8, seed=1234, init="normal")
    ref_o, ref_S, st = run_prefill(p, impl)
    assert st == 0
    for _ in range(4):
        o, S, st = run_prefill(p, impl)
        assert st == 0 and np.array_equal(o, ref_o) and np.array_equal(S, ref_S)
    o_ref, S_ref, _ = oracle_prefill(p)
    U.check_o(ref_o, o_ref, U.O_REL_L2_PREFILL)
    U.check_state(ref_S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("impl", ["stream", "auto"])
def test_many_short_sequences_stream_across_unit_boundaries(impl):
    """Far more (sequence, v-head) units than SMs, of mixed lengths (one to five chunks, ragged
    tails, empty sequences, a padding slot): every CTA of the persistent state pass walks a
    dozen units with its pipeline running across their boundaries.  Repeated runs must be
    bit-identical and every sequence must match the oracle."""
    rng = np.random.default_rng(77)
    lens = [int(x) for x in rng.integers(1, 330, size=200)]
    lens[5] = 0; lens[77] = 0; lens[120] = 64; lens[121] = 128; lens[199] = 1
    p = I.prefill_inputs(lens, 2, 8, seed=4321, init="normal")
    slots = np.arange(200, dtype=np.int32)
    slots[33] = -1
    o, S, st = run_prefill(p, impl, slot_idx=slots)
    assert st == 0
    o2, S2, _ = run_prefill(p, impl, slot_idx=slots)
    keep = slots >= 0                       # the padding slot's tile is never written
    assert np.array_equal(o, o2) and np.array_equal(S[keep], S2[keep])
    o_ref, S_ref, _ = oracle_prefill(p, slot_idx=slots)
    cu = p["cu_seqlens"]
    assert np.array_equal(o[cu[33]:cu[34]], np.zeros_like(o[cu[33]:cu[34]]))
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    for n in (0, 5, 6, 77, 120, 121, 150, 199):
        if cu[n + 1] > cu[n]:
            U.check_o(o[cu[n]:cu[n + 1]], o_ref[cu[n]:cu[n + 1]], 2 * U.O_REL_L2_PREFILL)
    U.check_state(S[keep].astype(np.float64), S_ref[keep], U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("lens", [[1], [6], [16], [3, 16, 0, 9], [17], [12, 35]])
def test_length_routed_entry_point_small_shapes(lens):
    """gdn_prefill itself (routing by length: up to 16 tokens per sequence the token-by-token
    kernel, beyond that the chunked kernels) on the tiny shapes of the short-prompt regime."""
    p = I.prefill_inputs(lens, 2, 4, seed=5000 + sum(lens), init="normal")
    o, S, o_ref, S_ref = compare(p, "auto")
    U.check_state(S.astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)


@pytest.mark.parametrize("impl", ["auto", "chunked", "stream"])
@pytest.mark.parametrize("N", [16, 17, 32, 33])
def test_small_batches_without_a_table_launch_and_the_first_batch_beyond(impl, N):
    """Up to 32 sequences the intra-chunk kernel finds its chunk and the state pass its units from
    cu_seqlens, and no table is written; 33 sequences take the table-building launch.  Equal chunk
    counts (ties in the ranking), an empty sequence, a padding slot, out-of-order bounds and an
    initial state must come out the same on both sides of that boundary."""
    lens = [70, 130, 64, 0, 200, 65, 1, 128, 129, 64, 70, 33, 192, 5, 100, 66, 90,
            64, 0, 1, 130, 65, 70, 128, 3, 64, 129, 0, 66, 200, 63, 127, 65][:N]
    p = I.prefill_inputs(lens, 2, 4, seed=900 + N, init="normal")
    slots = np.arange(N, dtype=np.int32)
    slots[2] = -1
    slots[-1] = -1 if N >= 32 else slots[-1]
    o, S, st = run_prefill(p, impl, slot_idx=slots)
    assert st == 0
    o_ref, S_ref, _ = oracle_prefill(p, slot_idx=slots)
    keep = slots >= 0
    U.check_o(o, o_ref, U.O_REL_L2_PREFILL)
    U.check_state(S[keep].astype(np.float64), S_ref[keep], U.STATE_REL_L2_PREFILL)
    # a batch with out-of-order bounds: flagged, the bad sequence skipped, the others right
    q = dict(p)
    cu = p["cu_seqlens"].copy()
    cu[5] = cu[4] - 3
    q["cu_seqlens"] = cu
    o_bad, S_bad, st_bad = run_prefill(q, impl, slot_idx=slots, pool_fill=7.0)
    assert st_bad == 2
    # sequence 4 runs backwards, 5 starts before 2 and 3 end: skipped; those in front and behind are as before
    ok = [n for n in range(N) if n not in (4, 5) and slots[n] >= 0]
    assert (S_bad[[4, 5]] == 7.0).all()
    assert np.array_equal(S_bad[ok], S[ok])
    for n in ok:
        if lens[n]:
            assert np.array_equal(o_bad[p["cu_seqlens"][n]:p["cu_seqlens"][n + 1]], o[p["cu_seqlens"][n]:p["cu_seqlens"][n + 1]])

