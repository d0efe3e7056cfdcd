"""Which sequences count when cu_seqlens is out of order: those that do are disjoint, so their chunks fit the workspace that
T and N give.  The rule's own source run on the host, against its definition, in the form for a warp and the one for a
block; and on the GPU batches with overlapping sequences, with marked memory behind the workspace."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")
BLOCK = 8      # threads of the emulated block: a batch takes several tiles

HARNESS = r"""
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
thread_local std::barrier<>* group;
int width;
int32_t words[32];
template <class F> auto exchange(int lane, int32_t mine, F f) {
    words[lane] = mine;
    group->arrive_and_wait();
    auto r = f();
    group->arrive_and_wait();
    return r;
}
thread_local int self;
bool all(bool mine) {
    return exchange(self, mine, [] { bool a = true; for (int i = 0; i < width; ++i) a = a && words[i]; return a; });
}
bool __all_sync(unsigned, bool mine) { return all(mine); }
bool __syncthreads_and(bool mine) { return all(mine); }
int32_t __shfl_sync(unsigned, int32_t mine, int from) { return exchange(self, mine, [&] { return words[from]; }); }
%s
int main() {
    std::vector<std::vector<int32_t>> cases;      // T, N, cu[0 .. N]
    for (int T, N; std::scanf("%%d %%d", &T, &N) == 2;) {
        cases.push_back({T, N});
        for (int i = 0; i <= N; ++i) {
            int x;
            if (std::scanf("%%d", &x) != 1) return 1;
            cases.back().push_back(x);
        }
    }
    for (int form = 0; form < 2; ++form) {
        width = form == 0 ? 32 : %d;
        std::barrier<> b(width);
        std::vector<std::vector<char>> ok(cases.size());
        for (size_t i = 0; i < cases.size(); ++i) ok[i].assign(cases[i][1], 0);
        int32_t ends[32], end_before = 0;
        std::vector<std::thread> lanes;
        for (int lane = 0; lane < width; ++lane)
            lanes.emplace_back([&, lane] {
                group = &b;
                self = lane;
                for (size_t i = 0; i < cases.size(); ++i) {
                    const int32_t T = cases[i][0], N = cases[i][1], *cu = cases[i].data() + 2;
                    if (form == 0) {
                        const bool r = warp_bounds_ok(lane < N ? cu[lane] : 0, lane < N ? cu[lane + 1] : 0, T, lane);
                        if (lane < N) ok[i][lane] = r;
                        continue;
                    }
                    if (lane == 0) end_before = 0;
                    b.arrive_and_wait();
                    for (int base = 0; base < N; base += width) {
                        const int n = base + lane;
                        const bool r = block_bounds_ok(n < N, n < N ? cu[n] : 0, n < N ? cu[n + 1] : 0, T, end_before, ends, lane);
                        if (n < N) ok[i][n] = r;
                        b.arrive_and_wait();
                        if (lane == 0)
                            for (int m = 0; m < width; ++m) end_before = ends[m] > end_before ? ends[m] : end_before;
                        b.arrive_and_wait();
                    }
                }
            });
        for (auto& t : lanes) t.join();
        for (auto& v : ok) {
            for (char c : v) std::putchar('0' + c);
            std::putchar('\n');
        }
    }
}
"""


def valid(cu, T):
    """The definition: own bounds in order and in range, and no earlier sequence of that kind ends behind the start."""
    out, end = [], 0
    for t0, t1 in zip(cu, cu[1:]):
        in_order = 0 <= t0 <= t1 <= T
        out.append(in_order and t0 >= end)
        if in_order:
            end = max(end, t1)
    return out


def test_rule(tmp_path):
    s = open(os.path.join(CSRC, "gdn_prefill_chunk.cuh")).read()
    text = s[s.index("__device__ __forceinline__ bool bounds_in_order("):s.index("// Workspace layout (all offsets")]
    (tmp_path / "b.cpp").write_text(HARNESS % (text, BLOCK))
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-pthread", str(tmp_path / "b.cpp"), "-o", str(tmp_path / "b")])
    rng = np.random.default_rng(3)
    cases = [(640, [0, 640, 0, 640]), (100, [0, 10, 1000, 20, 30]), (64, [-5, 64]), (64, [0, -1, 64]), (64, [0, 65]), (0, [0, 0]),
             (2**31 - 1, [0, 2**31 - 1, -2**31, 2**31 - 1])]
    for trial in range(120):
        n, T = int(rng.integers(1, 33)), int(rng.integers(1, 700))
        cu = np.sort(rng.integers(0, T + 1, n + 1))
        if trial % 4:                       # out of order in a few places, or altogether
            at = rng.integers(0, n + 1, trial % 4 if trial % 3 else n + 1)
            cu[at] = rng.integers(-20, T + 40, len(at))
        else:
            cu[0], cu[-1] = 0, T
        cases.append((T, cu.tolist()))
    text = "".join(f"{T} {len(cu) - 1} {' '.join(map(str, cu))}\n" for T, cu in cases)
    out = subprocess.run([str(tmp_path / "b")], input=text, text=True, capture_output=True, check=True, timeout=120).stdout.split()
    want = ["".join("01"[v] for v in valid(cu, T)) for T, cu in cases]
    assert out == want + want
    for T, cu in cases:
        chunks = sum(-(-(t1 - t0) // 64) for ok, t0, t1 in zip(valid(cu, T), cu, cu[1:]) if ok)
        assert chunks <= T // 64 + len(cu) - 1
    # without the comparison the first case has more chunks than the workspace, 20 against 13
    T, cu = cases[0]
    assert sum(-(-(t1 - t0) // 64) for t0, t1 in zip(cu, cu[1:]) if 0 <= t0 <= t1 <= T) > T // 64 + 3


@pytest.mark.gpu
@pytest.mark.parametrize("route", ["stream", "chunked", "fused", "overlap"])
@pytest.mark.parametrize("cu, hv", [
    ([0, 640, 0, 640], 32),                                     # items in a row, a warp finds the bounds
    ([0, 200, 100, 200], 2),                                    # items as a grid
    ([0, 130, 70, 300, 250, 640, 640], 4),
    ([0, 100, 90] + [100 + 10 * i for i in range(1, 30)] + [380, 400], 4),      # 33 sequences: the small table kernel
    ([0, 640] * 20 + [640], 8),
    ([0, 64, 50] + list(range(64, 400)) + [100, 640], 1),       # more than a block's: the general one, several tiles
])
def test_overlapping_sequences_are_skipped_and_nothing_is_written_behind_the_workspace(cu, hv, route):
    import torch

    import gpu_util as U
    import oracle
    from paper_2607_17979_b200 import api
    from paper_2607_17979_b200 import inputs as I
    T, N, hqk = max(cu), len(cu) - 1, max(hv // 2, 1)
    p = I.prefill_inputs([T], hqk, hv, seed=61 + N, alpha_lo=0.5, init="zero")
    size = api.gdn_prefill_workspace_bytes(T, N, hqk, hv)
    ws = torch.full((size + (64 << 20),), 0xa5, dtype=torch.uint8, device="cuda")
    final = torch.full((N, hv, 128, 128), 7.0, device="cuda")
    o = torch.full((T, hv, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.gdn_prefill(U.dev_bf16(p["q"]), U.dev_bf16(p["k"]), U.dev_bf16(p["v"]), U.dev(p["g"]), U.dev(p["beta"]),
                    U.dev(np.array(cu, np.int32)), None, final, None, o, p["scale"], ws[:size], max_seqlen_hint=T,
                    dev_status=status, route=route)
    torch.cuda.synchronize()
    assert int(status.item()) == 2
    assert bool((ws[size:] == 0xa5).all())
    rows, S = U.host_f64_from_bf16(o), final.cpu().numpy()
    touched = np.zeros(T, bool)
    for n, ok in enumerate(valid(cu, T)):
        t0, t1 = cu[n], cu[n + 1]
        if not ok:
            assert (S[n] == 7.0).all()
        elif t0 == t1:
            assert (S[n] == 0.0).all()
        else:
            touched[t0:t1] = True
            part = {k: p[k][t0:t1] for k in ("q", "k", "v", "g", "beta")}
            o_ref, S_ref, _ = oracle.prefill(part["q"], part["k"], part["v"], part["g"], part["beta"],
                                             np.array([0, t1 - t0], np.int32), None, None, p["scale"], num_slots=1)
            U.check_o(rows[t0:t1], o_ref, 2 * U.O_REL_L2_PREFILL if t1 - t0 < 16 else U.O_REL_L2_PREFILL)
            U.check_state(S[n:n + 1].astype(np.float64), S_ref, U.STATE_REL_L2_PREFILL)
    assert np.isnan(rows[~touched]).all()
