"""The intra-chunk pipeline when a wait runs out: prod_wait's own source on the host, 32 threads as a warp's lanes (its three
instructions replaced by their meaning), and what the CTA still waits for before its shared memory and TMEM go away."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")

HARNESS = r"""
#include <atomic>
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
#define __device__
#define __noinline__
constexpr uint32_t kSpinLimit = 300;
thread_local int lane;
unsigned completed;                        // bit i: lane i's polls see the barrier's phase completed
std::atomic<uint32_t> flag;
std::atomic<unsigned> polls;
bool votes[32];
std::barrier<> warp(32);
bool __all_sync(unsigned, bool mine) {
    votes[lane] = mine;
    warp.arrive_and_wait();
    bool all = true;
    for (bool v : votes) all = all && v;
    warp.arrive_and_wait();
    return all;
}
bool __any_sync(unsigned mask, bool mine) { return !__all_sync(mask, !mine); }
bool poll() { if (lane == 0) ++polls; return completed >> lane & 1u; }
%s
int main(int argc, char** argv) {
    completed = static_cast<unsigned>(std::strtoul(argv[1], nullptr, 16));
    flag = std::atoi(argv[2]);
    unsigned first = 0;
    std::vector<std::thread> lanes;
    for (int i = 0; i < 32; ++i)
        lanes.emplace_back([&, i] {
            lane = i;
            prod_wait(0, 0, 0);
            warp.arrive_and_wait();
            if (i == 0) first = polls.exchange(0);
            warp.arrive_and_wait();
            prod_wait(0, 0, 0);
        });
    for (auto& t : lanes) t.join();
    std::printf("%%u %%u %%u\n", first, polls.load(), flag.load());
}
"""


def source():
    return open(os.path.join(CSRC, "gdn_prefill_intra.cuh")).read()


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    s = source()
    at = s.index("static __device__ __noinline__ void prod_wait(")
    f = s[at:s.index("\n}\n", at) + 3]
    meaning = {"try_wait": "ok = __all_sync(0xffffffffu, poll());", "ld.volatile": "f = flag;", "st.volatile": "flag = 1;"}
    for block in re.findall(r"asm volatile\(.*?\);\n", f, re.S):
        (name,) = [k for k in meaning if k in block]
        f = f.replace(block, meaning.pop(name) + "\n")
    assert not meaning
    d = tmp_path_factory.mktemp("prod_wait")
    (d / "w.cpp").write_text(HARNESS % f)
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-pthread", str(d / "w.cpp"), "-o", str(d / "w")])
    return str(d / "w")


@pytest.mark.parametrize("completed, flag, want", [
    (0xffffffff, 0, (1, 1, 0)),            # through at the first poll
    (0, 0, (300, 1, 1)),                   # runs out after kSpinLimit polls; the next finds the flag
    (0x0000ffff, 0, (300, 1, 1)),          # lanes that see it differently: no lane is through alone
    (0, 1, (1, 1, 1)),                     # another warp has given up
    (0xffffffff, 1, (1, 1, 1)),
])
def test_a_wait_ends_together_and_in_bounded_time(harness, completed, flag, want):
    out = subprocess.check_output([harness, f"{completed:x}", str(flag)], timeout=60).split()
    assert tuple(map(int, out)) == want


def test_copies_and_products_in_flight_are_waited_for():
    """Every barrier that copies land on, and every warp that issues products, in front of the CTA's last barrier."""
    s = source()
    role, end = s[s.index("void produce_role("):].split("    if (abort_flag != 0) {", 1)
    end = end[:end.index("// A kernel's body")]
    armed = set(re.findall(r"mbar_expect_tx\(bar, \d+\)", role))
    assert len(armed) == 2 and set(re.findall(r"uint64_t\* bar = &bars\[(kB\w+) \+ s\.at\]", role)) == {"kBQk", "kBV"}
    assert set(re.findall(r"mbar_wait\(&bars\[(kB\w+) \+ \(", end)) == {"kBQk", "kBV", "kBDrain"}
    issuers = [x for x in role.split("} else if (") if "mma_commit(" in x]
    warps = {re.match(r"warp == (k\w+)\)", x).group(1) for x in issuers}
    assert warps == {"kPGramWarp", "kPMmaWarp"} and all(f"warp == {w}" in end for w in warps)
    assert "mma_commit(&bars[kBDrain" in end and "mbar_wait(&bars[kBDrain" in end
    for x in re.split(r"// =====================", role)[1:]:          # bulk copies out: read before the role goes on
        if "bulk_store(" in x:
            assert "bulk_wait_read" in x
