"""The verdict of a warp's bounded wait is the same on every lane, also when its lanes' polls end differently
(what follows are warp-wide instructions).  The functions' own source, run by 32 host threads as lanes."""
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
#define __forceinline__ inline
constexpr uint32_t kSpinLimit = 600;
thread_local int lane;
unsigned completed;                        // bit i: lane i's polls see the barrier's phase completed
bool votes[32];
std::barrier<> warp(32);
void __nanosleep(int) {}
void __syncwarp(unsigned = 0xffffffffu) { warp.arrive_and_wait(); }
bool __all_sync(unsigned, bool mine) {
    votes[lane] = mine;
    warp.arrive_and_wait();
    bool all = true;
    for (bool v : votes) all = all && v;
    warp.arrive_and_wait();
    return all;
}
bool __any_sync(unsigned mask, bool mine) { return !__all_sync(mask, !mine); }
bool mbar_try_wait(uint64_t*, uint32_t) { return completed >> lane & 1u; }
%s
int main(int argc, char** argv) {
    completed = static_cast<unsigned>(std::strtoul(argv[1], nullptr, 16));
    volatile int abort_flag = 0;
    std::atomic<unsigned> bits[2] = {0, 0};
    std::vector<std::thread> lanes;
    for (int i = 0; i < 32; ++i)
        lanes.emplace_back([&, i] {
            lane = i;
            uint64_t bar = 0;
            for (auto& b : bits)         // the second wait finds the flag the first has set
                if (warp_wait_or_abort(&bar, 0, &abort_flag, 2)) b |= 1u << i;
        });
    for (auto& t : lanes) t.join();
    std::printf("%%08x %%08x %%d\n", bits[0].load(), bits[1].load(), static_cast<int>(abort_flag));
}
"""


def function_text(source, name):
    """The definition of the function (template) `name`, to its closing brace."""
    at = re.search(r"(template <[^>]*>\n)?__device__ __forceinline__ bool " + name + r"\(", source).start()
    depth, i = 0, source.index("{", at)
    while True:
        depth += {"{": 1, "}": -1}.get(source[i], 0)
        i += 1
        if depth == 0:
            return source[at:i]


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    source = open(os.path.join(CSRC, "gdn_prefill_device.cuh")).read()
    d = tmp_path_factory.mktemp("wait")
    (d / "wait.cpp").write_text(HARNESS % "\n".join(function_text(source, n) for n in ("wait_or_abort", "warp_wait_or_abort")))
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-pthread", str(d / "wait.cpp"), "-o", str(d / "wait")])
    return str(d / "wait")


@pytest.mark.parametrize("completed", [0xffffffff, 0, 0x0000ffff, 0xfffffffe, 0x80000000])
def test_verdict_is_the_same_on_every_lane(harness, completed):
    first, second, flag = subprocess.check_output([harness, f"{completed:x}"], timeout=60).split()
    want = "ffffffff" if completed == 0xffffffff else "00000000"
    assert first.decode() == want and second.decode() == want
    assert int(flag) == (0 if completed == 0xffffffff else 2)


def test_issuing_warps_wait_as_one():
    """Every wait behind which a warp issues tensor-core instructions is the warp's."""
    source = open(os.path.join(CSRC, "gdn_prefill_stream.cuh")).read()
    issuer = source[source.index("===================== issuer"):source.index("===================== chain warps")]
    assert len(re.findall(r"!warp_wait_or_abort\(", issuer)) == 3
    item = open(os.path.join(CSRC, "gdn_prefill_device.cuh")).read()
    item = item[item.index("bool intra_item("):]
    for section in (issuer, item):
        assert not re.search(r"(?<!warp_)wait_or_abort[<(]", section)


def test_an_item_that_gives_up_waits_for_all_its_copies():
    """Every barrier on which the intra-chunk item's copies land is waited for (bounded) on the way out."""
    item = open(os.path.join(CSRC, "gdn_prefill_device.cuh")).read()
    item = item[item.index("bool intra_item("):]
    armed = set(re.findall(r"mbar_expect_tx\(&st\.(\w+)", item))
    bail = item[item.index("auto bail ="):]
    bail = bail[:bail.index("};")]
    assert armed == {"bar_tma", "bar_v"} and armed == set(re.findall(r"mbar_wait\(&st\.(\w+)", bail))
