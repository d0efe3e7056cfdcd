"""FastDiv divides exactly over its whole range: the functions' own source, run on the host."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")

MAIN = r"""
#include <cstdint>
#include <cstdio>
#define __host__
#define __device__
%s
int main() {
    const uint32_t top = 0x7fffffffu;
    unsigned long long bad = 0, n = 0;
    for (uint32_t k = 1; k < 70000; ++k) {
        // every small divisor, and powers of two and their neighbours
        const uint32_t d = k <= 4096 ? k : k <= 4096 + 3 * 30 ? ((1u << (k - 4097) / 3) + (k - 4097) %% 3 ? (1u << (k - 4097) / 3) + (k - 4097) %% 3 : 1) : 2147u * (k %% 999983u) + 1;
        const FastDiv f = fast_div(d);
        const uint32_t q = top / d;
        const uint32_t xs[] = {0, 1, d - 1, d, d + 1, 2 * d - 1, q * d, q * d - 1, top, top - 1, (q / 2) * d, (q / 2) * d + d - 1};
        for (uint32_t x : xs)
            if (x <= top) { ++n; bad += static_cast<uint32_t>(static_cast<int32_t>(x) / f) != x / d; }
    }
    std::printf("%%llu %%llu\n", n, bad);
}
"""


def test_exact(tmp_path):
    s = open(os.path.join(CSRC, "gdn_common.cuh")).read()
    text = s[s.index("struct FastDiv {"):s.index("struct DecodeParams {")]
    (tmp_path / "d.cpp").write_text(MAIN % text)
    subprocess.check_call(["g++", "-std=c++17", "-O1", str(tmp_path / "d.cpp"), "-o", str(tmp_path / "d")])
    n, bad = map(int, subprocess.check_output([str(tmp_path / "d")]).split())
    assert n > 500000 and bad == 0
