"""How many 16-token blocks of a chunk's accumulator the state pass overwrites with zeros comes from the chunk's record.  A record
that its producer never wrote (it left after a wait that ran out) holds anything: the function's own source, run on the host."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")

MAIN = r"""
#include <cstdint>
#include <cstdio>
#define __device__
#define __forceinline__ inline
%s
int main() {
    const uint32_t words[] = {0, 1, 2, 3, 4, 5, 64, 0x7fffffffu, 0x80000000u, 0xffffffffu, 0xfffffffcu, 0x7fc00000u};
    for (uint32_t w : words) std::printf("%%d ", record_blocks(&w));
}
"""


def test_no_word_leads_outside_the_four_blocks(tmp_path):
    s = open(os.path.join(CSRC, "gdn_prefill_chunk.cuh")).read()
    at = s.index("__device__ __forceinline__ int record_blocks(")
    (tmp_path / "b.cpp").write_text(MAIN % s[at:s.index("\n}\n", at) + 3])
    subprocess.check_call(["g++", "-std=c++17", "-O1", str(tmp_path / "b.cpp"), "-o", str(tmp_path / "b")])
    out = [int(x) for x in subprocess.check_output([str(tmp_path / "b")]).split()]
    assert out[:5] == [0, 1, 2, 3, 4] and all(0 <= n <= 4 for n in out)


def test_the_word_is_read_in_no_other_way():
    reads = 0
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        for line in open(f):
            if re.search(r"kRecGammaC \+ 4", line):
                assert "record_blocks(" in line, (f, line)
                reads += 1
    assert reads == 2
