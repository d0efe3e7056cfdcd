"""Where the state pass takes two CTAs per unit: the rule's own source, run on the host.  The caller's bound on the longest
sequence decides only as far as it can be true."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")

MAIN = r"""
#include <algorithm>
#include <cstdint>
#include <cstdio>
constexpr int kChunk = 64;
%s
%s
int main() {
    for (int T, N, Hv, hint; std::scanf("%%d %%d %%d %%d", &T, &N, &Hv, &hint) == 4;)
        std::putchar(half_units(T, N, Hv, known_longest(T, N, hint), 148) ? 'h' : 'w');
}
"""

CASES = [       # T, N, Hv, hint, form
    (200, 1, 32, 0, "h"), (9600, 37, 2, 0, "h"), (9600, 75, 1, 0, "w"),         # a half unit per SM, and one unit more
    (7680, 4, 32, 4096, "h"), (2048, 3, 32, 1337, "h"), (7680, 4, 32, 0, "w"),  # one long chain, known and not
    (7680, 4, 32, 3375, "w"), (7680, 4, 32, 3393, "h"),                         # either side of twice the average: 53 and 54 chunks
    (8192, 57, 32, 144, "w"), (8190, 15, 32, 546, "w"), (24000, 40, 16, 600, "w"),
    # bounds that the batch cannot reach: all tokens, a context length
    (8192, 57, 32, 8192, "w"), (8190, 15, 32, 8190, "w"), (8190, 15, 32, 131072, "w"), (24000, 40, 16, 32768, "w"),
    (7680, 4, 32, 7678, "w"), (7680, 4, 32, 7677, "h"),                         # 7677 + 1 + 1 + 1
    (32768, 1, 32, 0, "h"), (32768, 1, 100, 0, "w"), (6400, 1, 75, 100, "w"),   # one sequence: T is its length
]


def test_form(tmp_path):
    chunk, stream = (open(os.path.join(CSRC, f)).read() for f in ("gdn_prefill_chunk.cuh", "gdn_prefill_stream.cu"))
    at, rule = chunk.index("inline int32_t known_longest("), stream.index("static bool half_units(")
    text = MAIN % (chunk[at:chunk.index("\n}\n", at) + 3], stream[rule:stream.index("\n}\n", rule) + 3])
    (tmp_path / "r.cpp").write_text(text)
    subprocess.check_call(["g++", "-std=c++17", "-O1", str(tmp_path / "r.cpp"), "-o", str(tmp_path / "r")])
    out = subprocess.run([str(tmp_path / "r")], input="\n".join(" ".join(map(str, c[:4])) for c in CASES), text=True,
                         capture_output=True, check=True).stdout
    assert out == "".join(c[4] for c in CASES)
