"""The state pass's CTAs together take every unit exactly once, whichever CTAs are left out of the later passes: the walk's own
source, run on the host."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")

MAIN = r"""
#include <cstdio>
#include <vector>
#define __device__
#define __forceinline__ inline
%s
int main() {
    int bad = 0, cases = 0;
    for (int n_ctas : {1, 2, 7, 148})
        for (int first_later = 0; first_later < n_ctas; first_later += n_ctas > 7 ? 21 : 1)
            for (int total : {1, n_ctas - 1, n_ctas, n_ctas + 1, 2 * n_ctas, 2 * n_ctas + 5, 5 * n_ctas + 3}) {
                std::vector<int> taken(total > 0 ? total : 0, 0);
                for (int cta = 0; cta < n_ctas; ++cta) {
                    const UnitWalk walk = {cta, n_ctas, first_later};
                    for (int i = 0, unit = walk.at(0); unit < total; unit = walk.at(++i)) ++taken[unit];
                }
                for (int t : taken) bad += t != 1;
                ++cases;
            }
    std::printf("%%d %%d\n", cases, bad);
}
"""


def test_every_unit_once(tmp_path):
    s = open(os.path.join(CSRC, "gdn_prefill_stream.cuh")).read()
    at = s.index("struct UnitWalk {")
    (tmp_path / "w.cpp").write_text(MAIN % s[at:s.index("};", at) + 2])
    subprocess.check_call(["g++", "-std=c++17", "-O1", str(tmp_path / "w.cpp"), "-o", str(tmp_path / "w")])
    cases, bad = map(int, subprocess.check_output([str(tmp_path / "w")]).split())
    assert cases > 100 and bad == 0
