"""How far ahead of the chains the producers of the two-part route may run: the model's own source on the host, in a simulation of
chains and producers.  Where the producers make less than the chains read, holding them to the window in front of the first chain
leaves them idle first and late afterwards; the bound must not cost time against no bound, and must be the window where they keep up."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")

MAIN = r"""
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>
#define __device__
#define __forceinline__ inline
%s
%s
// chunk steps until the last chain is through; a producer takes 1 / kPaceRate steps an item, ready six steps after its begin
double steps(const SplitModel& m, int max_nc, long long cut, long long total, const std::vector<long long>& bound) {
    const double dt = 0.05;
    std::vector<double> begun;              // how many items had been begun at each instant
    double t = 0, made = 0, chain = 0;
    for (long n = 0; chain < max_nc && n < 4000000; ++n, t += dt) {
        const int at = static_cast<int>(chain);
        const long long busy = 2ll * m.Hv * (m.pos[at + 1] - m.pos[at]);
        const long long until = std::min(bound[at], total);
        if (cut + made < until) made = std::min(made + kPaceRate * (m.sms - busy) * dt, static_cast<double>(until - cut));
        begun.push_back(made);
        const long back = n - static_cast<long>(6 / dt);
        const double ready = cut + (back >= 0 ? begun[back] : 0);
        if (ready >= m.needed(at) || ready >= total) chain += dt;
    }
    return t;
}
int main(int argc, char** argv) {
    const int Hv = std::atoi(argv[1]), sms = std::atoi(argv[2]);
    std::vector<int> nc;
    for (int i = 3; i < argc; ++i) nc.push_back(std::atoi(argv[i]));
    const int max_nc = *std::max_element(nc.begin(), nc.end());
    std::vector<int32_t> pos(max_nc + 2, 0);
    for (int j = 0; j <= max_nc; ++j)
        pos[j + 1] = pos[j] + static_cast<int32_t>(std::count_if(nc.begin(), nc.end(), [&](int x) { return x > j; }));
    const SplitModel m = {pos.data(), Hv, sms};
    const long long total = static_cast<long long>(Hv) * pos[max_nc];
    long long cut = 0, lacks = 0;
    int step = 0;
    for (int j = 0; j < max_nc; ++j) {
        cut = std::max(cut, m.cut_for(j));
        if (m.short_of(j) >= lacks && m.short_of(j) > 0) lacks = m.short_of(j), step = j;
    }
    cut = std::min(cut + kSplitMarginItems, total);
    std::vector<long long> bound, window, none(max_nc, total);
    long long beyond = 0;
    for (int j = 0; j < max_nc; ++j) {
        bound.push_back(m.bound(j, lacks, step));
        window.push_back(static_cast<long long>(Hv) * pos[j] + kPaceItems);
        beyond = std::max(beyond, bound[j] - window[j]);
    }
    std::printf("%%f %%f %%f %%lld\n", steps(m, max_nc, cut, total, bound), steps(m, max_nc, cut, total, none),
                steps(m, max_nc, cut, total, window), beyond);
}
"""


@pytest.fixture(scope="module")
def simulate(tmp_path_factory):
    s = open(os.path.join(CSRC, "gdn_prefill_fused.cu")).read()
    consts = "\n".join(re.findall(r"^constexpr (?:int|float) k(?:Split|Pace)\w+ = [^;]+;", s, re.M))
    at = s.index("struct SplitModel {")
    d = tmp_path_factory.mktemp("pace")
    (d / "p.cpp").write_text(MAIN % (consts, s[at:s.index("\n};\n", at) + 4]))
    subprocess.check_call(["g++", "-std=c++17", "-O2", str(d / "p.cpp"), "-o", str(d / "p")])

    def run(heads, lens, sms=148):
        out = subprocess.check_output([str(d / "p"), str(heads), str(sms), *map(str, lens)]).split()
        return [float(x) for x in out[:3]] + [int(out[3])]
    return run


@pytest.mark.parametrize("heads, chunks", [(32, [128, 128]), (16, [100] * 3), (16, [64] * 3), (8, [100] * 6), (64, [128]), (40, [256]),
                                           (70, [512]), (32, [86, 28]), (32, [64, 8]), (32, [469, 16]), (16, [312, 62, 16]), (2, [500] * 35)])
def test_no_later_than_without_a_bound(simulate, heads, chunks):
    bounded, free, window, _ = simulate(heads, chunks)
    assert bounded <= 1.01 * free + 1
    if heads * len(chunks) >= 48 and min(chunks) >= 100:        # the fault: the window alone
        assert window > 1.05 * free


@pytest.mark.parametrize("heads, chunks", [(32, [512]), (8, [512]), (4, [1000]), (1, [2000] * 32)])
def test_the_window_where_the_producers_keep_up(simulate, heads, chunks):
    bounded, free, _, beyond = simulate(heads, chunks)
    assert beyond <= 64 and bounded <= 1.01 * free + 1
