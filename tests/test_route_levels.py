"""Where gdn_prefill produces the records in two parts (no GPU needed): both sides of the line, shapes where one route was
measured faster by more than 3 % on 148 SMs, and what the caller's bound on the longest sequence can do to it."""
import pytest

from paper_2607_17979_b200 import api


@pytest.mark.parametrize("units, tokens", [(1, 80512), (4, 20096), (16, 5056), (32, 2496), (36, 2624), (48, 3712), (64, 4544), (70, 4800)])
def test_lines_of_one_sequence(units, tokens):
    assert api.gdn_prefill_route(tokens, 1, 0, units) == "overlap"
    assert api.gdn_prefill_route(tokens - 1, 1, 0, units) == "stream"


@pytest.mark.parametrize("n, heads, route", [(35, 2, "overlap"), (71, 1, "stream"), (2, 35, "overlap"), (2, 36, "stream"), (18, 4, "stream")])
def test_most_units(n, heads, route):
    """Every half unit needs an SM, and eight more are left to the producers: 70 units of 148 SMs."""
    assert api.gdn_prefill_route(80000, n, 30000, heads) == route


@pytest.mark.parametrize("lens, heads, route, us", [
    ([60 * 64], 8, "stream", "83.7, in two parts 92.2"), ([240 * 64], 8, "overlap", "293.7, three launches 305.8"),
    ([18 * 64], 32, "stream", "40.1, in two parts 53.3"), ([50 * 64], 32, "overlap", "91.2, three launches 96.0"),
    ([320 * 64], 32, "overlap", "428, three launches 564"), ([70 * 64], 40, "overlap", "136.7, three launches 142.7"),
    ([50 * 64], 48, "stream", "115.2, in two parts 119.2"), ([40 * 64], 64, "stream", "115.0, in two parts 123.1"),
    ([86 * 64, 28 * 64], 32, "overlap", "174.7, three launches 180.8"),
    ([60 * 64] + [30 * 64] * 6, 10, "stream", "126.9, in two parts 138.0"),
    ([53 * 64] + [16 * 64] * 34, 2, "stream", "98.9, in two parts 109.0"),
])
def test_the_measured_faster_route(lens, heads, route, us):
    assert api.gdn_prefill_route(sum(lens), len(lens), max(lens), heads) == route, us


def test_a_bound_that_cannot_be_true_counts_as_none():
    for T, n, heads in ((8192, 2, 32), (8192, 2, 16), (6000, 4, 16)):
        for hint in (T, T - n + 2, 1 << 20):
            assert api.gdn_prefill_route(T, n, hint, heads) == api.gdn_prefill_route(T, n, 0, heads)
    # one sequence is as long as it is
    assert api.gdn_prefill_route(4096, 1, 100, 32) == api.gdn_prefill_route(4096, 1, 0, 32) == "overlap"
