"""The lengths from which gdn_prefill takes the cooperative launch or the two-part production (no GPU needed): both
sides of each line of the rule, and shapes where one route was measured faster by more than 3 % on 148 SMs."""
import pytest

from paper_2607_17979_b200 import api


@pytest.mark.parametrize("units, tokens, hinted, route", [
    (4, 2624, False, "stream"), (4, 2625, False, "fused"), (8, 2432, False, "stream"), (8, 2433, False, "fused"),
    (16, 2048, False, "stream"), (16, 2049, False, "fused"), (28, 1472, False, "stream"), (28, 1473, False, "fused"),
    (32, 1472, False, "stream"), (32, 1473, False, "fused"), (40, 1920, True, "stream"), (40, 1921, True, "fused"),
    (44, 3200, False, "stream"), (44, 3201, False, "fused"), (45, 32768, False, "stream"), (48, 2559, True, "stream"),
    (37, 4000, True, "fused"), (38, 2559, True, "fused"), (38, 2560, True, "overlap"), (48, 2560, True, "overlap"),
    # a hinted chain of 40 chunks that is too short for the cooperative launch is not the two parts' either
    (4, 2560, True, "stream"),
])
def test_lines(units, tokens, hinted, route):
    # one sequence, and for a hint below T a second one
    n = 2 if hinted else 1
    if units % n:
        n = 1
    total = tokens * n if n > 1 else tokens
    assert api.gdn_prefill_route(total, n, tokens if hinted else 0, units // n) == route


@pytest.mark.parametrize("lens, heads, hinted, route, us", [
    ([18 * 64], 32, True, "stream", "51.8, fused 56.7"), ([20 * 64], 28, False, "stream", "54.3, fused 57.7"),
    ([30 * 64], 32, True, "fused", "74.6, stream 80.0"), ([50 * 64], 16, False, "fused", "102.1, stream 106.7"),
    ([60 * 64], 48, False, "stream", "170.5, fused 182.3"), ([90 * 64], 49, False, "stream", "254.2, fused 270.5"),
    ([70 * 64], 40, True, "overlap", "155.4, fused 167.0"), ([64 * 64] * 3, 16, True, "overlap", "151.1, fused 192.1"),
    ([64 * 64] * 6, 8, True, "overlap", "152.0, fused 191.3"), ([10 * 64] * 4, 8, False, "stream", "35.5, fused 40.6"),
    ([60 * 64, 30 * 64, 20 * 64, 15 * 64, 12 * 64, 10 * 64], 8, True, "fused", "121.5, overlap 131.1"),
    ([128 * 64, 64 * 64, 42 * 64, 32 * 64, 25 * 64, 21 * 64], 8, False, "fused", "228.5, stream 260.8"),
])
def test_the_measured_faster_route(lens, heads, hinted, route, us):
    assert api.gdn_prefill_route(sum(lens), len(lens), max(lens) if hinted else 0, heads) == route, us
