"""The lengths from which gdn_prefill takes the cooperative launch, at both sides of each line (no GPU needed)."""
import pytest

from paper_2607_17979_b200 import api


@pytest.mark.parametrize("units, tokens, hinted, route", [
    (4, 2560, False, "stream"), (4, 2561, False, "fused"), (8, 2304, False, "stream"), (8, 2305, False, "fused"),
    (16, 1792, True, "stream"), (16, 1793, True, "fused"), (28, 1024, False, "stream"), (28, 1025, False, "fused"),
    (40, 1920, True, "stream"), (40, 1921, True, "fused"), (48, 2559, True, "stream"), (37, 4000, True, "fused"),
    (38, 2559, True, "fused"), (38, 2560, True, "overlap"), (48, 4095, True, "overlap"), (48, 4096, True, "fused"),
    (48, 2944, False, "stream"), (48, 2945, False, "fused"),
])
def test_lines(units, tokens, hinted, route):
    # one sequence, and for a hint below T a second one
    n = 2 if hinted else 1
    if units % n:
        n = 1
    total = tokens * n if n > 1 else tokens
    assert api.gdn_prefill_route(total, n, tokens if hinted else 0, units // n) == route
