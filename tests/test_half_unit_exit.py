"""On the way out of the half-unit state pass after a failed wait nothing of the CTA's is in flight: each issuing warp waits
(bounded) for its products, the CTA for the copies of every ring."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")


def test_products_and_copies_are_waited_for():
    s = open(os.path.join(CSRC, "gdn_prefill_half.cuh")).read()
    issuers = s[s.index("===================== issuers"):s.index("===================== chain warps")]
    leaving = issuers[issuers.rindex("if (!live)"):]
    assert re.search(r"mma_commit\(&bar_drain\[outputs\]\);\s*mbar_wait\(&bar_drain\[outputs\], 0u, 1u << \d+\);", leaving)
    # behind the last product, and no other way out of the loops
    assert issuers.rindex("if (!live)") > issuers.rindex("mma_ts_c") and "return" not in issuers
    assert re.search(r"mbar_init\(&bar_drain\[st\], 1\)", s)
    armed = set(re.findall(r"mbar_expect_tx\(&(bar_full_\w)", s))
    tail = s[s.index("if (abort_flag != 0"):]
    assert armed == set(re.findall(r"bar_full_\w", tail)) == {"bar_full_a", "bar_full_b", "bar_full_c"}
