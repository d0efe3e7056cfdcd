"""The intra-chunk pipeline's way out when a wait runs out: a role finishes its item with whatever is there, so what it addresses by
must be its own by then; the item's place in shared memory may already be the next one's."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17979_b200", "csrc")


def role_sections():
    s = open(os.path.join(CSRC, "gdn_prefill_intra.cuh")).read()
    s = s[s.index("void produce_role("):]
    sections = s[:s.index("if (abort_flag != 0)")].split("// =====================")[1:]
    return [x for x in sections if not x.startswith(" items")]      # (that warp writes the places)


def test_an_items_place_is_not_asked_again_behind_a_wait():
    sections = role_sections()
    assert len(sections) == 8
    for section in sections:
        body = section[section.index("item_at("):]
        behind = body[body.index("wait(kB"):]
        again = re.findall(r"info(?:s\[[^\]]*\])?\.(?:rec|len|t0|hv|hqk)\b", behind)
        assert not again, (section.splitlines()[0], again)
