"""The key that a replayed graph is looked up by covers every device array a captured step reads (source check: a key that
leaves one out replays a graph on freed memory, which no test may do)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_18408_gb300", "csrc")

# parts of the table that blk_v0 heads, and a pointer into the handle
DERIVED = {"blk_len", "blk_cs", "blk_list", "blk_prob", "prob_b0", "pflag", "ilu_host"}


def _body(name, start, end):
    text = open(os.path.join(CSRC, name)).read()
    a = text.index(start)
    return text[a:text.index(end, a)]


def test_plan_key_holds_every_pointer_of_the_plan():
    plan = _body("kernels.h", "struct Plan {", "\n};")
    pointers = set(re.findall(r"^\s+(?:const\s+)?[\w ]+\*\s*(\w+) = nullptr;", plan, re.M)) - DERIVED
    assert {"so_off", "so_len", "so_base", "rp", "ent", "U", "ost"} <= pointers and len(pointers) > 50
    key = _body("api.cu", "std::vector<uint64_t> plan_key(", "\n}\n")
    assert sorted(p for p in pointers if not re.search(rf"\bP\.{p}\b", key)) == []


def test_plan_key_holds_the_version_of_the_list_blocks():
    assert "h->geo_ver" in _body("api.cu", "std::vector<uint64_t> plan_key(", "\n}\n")
