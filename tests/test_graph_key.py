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


def test_copies_are_marked_as_built_by_their_last_allocation():
    """A build that runs out of memory half way is taken up again by the next call, not read through null pointers."""
    body = _body("api.cu", "int ensure_transpose(sfgmres_ctx* h) {", "\n}\n")
    assert re.search(r"if \(h->(\w+)\) return 0;", body).group(1) == re.findall(r"dev_alloc\(h, &h->(\w+),", body)[-1]
    body = _body("api.cu", "int ensure_sell(sfgmres_ctx* h, bool transpose) {", "\n}\n")
    assert re.search(r"if \(!S\.(\w+)\) \{", body).group(1) == re.findall(r"dev_alloc\(h, &S\.(\w+),", body)[-1]
    body = _body("api.cu", "int ensure_sorted(sfgmres_ctx* h, bool transpose, bool f32) {", "\n}\n")
    assert body.rindex("S.ver = h->vals_ver;") > body.rindex("dev_alloc(")
