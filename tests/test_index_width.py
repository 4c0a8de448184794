"""Index widths of the dense level arrays (source level, CPU).  At D = 10 and leaf sizes below 8 the
levels have 1,227,133,513 slots: any multiple of that from 2 on needs 64 bits (an evaluation there
takes 120 GB, and a 32-bit product is an address before its array)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_10059_gb300", "csrc")


def _body(src, head):
    s = src[src.index(head):]
    return s[:s.index("\n}\n")]


def test_slots_of_the_deepest_tree_need_64_bits():
    slots = sum(8 ** l for l in range(11))
    assert slots == 1227133513 and slots < 2 ** 31 < 2 * slots


def test_list_arrays_are_offset_in_64_bits():
    s = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "sph_api.cu")).read())
    body = _body(s, "ListDev list_dev(sph_ctx *c)")
    assert re.search(r"const (size_t|int64_t) nb = std::max\(c->list_cap, 1\);", body)
    assert "(int)(4 *" not in s
    k = open(os.path.join(CSRC, "k_tree.cu")).read()
    assert "size_t scan_tmp_ints(int64_t n)" in k and "const int64_t ntiles" in _body(k, "size_t scan_tmp_ints(int64_t n)")
