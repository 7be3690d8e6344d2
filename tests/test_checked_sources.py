"""The bounds-checked build covers the counting sort: every kernel of it that
indexes by a fine key or by a slot has a check for it before the access."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_03056_gb300", "csrc",
                   "relax.cu")


def kernel(name):
    src = re.sub(r"//[^\n]*", "", open(SRC).read())
    m = re.search(r"\b%s\([^{;]*\{" % name, src)
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    return src[m.end():i]


@pytest.mark.parametrize("name,check,access", [
    ("k_keys_count", r"FPPG_CHECK\(k < F,", r"cnt \+ k"),
    ("k_crowd_counts", r"FPPG_CHECK\(k < F,", r"cnt \+ k"),
    ("k_place", r"FPPG_CHECK\(key\[i\] < F1 - 1,", r"fstart\[key\[i\]\]"),
    ("k_place", r"FPPG_CHECK\(k < N,", r"id_a\[k\]"),
    ("k_rank_gather", r"FPPG_CHECK\(f < F,", r"fstart\[f\]"),
    ("k_rank_gather", r"FPPG_CHECK\(slot < N,", r"put_slot\(slot"),
])
def test_the_counting_sort_checks_what_it_indexes(name, check, access):
    body = kernel(name)
    c, a = re.search(check, body), re.search(access, body)
    assert c and a and c.start() < a.start()
