"""Hand-offs inside kernels that no run on a GPU shows reliably, read from the source.

A word that one lane writes to shared memory and another lane of its warp reads
needs a __syncwarp between the two: votes, shuffles and reductions order no
memory.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_03298_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)  # code, not comments


def test_scan_tc_flush_orders_its_picked_columns():
    code = source("scan_tc.cu")
    writes = [m.end() for m in re.finditer(r"\bs_pick\[[^;]*?\]\s*=[^=]", code)]
    reads = [m.start() for m in re.finditer(r"[=?]\s*s_pick\[", code)]
    assert len(writes) == 1 and len(reads) == 1 and writes[0] < reads[0]
    assert "__syncwarp()" in code[writes[0]:reads[0]]
    # and the next flush writes only after this one's reads
    assert "__syncwarp()" in code[reads[0]:code.index("if (!ok) break;", reads[0])]
