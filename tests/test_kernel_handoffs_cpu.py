"""Hand-offs that no run on a GPU shows reliably, read from the source.

A word that one lane writes to shared memory and another lane of its warp reads
needs a __syncwarp between the two: votes, shuffles and reductions order no
memory.  A kernel that may give up a bounded wait leaves outputs unwritten:
nothing may index with them before its status has been read.
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


def test_build_reads_the_assignment_status_before_indexing_with_the_lists():
    code = source("index.cu")
    lloyd = code[code.index("static int lloyd("):]
    lloyd = lloyd[:lloyd.index("\n}\n")]
    # within the rounds the sums are taken at once: undecided rows must hold a list
    assert "cudaMemsetAsync(a, 0" in lloyd[lloyd.index("cudaMalloc(&a,"):lloyd.index("assign_rows(")]
    assert "T->check(st)" in lloyd[lloyd.index("k_centroid_accum<<<"):]
    build = code[code.index("int ksc_build_index("):]
    build = build[build.index("assign_rows(T, ix->assign"):]
    assert "T.check(st)" in build[:build.index("k_centroid_accum<<<")]
