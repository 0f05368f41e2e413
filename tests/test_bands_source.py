"""Order of the shared-memory accesses of k_window_refine's in-place compaction,
read from its source: a lane may write an entry that another lane reads in the
same trip, so a __syncwarp (a vote alone orders no memory) stands between the
trip's reads and its writes, and another after them."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_compaction_separates_reads_and_writes():
    src = open(os.path.join(ROOT, "paper_1412_1840_gb300", "csrc", "cp_bands.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    body = src[src.index("int kept = 0;"):src.index("rel = kept;")]
    read = [m.end() for m in re.finditer(r"= r < rel \? (kk|val|eb)\[r\]|, f = r < rel \? fv\[r\]", body)]
    write = [m.start() for m in re.finditer(r"(val|eb|fv|kk)\[q\] =", body)]
    sync = [m.start() for m in re.finditer(r"__syncwarp\(\)", body)]
    assert len(read) == 4 and len(write) == 4 and len(sync) == 2
    assert max(read) < sync[0] < min(write) and max(write) < sync[1]
