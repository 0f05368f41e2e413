"""cp_whiten's staging buffer, read from its source: its allocation cannot throw
through the C entry point, and an error return waits for the asynchronous copy
that reads it."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_staging_buffer_of_cp_whiten():
    src = open(os.path.join(ROOT, "paper_1412_1840_gb300", "csrc", "cp_prep.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    body = src[src.index('extern "C" cp_status cp_whiten'):]
    host = re.search(r"cudaMemcpyAsync\(tmp, (\w+)\.", body).group(1)
    decl = re.search(r"[^;{}]*\b%s\b\(([^;]*);" % host, body)
    assert "std::nothrow" in decl.group(1)
    done = body[body.index("\ndone:"):]
    assert "cudaStreamSynchronize" in done[:done.index("return st;")]
