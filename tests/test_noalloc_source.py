"""Lifetimes in cp_best_period_noalloc, read from its source: host memory that
an asynchronous copy reads or writes has to outlive the stream's
synchronisation, which on an error is the guard's destructor."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_copied_host_memory_outlives_the_guard():
    src = open(os.path.join(ROOT, "paper_1412_1840_gb300", "csrc", "cp_noalloc.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    body = src[src.index('extern "C" cp_status cp_best_period_noalloc'):]
    body = body[body.index("{"):]
    guard = body.index("SyncOnError guard")
    copies = re.findall(r"cudaMemcpyAsync\(([^;]*?)(cudaMemcpyHostToDevice|cudaMemcpyDeviceToHost)", body)
    assert len(copies) == 2
    for args, kind in copies:
        host = re.sub(r"\W", "", args.split(",")[1 if kind == "cudaMemcpyHostToDevice" else 0])
        decl = re.search(r"^[ ]*(char|unsigned long long) %s\b[^;]*;" % host, body, re.M)
        assert decl, host
        before = body[:decl.start()]
        assert before.count("{") - before.count("}") == 1, "%s is declared in an inner block" % host
        assert decl.start() < guard, "%s is destroyed before the guard synchronises" % host
