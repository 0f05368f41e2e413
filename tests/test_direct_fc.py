"""Frequencies per direct-form unit (csrc/cp_internal.cuh), on the CPU: a count
tuned by the caller is lowered only where the kernel's trig table (192 KB, 12
bytes a point and frequency) does not hold it, as include/cp.h says; without one,
short batches take the smaller table that lets four blocks share an SM."""
import os
import subprocess

import pytest

from paper_1412_1840_gb300 import build

SRC = r"""
#include <cstdio>
#include "cp_internal.cuh"
int main()
{
    using namespace cpk;
    for (int n = 2; n <= kMaxN; n++)
        for (int tuned : {0, 2, 4, 8, 16})
            for (int table : {kShortTable, kTableBytes}) std::printf("%d %d %d %d\n", n, tuned, table, direct_fc(n, tuned, table));
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    d = tmp_path_factory.mktemp("fc")
    (d / "fc.cu").write_text(SRC)
    subprocess.check_call([build.nvcc(), "-std=c++17", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                           str(d / "fc.cu"), "-o", str(d / "fc")])
    return [tuple(map(int, line.split())) for line in subprocess.check_output([str(d / "fc")]).splitlines()]


def test_tuned_counts_are_kept_where_they_fit(table):
    seen = 0
    for n, tuned, room, fc in table:
        limit, fc0 = (196608, tuned) if tuned else (room, 16)
        want = next((f for f in (16, 8, 4, 2) if f <= fc0 and (n + 31) // 32 * 32 * f * 12 <= limit), 2)
        assert fc == want, (n, tuned, room)
        seen += 1
    assert seen == 4095 * 5 * 2
    assert (400, 16, 55296, 16) in table and (400, 0, 55296, 8) in table
