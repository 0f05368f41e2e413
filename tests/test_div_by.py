"""div_by (csrc/cp_internal.cuh), on the CPU: the quotient of the whitening's
phases and window means equals the rounded a / b, for random
significands, divisors of nearly all ones or of 1 and a little, small integers
(window lengths), and dividends whose quotient lies next to the middle of two
neighbouring values; infinities and NaN pass through as in a / b."""
import os
import subprocess

from paper_1412_1840_gb300 import build

SRC = r"""
#include <cstdio>
#include <limits>
#include <random>
#include "cp_internal.cuh"
int main()
{
    using namespace cpk;
    std::mt19937_64 g(1);
    long bad = 0, n = 0;
    auto check = [&](double a, double b) {
        const double rb = 1.0 / b, want = a / b, got = div_by(a, b, rb);
        bad += !(got == want || (got != got && want != want));
        n++;
    };
    for (long it = 0; it < 4000000; it++) {
        uint64_t mb = (1ull << 52) | (g() >> 12), ma = (1ull << 52) | (g() >> 12);
        if (it % 4 == 1) mb = (1ull << 53) - 1 - g() % 64;
        if (it % 4 == 2) mb = (1ull << 52) + g() % 64;
        if (it % 4 == 3) mb = 1 + g() % 4096;
        if (it & 4) {                                  // 54-bit odd quotient times b, cut to 53 bits
            unsigned __int128 t = (unsigned __int128)(((1ull << 53) | (g() >> 11)) | 1) * mb;
            while (t >> 53) t >>= 1;
            ma = (uint64_t)t + (it >> 3 & 1);
        }
        const int shift = (int)(g() % 400) - 200;
        check(std::ldexp((double)ma, shift), std::ldexp((double)mb, it % 4 == 3 ? 0 : (int)(g() % 40) - 20));
        check(-(double)ma, (double)mb);
    }
    const double inf = std::numeric_limits<double>::infinity();
    for (double b : {1.0, 3.0, 30.0, 4096.0, 0.7})
        for (double a : {inf, -inf, inf - inf, 0.0, 1.401298464324817e-45, 3.5e42}) check(a, b);
    std::printf("%ld %ld\n", n, bad);
}
"""


def test_quotients_equal_the_division(tmp_path):
    (tmp_path / "d.cu").write_text(SRC)
    subprocess.check_call([build.nvcc(), "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I",
                           os.path.join(build.ROOT, "include"), "-I", build.CSRC, str(tmp_path / "d.cu"), "-o",
                           str(tmp_path / "d")])
    n, bad = map(int, subprocess.check_output([str(tmp_path / "d")]).split())
    assert n == 8000030 and bad == 0
