"""The division of the multigrid sweeps (quotient() of mg_pcg.cuh: a product with the
stored reciprocal, corrected once by its exact remainder) against the IEEE
division, on the host: the function's own text compiled as C++.

Where no intermediate leaves the normal range the two are equal, except for
quotients within 2^-105 of a rounding boundary, which random operands do not
meet.  Operands of a few significant bits meet exact quotients and halfway
neighbours."""
import os
import re
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <initializer_list>
using std::fma;
%s
static uint64_t s = 0x9e3779b97f4a7c15ull;
static uint64_t next() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
// random sign and significand of `bits` bits, exponent in [-e, e]
static double draw(int bits, int e) {
    const uint64_t m = (next() >> 12) >> (52 - bits) << (52 - bits);
    const double x = 1.0 + (double)m / 4503599627370496.0;
    return std::ldexp(next() & 1 ? x : -x, (int)(next() %% (2 * e + 1)) - e);
}
int main() {
    long bad = 0;
    for (int bits : {52, 26, 8, 3})
        for (long k = 0; k < 2000000; ++k) {
            const double v = draw(bits, 300), d = std::fabs(draw(k %% 2 ? 52 : bits, 300));
            if (quotient(v, d, 1.0 / d) != v / d) ++bad;
        }
    // the ends of the significand's range, and zero
    const double ends[] = {1.0, 1.0 + 0x1p-52, 1.0 + 0x1p-51, 1.5, 2.0 - 0x1p-52, 2.0 - 0x1p-51};
    for (double v : ends)
        for (double d : ends) bad += quotient(v, d, 1.0 / d) != v / d;
    bad += quotient(0.0, 3.0, 1.0 / 3.0) != 0.0;
    std::printf("%%ld\n", bad);
}
"""


def test_quotient_equals_division():
    path = os.path.join(ROOT, "paper_1407_0674_gb300", "csrc", "mg_pcg.cuh")
    body = re.search(r"__device__ __forceinline__ (double quotient\(.*?\n\})", open(path).read(), re.S).group(1)
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.cpp"), os.path.join(d, "t")
        open(src, "w").write(PROGRAM % ("static " + body))
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", src, "-o", exe, "-lm"])
        assert int(subprocess.check_output([exe])) == 0
