"""The comparisons of doubles on their bit patterns (csrc/moss_bits.h), compiled
for the host with signed overflow trapped, against the comparisons themselves."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_10661_gb300", "csrc")

PROGRAM = r"""
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <limits>
#include "moss_bits.h"

static unsigned long long bits(double x) { unsigned long long b; std::memcpy(&b, &x, 8); return b; }
static int hi(double x) { return (int)(unsigned)(bits(x) >> 32); }

int main() {
    const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
    double v[64];
    int n = 0;
    for (double m : {0.0, 4.9e-324, DBL_MIN, 1e-300, 1e-9, 1e-3, 0.5, 1.0, 2.0, 50.0, 1e9, 1e300, DBL_MAX, inf, nan}) {
        v[n++] = m; v[n++] = -m;
        if (m > 0 && m < 1e300) { v[n++] = std::nextafter(m, inf); v[n++] = -std::nextafter(m, inf); }
    }
    int bad = 0;
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) {
            const double x = v[i], t = v[j];
            if (!std::signbit(t) && t == t && moss::bits_gt(bits(x), bits(t)) != (x > t)) { ++bad; std::printf("gt %a %a\n", x, t); }
            // the caller's bands are >= 0 and its scales >= 1 and finite
            if (!std::signbit(t) && t == t)
                for (double scale : {1.0, 1.5, 50.0, 1e9})
                    if (moss::bits_not_within(hi(x), hi(t), hi(scale)) && std::fabs(x) < t * scale) {
                        ++bad; std::printf("within %a %a %a\n", x, t, scale);
                    }
        }
    return bad != 0;
}
"""


def test_bit_comparisons(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fsanitize=signed-integer-overflow",
                           "-fno-sanitize-recover=all", "-I", CSRC, "-o", str(exe), str(src)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
