"""Conversions between float64 and the fixed point of csrc/tc_fx.cuh at the ends
of the float64 range, on the host: the float64 nearest to a fixed-point value
exactly (compared with ldexp) down to the smallest, infinity of the value's sign
beyond the largest, and the fixed-point value of a subnormal number exactly."""
import shutil
import subprocess
import os

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0711_1429_gb300", "csrc")

PROGRAM = r"""
#include "tc_fx.cuh"
#include <cstdio>
#include <cstring>
static double value(unsigned long long u) { double d; memcpy(&d, &u, 8); return d; }
int main() {
    const fx_t F[] = {1, 3, (1LL << 30) + 1, (1LL << 52) + 1, (1LL << 61) + 12345, (1LL << 62) - 1, (1LL << 53) - 1, 1LL << 61};
    for (fx_t f : F)
        for (int neg = 0; neg < 2; ++neg)
            // F 2^(eb - 1023) around 2^1024
            for (int eb = 1950; eb < 2120; ++eb) {
                const fx_t x = neg ? -f : f;
                // to 53 bits, halves away from zero as the conversion does
                int top = 63 - __builtin_clzll((unsigned long long)f), cut = top - 52;
                unsigned long long m = cut > 0 ? ((unsigned long long)f >> cut) + (((unsigned long long)f >> (cut - 1)) & 1) : (unsigned long long)f;
                const double want = std::ldexp((double)m, eb - 1023 + (cut > 0 ? cut : 0)) * (neg ? -1.0 : 1.0);
                const double got = value(fx_bits(x, eb));
                if (!(got == want)) printf("top %lld %d %a %a\n", (long long)x, eb, got, want);
            }
    for (fx_t f : F)
        for (int neg = 0; neg < 2; ++neg)
            // around the subnormal range; ties away from zero as above
            for (int eb = -150; eb < 30; ++eb) {
                const fx_t x = neg ? -f : f;
                const int top = 63 - __builtin_clzll((unsigned long long)f);
                const int last = top + eb - 1023 - 52 < -1074 ? -1074 : top + eb - 1023 - 52;     // exponent of the last bit kept
                const int cut = last - (eb - 1023);
                const unsigned long long m = cut > 63 ? 0 : cut > 0 ? ((unsigned long long)f >> cut) + (((unsigned long long)f >> (cut - 1)) & 1) : (unsigned long long)f;
                const double want = std::ldexp((double)m, eb - 1023 + (cut > 0 ? cut : 0)) * (neg ? -1.0 : 1.0);
                const double got = value(fx_bits(x, eb));
                if (!(got == want)) printf("bottom %lld %d %a %a\n", (long long)x, eb, got, want);
            }
    // fixed-point value of numbers down to the smallest, with the scale a column of them has
    for (int e = -1074; e < -1000; ++e)
        for (double q : {1.0, -1.0, 1.5, -1.3, 1.9999}) {
            const double v = std::ldexp(q, e);
            unsigned long long u;
            memcpy(&u, &v, 8);
            const unsigned hi = (unsigned)(u >> 32), ab = hi & 0x7fffffffu;
            const int EB = fx_scale<96, 1>(ab, 96 * fx_mag(ab, ab >> 20), 1);
            const fx_t f = fx_from(hi, (unsigned)u, EB);
            const long double want = std::ldexp((long double)v, 62 - (EB - 1023));
            if (want != std::floor(want) ? std::fabs((long double)f - want) >= 1.0L : (long double)f != want) printf("from %a %d %lld\n", v, EB, (long long)f);
            if (std::fabs(want) > 4611686018427387904.0L) printf("from scale %a %d\n", v, EB);
            if (value(fx_bits(f, EB - 62)) != v) printf("from and back %a %d\n", v, EB);
        }
    return 0;
}
"""


@pytest.fixture(scope="module")
def output(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(PROGRAM)
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, str(d / "fx.cpp"), "-o", str(d / "fx")], check=True)
    return subprocess.run([str(d / "fx")], check=True, capture_output=True, text=True).stdout.splitlines()


def test_values_beyond_the_largest_become_infinite(output):
    assert not [l for l in output if l.startswith("top")]


def test_values_down_to_the_smallest(output):
    assert not [l for l in output if l.startswith("bottom")]


def test_subnormal_numbers_keep_their_bits(output):
    assert not [l for l in output if l.startswith("from")]
