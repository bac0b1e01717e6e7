"""Conversions between float64 and the fixed point of csrc/tc_fx.cuh at the ends
of the float64 range, on the host: the float64 nearest to a fixed-point value
exactly (compared with ldexp), and infinity of the value's sign beyond it."""
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
