"""The fixed-point transforms of csrc/tc_fx.cuh, run on the host (the same
functions, plans, tables and scales as in the kernels), against the direct
sum in long double, for every planned length and both directions.

Bound: the input is rounded at 2^-62 of the scale and every product at
2^-62; with a scale at most 2^9 times the column's root mean square and some
2^2 rounding errors per output the error stays below 2^-50 of the result's
norm for any spectrum; the steep, flat, single-mode and mean-dominated ones of
the test stay below 2^-52 (2.2e-16), the size of one float64 rounding."""
import shutil
import subprocess
import os

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0711_1429_gb300", "csrc")

PROGRAM = r"""
#include "tc_fx.cuh"
#include <cstdio>
#include <cstring>
#include <complex>
#include <random>
typedef std::complex<long double> cl;
static unsigned long long word(double d) { unsigned long long u; memcpy(&u, &d, 8); return u; }
// the levels in place, upwards (inverse) or downwards (forward)
template <int M, int S, bool SCALED, int L> void level(std::vector<fxc>& b, const fxw* tw) {
    constexpr int R = fx_radix<M, L>();
    for (int t = 0; t < M / R; ++t) {
        fxc v[R];
        for (int r = 0; r < R; ++r) {
            if (fx_at<M, L>(t, r) != fx_pad(fx_pos<M, L>(t, r))) printf("place\n");
            v[r] = b[fx_at<M, L>(t, r)];
        }
        fx_butterfly<M, S, L, SCALED && L == 0>(v, t, tw);
        for (int r = 0; r < R; ++r) b[fx_at<M, L>(t, r)] = v[r];
    }
}
template <int M, int S, bool SCALED> void passes(std::vector<fxc>& b, const fxw* tw) {
    if (S > 0) { level<M, S, SCALED, 0>(b, tw); level<M, S, SCALED, 1>(b, tw); }
    if constexpr (FxPlan<M>::NP == 3) level<M, S, SCALED, 2>(b, tw);
    if (S < 0) { level<M, S, SCALED, 1>(b, tw); level<M, S, SCALED, 0>(b, tw); }
}
template <int M, int S, bool SCALED> void check(int kind, std::mt19937_64& g) {
    const long double tp = 6.283185307179586476925286766559005768L, f = SCALED ? 0.7L : 1.0L;
    std::normal_distribution<double> nd;
    std::vector<double> x(2 * M);
    for (int i = 0; i < M; ++i) {
        const int k = i <= M / 2 ? i : M - i;
        const double a = kind == 0 ? 1.0 : kind == 1 ? pow(1.0 + k, -1.5) : kind == 2 ? (i == 1) : kind == 3 ? pow(1.0 + k, -4.0)
                                                                                              : (i == 0 ? 1.0 : 1e-9);
        x[2 * i] = 1e-3 * a * nd(g);
        x[2 * i + 1] = 1e-3 * a * nd(g);
    }
    unsigned um = 0, us = 0;
    for (double v : x) { const unsigned h = (unsigned)(word(v) >> 32) & 0x7fffffffu; um = h > um ? h : um; }
    for (double v : x) us += fx_mag((unsigned)(word(v) >> 32) & 0x7fffffffu, um >> 20);
    const int EB = fx_scale<M, S>(um, us, 1);
    std::vector<fxc> b(fx_pad(M) + 8);
    auto in = [&](double v) { return fx_from((unsigned)(word(v) >> 32), (unsigned)word(v), EB); };
    // digit-reversed order in front of the forward, behind the inverse
    for (int p = 0; p < M; ++p) {
        const int i = S > 0 ? p : fx_index<M>(p);
        b[fx_pad(p)].x = in(x[2 * i]); b[fx_pad(p)].y = in(x[2 * i + 1]);
    }
    const std::vector<fxw> tw = fx_table(M, f);
    if ((int)tw.size() != fx_tw_count<M>()) printf("table\n");
    passes<M, S, SCALED>(b, tw.data());
    const int eb = EB - 62 + fx_gain<M>();
    std::vector<cl> root(M);
    for (int i = 0; i < M; ++i) root[i] = cl(cosl(tp * i / M), S * sinl(tp * i / M));
    long double e = 0, n = 0;
    for (int p = 0; p < M; ++p) {
        const int k = S > 0 ? fx_index<M>(p) : p;
        cl s = 0;
        for (int i = 0; i < M; ++i) s += cl(x[2 * i], x[2 * i + 1]) * root[(long long)i * k % M];
        s *= f;
        const unsigned long long re = fx_bits(b[fx_pad(p)].x, eb), im = fx_bits(b[fx_pad(p)].y, eb);
        double dr, di;
        memcpy(&dr, &re, 8); memcpy(&di, &im, 8);
        e += std::norm(cl(dr, di) - s);
        n += std::norm(s);
    }
    printf("%d %d %d %d %.3Le\n", M, S, (int)SCALED, kind, sqrtl(e / n));
}
int main() {
    std::mt19937_64 g(7);
#define ALL(M) for (int k = 0; k < 5; ++k) { check<M, 1, false>(k, g); check<M, -1, false>(k, g); check<M, -1, true>(k, g); }
    FX_LENGTHS(ALL)
    for (int m = 6; m <= 1600; ++m) printf("length %d %d\n", m, fx_length(m));
    // conversions: exact where 53 bits fit, zero below the scale
    for (double v : {0.0, 1.0, -1.0, 3.25, -1e-3, 7.0 / 3.0}) {
        const fx_t F = fx_from((unsigned)(word(v) >> 32), (unsigned)word(v), 1023 + 2);
        const unsigned long long u = fx_bits(F, 1023 + 2 - 62);
        double back; memcpy(&back, &u, 8);
        printf("convert %d\n", back == v);
    }
    printf("convert %d\n", fx_from(0x3ff00000u, 0, FX_ZERO) == 0 && fx_bits(1, -100) == 0);
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


def test_transforms_of_every_planned_length(output):
    assert not [l for l in output if l in ("place", "table")]
    rows = [l.split() for l in output if l[0].isdigit()]
    assert len({r[0] for r in rows}) >= 20
    for M, S, scaled, kind, err in rows:
        assert float(err) < 2.0 ** -52, (M, S, scaled, kind, err)


def test_planned_length_is_the_smallest_that_holds_the_padded_one(output):
    got = {int(a): int(b) for _, a, b in (l.split() for l in output if l.startswith("length"))}
    planned = sorted({v for v in got.values() if v})
    for m, v in got.items():
        want = [p for p in planned if p >= m]
        assert v == (want[0] if want else 0)


def test_conversions(output):
    assert [l for l in output if l.startswith("convert")] == ["convert 1"] * 7
