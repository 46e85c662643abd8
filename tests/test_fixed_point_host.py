"""The fixed-point functions of csrc/gbpf_fx.cuh as host code, over their whole
ranges, against long double (64 mantissa bits or more): whole numbers and
conversions exactly, series and reciprocal within the units they state."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1811_02512_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "gbpf_fx.cuh"
using namespace gbpf;
typedef long double ld;
static ld units(long long got, ld want, int q) { return fabsl(ld(got) - ldexpl(want, q)); }
static int bad = 0;
static void check(const char *name, ld worst, ld bound) {
    std::printf("%-16s %.3Lf of %.3Lf\n", name, worst, bound);
    if (!(worst <= bound)) bad = 1;
}
int main() {
    std::mt19937_64 rng(11);
    auto uni = [&](double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); };
    ld ws = 0, wc = 0, wr = 0, wd = 0, w1 = 0, wv = 0;
    auto sincos = [&](double x) {
        long long s, c;
        const long long t = fx_from_double(x, 60);
        const ld xt = ldexpl(ld(t), -60);
        fx_sincos60(t, s, c);
        ws = fmaxl(ws, units(s, sinl(xt), 60));
        wc = fmaxl(wc, units(c, cosl(xt), 60));
    };
    for (int k = 0; k < 400000; k++) sincos(uni(-kFxThMax, kFxThMax));
    for (int k = 0; k < 20000; k++) sincos(std::ldexp(uni(-1, 1), -int(rng() % 60)));
    for (int q = -9; q <= 9; q++)  // quadrant boundaries and where the reduction turns
        for (int k = -200; k <= 200; k++) {
            const double x = q * 0.78539816339744830962 + k * std::ldexp(1.0, -50 + std::abs(k) / 8);
            if (std::fabs(x) < kFxThMax) sincos(x);
        }
    check("sin", ws, 3);
    check("cos", wc, 3);
    auto recip = [&](double x) {
        const long long v = fx_from_double(x, kFxV);
        wr = fmaxl(wr, units(fx_recip(v), 1 / ldexpl(ld(v), -kFxV), 60));
    };
    for (int k = 0; k < 400000; k++) recip((k & 1 ? -1 : 1) * uni(9.0 / 16, kFxVmax));
    for (double e : {9.0 / 16, 1.0, 1.9374999999999998, 0.99999999999999989, 1.0000000000000002})
        for (int s : {-1, 1}) recip(s * e);
    check("recip", wr, 6);
    auto small = [&](long long d, bool sm) {
        long long s, c;
        fx_small_sincos(d, sm, s, c);
        const ld x = ldexpl(ld(d), -60), h = sinl(x / 2);
        wd = fmaxl(wd, units(s, sinl(x), 60));
        w1 = fmaxl(w1, units(c, 2 * h * h, 60));
    };
    const long long edge = (1ll << 50) - 1, most = 230584300921369395ll;  // 2^-10, 0.2
    for (int k = 0; k < 400000; k++) {
        small((long long)(rng() % (2ull * edge + 1)) - edge, true);
        small((long long)(rng() % (2ull * most + 1)) - most, false);
    }
    for (long long d = edge - 2000; d <= edge; d++) {
        small(d, true), small(-d, true), small(d, false);
    }
    for (long long d = most - 2000; d <= most; d++) small(d, false), small(-d, false);
    for (long long d = -2000; d <= 2000; d++) small(d, true), small(d, false);
    // the 32-bit terms' last place, 2^-43 d^7 at 0.2, is 1.7 units, the first
    // term left out 0.15, the rounding 0.5
    check("small sin", wd, 2.5);
    check("small 1 - cos", w1, 2);
    for (int k = 0; k < 200000; k++) {
        const long long v = fx_from_double(uni(-kFxVmax, kFxVmax), kFxV), c = fx_from_double(uni(-1, 1), 60);
        wv = fmaxl(wv, fabsl(ld(fx_scale_v(v, c)) - ld(v) * ldexpl(ld(c), -60)));
    }
    check("scale", wv, 1);
    // conversions: round to nearest (ties away in, ties to even out), limbs
    for (int k = 0; k < 400000; k++) {
        const int q = int(rng() % 121) - 60;
        const double x = std::ldexp(uni(-1, 1), int(rng() % 80) - 20 - q);
        const float xf = float(std::ldexp(uni(-1, 1), int(rng() % 80) - 20 - q));
        if (fx_fits(x, q) && ld(fx_from_double(x, q)) != roundl(ldexpl(ld(x), q))) bad = 2;
        if (std::fabs(xf) >= 1.2e-38f && fx_fits(xf, q) && ld(fx_from_double(xf, q)) != roundl(ldexpl(ld(xf), q))) bad = 3;
        const long long v = (long long)(rng()) >> (rng() % 63);
        if (v != (-9223372036854775807ll - 1) && fx_to_double(v, q) != double(ldexpl(ld(v), -q))) bad = 4;
        const FxLimbs l = fx_split(v >> 2);
        if (fx_join(l.h, l.l) != (v >> 2) || l.l < -(1 << 29) || l.l >= (1 << 29)) bad = 5;
    }
    for (double x : {0.0, -0.0, 4.9e-324, 0.5, -0.5, 1.5, 2.5, 1e300})
        if (fx_fits(x, 0) && ld(fx_from_double(x, 0)) != (x == 4.9e-324 ? 0 : roundl(x))) bad = 6;
    if (fx_fits(INFINITY, -400) || fx_fits(NAN, -400) || fx_fits(0x1p61, 0) || !fx_fits(0x1.fffffffffffffp60, 0)) bad = 7;
    return bad;
}
"""


def test_fixed_point_functions(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "fx.cpp", tmp_path / "fx"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-x", "c++", "-I", CSRC, "-o", str(exe), str(src)], check=True,
                   capture_output=True, text=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout
