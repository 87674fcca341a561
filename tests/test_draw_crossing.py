"""The token that an inverse-CDF draw takes has mass, whatever its sums round to.  The walk's crossing of four tokens is compiled for the host
and run over groups of masses as a thread of the walk has them: zeros among and behind them, magnitudes that round away in fp64, goals at
and next to every running sum."""
import shutil
import subprocess

import pytest

from paper_2505_13254_b200 import build

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "draw_cross.h"
const int N = 16;
// the walk's loop over a thread's tokens
int draw(const double* m, double run, double goal) {
    for (int g = 0; g < N; g += 4) {
        const double t[4] = {m[g], m[g + 1], m[g + 2], m[g + 3]};
        const int at = crossing_of_four(t, goal, run);
        if (at >= 0) return g + at;
    }
    return -1;
}
int check(const double* m, double run, double goal) {
    const int at = draw(m, run, goal);
    if (at >= 0 && !(m[at] > 0.0)) return printf("token %d without mass, goal %a behind %a\n", at, goal, run), 1;
    // one by one: the first crossing; a sum taken in another order moves it by its rounding, far less than a token where masses are alike
    double r = run, size = 0.0, least = 1e300;
    int first = -1;
    for (int i = 0; i < N; ++i) {
        r += m[i]; size += m[i];
        if (first < 0 && r > goal) first = i;
        if (m[i] > 0.0) least = std::fmin(least, m[i]);
    }
    double near = 1e300;
    r = run;
    for (int i = 0; i < N; ++i) { r += m[i]; near = std::fmin(near, std::fabs(r - goal)); }
    if (near > 64 * 0x1p-53 * (run + size) && at != first) return printf("token %d, one by one %d\n", at, first), 1;
    return 0;
}
int main() {
    // four masses whose sum passes the goal in pairs and not one by one, nothing behind them
    double m[N] = {0x1p-53, 0x1p-53, 0x1p-53, 0x1p-53};
    if (draw(m, 1.0, 1.0) != 3) return printf("rounded crossing: token %d\n", draw(m, 1.0, 1.0)), 1;
    m[3] = 0.0; m[1] = 0x1.8p-53; m[2] = 0.0;
    if (check(m, 1.0, 1.0)) return 1;
    std::mt19937_64 rng(7);
    for (int it = 0; it < 200000; ++it) {
        const double run = it % 3 ? std::ldexp((double)(rng() >> 11), -53 + (int)(rng() % 4)) : 0.0;
        const int spread = 1 + (int)(rng() % 60);
        for (int i = 0; i < N; ++i)
            m[i] = rng() % 4 ? (double)(float)std::ldexp(1.0 + (double)(rng() >> 41) * 0x1p-23, -(int)(rng() % spread) - (int)(rng() % 3) * 20) : 0.0;
        double r = run;
        const int k = (int)(rng() % N);
        for (int i = 0; i <= k; ++i) r += m[i];
        for (double goal : {r, std::nextafter(r, 0.0), std::nextafter(r, 4.0), run + (r - run) * 0.5})
            if (goal >= run && check(m, run, goal)) return 1;
    }
    return 0;
}
"""


def test_the_drawn_token_has_mass(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src, exe = tmp_path / "cross.cpp", tmp_path / "cross"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", build.CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
