"""What an expansion level reads of the row statistics: row b * top_k + j exists for frontier node j of sequence b only, so a
caller's arrays may end behind the last sequence's frontier (one row at the first level).  The kernel's load routine is compiled for
the host with pointers that record where they are read."""
import shutil
import subprocess

import pytest

from paper_2505_13254_b200 import build

SOURCE = r"""
#include <cstdio>
#include <vector>
#include "expand_child.h"
struct Span { const char* what; long n, worst; };
template <class T> struct Checked {              // an array of n entries that remembers the largest index asked for
    Span* s; std::vector<T>* v;
    T operator[](size_t i) const { if ((long)i > s->worst) s->worst = (long)i; return i < v->size() ? (*v)[i] : T(-7); }
};
int main() {
    for (int k : {1, 2, 10, 16}) for (int B : {1, 4}) for (int nf = 1; nf <= k; ++nf) for (int stride : {k, k + 6}) {
        const long rows = (long)(B - 1) * k + nf;                     // the arrays end behind the last sequence's frontier
        std::vector<float> val(rows * stride), lse(rows);
        std::vector<int> idx(rows * stride);
        for (long r = 0; r < rows; ++r) { lse[r] = 0.5f * r; for (int i = 0; i < stride; ++i) { val[r * stride + i] = 100.f * r + i; idx[r * stride + i] = 1000 * r + i; } }
        Span sv{"val", rows * stride, -1}, si{"idx", rows * stride, -1}, sl{"lse", rows, -1};
        for (int b = 0; b < B; ++b) {
            const int f = b == B - 1 ? nf : k;
            for (int t = 0; t < 256; ++t) {
                int tok = -1; float lc = 0.f;
                const bool child = load_child(t, b, k, f, stride, Checked<float>{&sv, &val}, Checked<int>{&si, &idx}, Checked<float>{&sl, &lse}, tok, lc);
                const long r = (long)b * k + t / k;
                if (child != (t < f * k)) return printf("child %d of frontier %d x %d\n", t, f, k), 1;
                if (child && (tok != 1000 * r + t % k || lc != 100.f * r + t % k - 0.5f * r)) return printf("wrong slot\n"), 1;
            }
        }
        for (const Span& s : {sv, si, sl}) if (s.worst >= s.n) return printf("%s read at %ld of %ld (k %d, frontier %d)\n", s.what, s.worst, s.n, k, nf), 1;
    }
    return 0;
}
"""


def test_nothing_is_read_past_the_frontier(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src, exe = tmp_path / "range.cpp", tmp_path / "range"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", build.CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
