"""The settled path's row arithmetic (csrc/ks_window.h), compiled for the host
with signed overflow trapped: every row after the head is some window's own,
and every window lies in its sequence, up to the longest sequence accepted."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_13002_gb300", "csrc")

PROGRAM = r"""
#include "ks_window.h"
#include <cstdio>
#include <cstdlib>
using namespace ks;
static void require(bool ok, int len, int j) {
    if (!ok) { std::printf("len %d window %d\n", len, j); std::exit(1); }
}
int main(int argc, char** argv) {
    for (int a = 1; a < argc; ++a) {
        const int len = (int)std::strtoll(argv[a], nullptr, 10), nt = steady_windows(len);
        int at = kStHead;
        for (int j = 0; j < nt; ++j) {
            const StWindow w = steady_window(len, j);
            require(w.o0 == at && w.head == (j == 0) && w.last == (j == nt - 1), len, j);
            require(w.rows >= 0 && w.rows <= kStWin && w.w0 <= w.o0, len, j);
            require(len <= kStHead ? w.rows == 0 : w.rows <= len - w.w0 && w.w0 + (long long)w.rows >= w.o1, len, j);
            require(w.head || w.o0 - w.w0 == kStHalo, len, j);
            require(w.last || w.w0 + (long long)w.rows - w.o1 == kStHalo, len, j);
            int rows = 0;
            for (int t = 0; t < kStNT; ++t) rows += steady_chunk(w.rows, t * kStCH);
            require(rows == w.rows, len, j);
            at = w.o1;
        }
        require(at == len, len, nt);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("windows")
    src, exe = str(d / "windows.cpp"), str(d / "windows")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fsanitize=signed-integer-overflow",
                           "-fsanitize-undefined-trap-on-error", "-I", CSRC, src, "-o", exe])
    return exe


TOP = 2 ** 31 - 1


@pytest.mark.parametrize("lens", [list(range(1, 200)), list(range(2170, 2180)), list(range(3700, 3720)),
                                  [5300, 100003, 1 << 20], [TOP - 3072, TOP - 1537, TOP - 1536, TOP - 1535],
                                  [TOP - 1, TOP]])
def test_windows_cover_the_sequence(program, lens):
    assert subprocess.run([program, *map(str, lens)]).returncode == 0
