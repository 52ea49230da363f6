"""The kernels' step arithmetic (csrc/range.h) at the largest counts, on the CPU.

A call accepts up to 2^31 - 1 nonzeros, rows and fibers.  The kernels walk them
in steps of 2 to 512; a sum of a position and a step passes the largest int in
the last step.  The header is compiled for the host as it is.
"""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_11622_gb300", "csrc")
MOST = 2 ** 31 - 1

SOURCE = """
#include "range.h"
extern "C" {
int step_end(int p, int n, int end) { return slnr::step_end(p, n, end); }
int inside(int p, int i, int end) { return slnr::inside(p, i, end); }
int pieces(int count, int n) { return slnr::pieces(count, n); }
// steps of n from p to end, every lane of each step: items visited (-1: one outside [p, end))
long long walk(int p, int n, int end) {
  long long items = 0;
  for (int q = p; q < end;) {
    const int e = slnr::step_end(q, n, end);
    if (e <= q || e > end) return -1;
    for (int i = 0; i < 2 * n; ++i) {
      const bool in = slnr::inside(q, i, e);
      if (in && (long long)q + i >= e) return -1;
      items += in;
    }
    q = e;
  }
  return items;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("range")
    (d / "range.cpp").write_text(SOURCE)
    so = str(d / "range.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, str(d / "range.cpp"),
                    "-o", so], check=True)
    l = ctypes.CDLL(so)
    l.walk.restype = ctypes.c_longlong
    return l


@pytest.mark.parametrize("n", [1, 2, 4, 8, 32, 64, 128, 256, 512])
@pytest.mark.parametrize("end", [0, 1, 700, MOST - 1, MOST])
def test_steps_cover_the_last_items_once(lib, n, end):
    p = max(0, end - 3 * n - 1)
    assert lib.walk(p, n, end) == end - p
    for i in (0, 1, n - 1, n):
        assert lib.inside(end, i, end) == 0
        assert lib.inside(max(0, end - 1), i, end) == (end > 0 and i == 0)
    assert lib.step_end(end, n, end) == end
    assert lib.pieces(end, n) == -(-end // n)
