"""The library's own plane arithmetic (csrc/planes.h), compiled for the host: a
row holds its nodes and ghost nodes, rows and planes start on the stated
boundaries, no plane takes more than rows of whole lines would, and the walks
of the 3D updates -- pairs of rows, single nodes, pairs of a row -- meet every
node exactly once for every block size the autotuner tries."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2004_11863_gb300 import build

SOURCE = r"""
#include "planes.h"
using namespace mlbm;
extern "C" void pitch(int D, int n0, int n1, int g0, int g1, int* s) {
  plane_pitch(D, n0, n1, g0, g1, s[0], s[1]);
}
// Adds one to count[y * n0 + x] for every node that the threads of whole blocks
// take: `rows` rows by `width` elements a thread.
extern "C" void walk(int SX, int n0, int n1, int rows, int width, int threads, int* count) {
  const long long n = plane_elements(SX / width, (n0 + width - 1) / width, (n1 + rows - 1) / rows);
  for (long long e = 0; e < (n + threads - 1) / threads * threads; ++e) {
    int x, y;
    plane_node(SX / width, (unsigned)e, x, y);
    x *= width;
    y *= rows;
    if (x >= n0 || y >= n1) continue;
    for (int dy = 0; dy < rows; ++dy)
      for (int dx = 0; dx < width; ++dx)
        if (x + dx < n0 && y + dy < n1) ++count[(y + dy) * n0 + x + dx];
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("planes")
    (d / "planes.cc").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", f"-I{build.CSRC}",
                    "-o", str(d / "libplanes.so"), str(d / "planes.cc")], check=True)
    return ctypes.CDLL(str(d / "libplanes.so"))


def pitch_of(lib, D, n0, n1, g0, g1):
    s = (ctypes.c_int * 2)()
    lib.pitch(D, n0, n1, g0, g1, s)
    return s[0], s[1]


SIZES = [(4, 4), (5, 7), (23, 5), (24, 6), (25, 9), (32, 9), (33, 8), (63, 5), (65, 6), (81, 10),
         (160, 4), (161, 7), (193, 5), (257, 3), (1023, 4)]


@pytest.mark.parametrize("n0,n1", SIZES)
@pytest.mark.parametrize("g0", [0, 1])
@pytest.mark.parametrize("g1", [0, 1])
def test_pitch(lib, n0, n1, g0, g1):
    whole = -(-(n0 + 2 * g0) // 32) * 32
    assert pitch_of(lib, 2, n0, n1, g0, g1) == (whole, n1 + 2 * g1)
    sx, sy = pitch_of(lib, 3, n0, n1, g0, g1)
    assert sx >= n0 + 2 * g0 and sy >= n1 + 2 * g1
    assert sx % 8 == 0 and (sx * sy) % 32 == 0
    assert sx * sy <= whole * (n1 + 2 * g1)


@pytest.mark.parametrize("n0,n1", SIZES)
@pytest.mark.parametrize("g", [0, 1])
def test_every_node_once(lib, n0, n1, g):
    sx, _ = pitch_of(lib, 3, n0, n1, g, g)
    for threads in (32, 64, 96, 128):
        for rows, width in ((2, 1), (1, 1), (1, 2)):
            count = np.zeros(n0 * n1, dtype=np.int32)
            lib.walk(sx, n0, n1, rows, width, threads,
                     count.ctypes.data_as(ctypes.POINTER(ctypes.c_int)))
            assert np.all(count == 1)
