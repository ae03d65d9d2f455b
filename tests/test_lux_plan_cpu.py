"""How tensor-core RANLUX fills are divided (csrc/lux_plan.cuh), compiled as plain
C++: the arithmetic that the host sizes scratch with and the kernels index by."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <vector>
#include "lux_plan.cuh"
using namespace prng;

// Walks the items of a single fill as the kernels do.  0: every item that a
// segment's start is written for was allocated, is written once and is the item
// of that segment and row; every block of the fill lies in one of them.
extern "C" int walk(uint64_t n, uint32_t pos, uint64_t rows, int lgb) {
  const uint64_t warps = (rows + 31) / 32, segs = lux_segments(n, lgb);       // the host's sizes
  const uint64_t n_items = warps * segs, n_groups = lux_groups(segs, warps);
  std::vector<int> seen(n_items, 0);
  for (uint64_t g = 0; g < n_groups; g++) {                                     // the kernel's indices
    const uint32_t it = lux_first_item((uint32_t)g, (uint32_t)warps);
    if (it >= n_items) return 1;
    const uint32_t seg = it / (uint32_t)warps;
    const uint32_t cnt = lux_group_size(lux_segments(n, lgb), seg);
    for (uint32_t j = 0; j < cnt; j++) {
      const uint64_t at = it + j * warps;
      if (at >= n_items) return 2;
      if (at / warps != seg + j || at % warps != it % warps) return 3;
      if (seen[at]++) return 4;
    }
  }
  for (int s : seen)
    if (s != 1) return 5;
  const LuxPieces p(n, pos);
  if (p.h + 24 * p.nb + p.m != n || p.m >= 24) return 6;
  return segs << lgb >= p.nb ? 0 : 7;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("lux_plan")
    src, so = d / "plan.cpp", d / "plan.so"
    src.write_text(SOURCE)
    cxx = shutil.which("g++") or shutil.which("c++")
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1003_1898_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.walk.argtypes = [ctypes.c_uint64, ctypes.c_uint32, ctypes.c_uint64, ctypes.c_int]
    return L


@pytest.mark.parametrize("pos", [0, 1, 4, 12, 23, 24])
def test_segment_starts_stay_in_their_scratch(lib, pos):
    # Around multiples of a segment, where a row's open block decides whether its
    # blocks fill one segment more; more and fewer than a group of segments.
    for lgb in (3, 4, 6):
        B = 24 << lgb
        for segs in (1, 2, 5, 15, 16, 17, 31, 32, 33, 50):
            for d in (-24, -1, 0, 1, 23 - pos, 24 - pos, 24, 25):
                for rows in (1, 32, 33, 256):
                    n = segs * B + d
                    assert lib.walk(n, pos, rows, lgb) == 0, (n, rows, lgb)


@pytest.mark.parametrize("rows,n,lgb", [(256, 984, 3), (4096, 984, 3), (1, 24, 3), (1, 1, 3)])
def test_fresh_handles(lib, rows, n, lgb):
    assert lib.walk(n, 0, rows, lgb) == 0
