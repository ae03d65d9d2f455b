"""How tensor-core RANLUX fills are divided (csrc/lux_plan.cuh), compiled as plain
C++: the arithmetic that the host sizes scratch with and the kernels index by."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
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

// log2 of the segments' blocks on 152 SMs, or -1 when the streams stay whole.
extern "C" int split(uint64_t warp_blocks, uint64_t longest) {
  const LuxSplit s = lux_split(warp_blocks, longest, 152);
  return s.cut ? s.lgb : -1;
}
extern "C" uint64_t pieces(uint64_t n, uint32_t pos) {
  const LuxPieces p(n, pos);
  return p.nb + p.h + p.m;
}
extern "C" int powers() { return kLuxPowers; }
extern "C" int tiles_reach(uint64_t pitch, uint64_t rows) { return lux_tiles_reach(pitch, rows); }
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
    L.pieces.argtypes = [ctypes.c_uint64, ctypes.c_uint32]
    L.split.argtypes = L.tiles_reach.argtypes = [ctypes.c_uint64, ctypes.c_uint64]
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


@pytest.mark.parametrize("warps", [1, 8, 4096, 2**27])
def test_every_power_of_a_cut_fill_has_an_operand(lib, warps):
    # A segment's start takes the power lgb, group g's first one lgb + 4 + (the bits of g).
    powers = lib.powers()
    for e in range(3, 64):
        for longest in (2**e - 1, 2**e, 2**e + 1, 3 * 2**e // 2):
            if longest * warps >= 2**64:
                continue
            lgb = lib.split(warps * longest, longest)
            if lgb < 0:
                continue
            segs = -(-longest // 2**lgb)
            used = [lgb] + [lgb + 4 + i for i in range(((segs - 1) >> 4).bit_length())]
            assert max(used) < powers, (longest, lgb)
            assert segs * warps < 2**31


def test_long_streams_are_cut_as_finely_as_shorter_ones(lib):
    # One stream: from 2^20 blocks on (a share of more than 24 per warp) at least a
    # segment for each of the GPU's 16 x 152 warps.
    for e in range(20, 32):
        lgb = lib.split(2**e, 2**e)
        assert lgb >= 0 and 2**e >> lgb >= 2432, e


def test_operands_are_the_powers_of_the_luxury_cycle():
    """Column k < 72 of power i at level p: the bytes of 256^k b^(-p 2^i) mod m."""
    from paper_1003_1898_gb300 import build
    L = ctypes.CDLL(build.build())
    f = L._ZN4prng15lux_host_tablesEv
    f.restype = ctypes.POINTER(ctypes.c_void_p * 2)              # a vector: begin, end
    begin, end = f().contents
    tab = np.ctypeslib.as_array(ctypes.cast(begin, ctypes.POINTER(ctypes.c_uint16)), ((end - begin) // 2,))
    levels, K = (97, 223, 389, 120, 240, 408), 80
    tab = tab.reshape(len(levels), -1, K // 8, K // 8, 8, 8)      # level, power, k / 8, n / 8, n % 8, k % 8
    assert tab.shape[1] == 32
    b = 2**24
    m = b**24 - b**10 + 1
    for l, p in enumerate(levels):
        a = pow(b, -p, m)
        for i in range(32):
            got = tab[l, i].transpose(1, 2, 0, 3).reshape(K, K).view(np.float16)   # [n][k]
            for k in (0, 1, 37, 71):
                want = (pow(256, k, m) * a % m).to_bytes(72, "little")
                np.testing.assert_array_equal(got[:72, k], np.frombuffer(want, np.uint8), err_msg=f"p {p} power {i}")
            a = a * a % m


@pytest.mark.parametrize("pitch", [4, 32, 36, 2**30, 2**31 - 64, 2**31 - 32, 2**31 - 4, 2**31, 2**31 + 32, 2**32 - 4,
                                   2**32, 2**40])
def test_tile_coordinates_are_signed_32_bit(lib, pitch):
    # The last tile of a row starts at column (pitch - 1) / 32 * 32, and a full one ends 32 on.
    last = (pitch - 1) // 32 * 32
    for p, r in ((pitch, 1), (4, pitch)):
        if lib.tiles_reach(p, r):
            assert last + 32 <= 2**31 - 1
        else:
            assert pitch > 2**31 - 32


@pytest.mark.parametrize("pos", [0, 1, 23, 24])
def test_a_head_without_draws_asks_for_nothing(lib, pos):
    # What the segments' kernel is left when a start was given up: no block, no
    # head and no tail, whatever the segment.
    assert lib.pieces(0, pos) == 0
