// lux_plan.cuh -- how tensor-core RANLUX fills are divided: a row's pieces, its
// segments and their groups.  Whole-number arithmetic that the host (which sizes
// the work items and their scratch) and the kernels (which write them) share, and
// that compiles as plain C++ too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define PRNG_HD __host__ __device__ __forceinline__
#else
#define PRNG_HD inline
#endif

namespace prng {

// Multiplier operands per level: one for 2^i luxury cycles each, i < kLuxPowers.
constexpr int kLuxPowers = 32;

// Segments whose starts one row walks after one another.
constexpr int kLgLuxGroup = 4;
constexpr uint32_t kLuxGroup = 1u << kLgLuxGroup;

// A row's pieces: h draws that finish an open block (pos of its 24 delivered),
// nb blocks, m < 24 more.
struct LuxPieces {
  uint64_t nb;
  int h, m;
  PRNG_HD LuxPieces(uint64_t n, uint32_t pos) {
    const uint64_t left = pos < 24 ? 24 - pos : 0;
    h = (int)(left < n ? left : n);
    nb = (n - h) / 24;
    m = (int)(n - h - 24 * nb);
  }
};

// How long the segments are of fills that have warp_blocks blocks in all (per 32
// streams) and `longest` blocks in the longest stream, on `sms` SMs; cut: whether
// any stream is.
struct LuxSplit {
  int lgb = 0;
  bool cut = false;
};
PRNG_HD LuxSplit lux_split(uint64_t warp_blocks, uint64_t longest, uint64_t sms) {
  // Four CTAs per SM of four warps each.  Few blocks: a segment for each of those
  // warps, of 8 blocks at least (a segment's start costs about three).  Many: three
  // or four segments per warp, which even out the last wave.
  const uint64_t slots = 16 * sms, share = warp_blocks / slots;
  const uint64_t want = share < 24 ? (share + 1 > 8 ? share + 1 : 8) : (share / 4 > 16 ? share / 4 : 16);
  LuxSplit sp;
  while (sp.lgb < 40 && (1ull << sp.lgb) < want) sp.lgb++;
  // A segment's start is lgb cycles' power after the one before, group g's first
  // start the powers lgb + 4 .. lgb + 4 + log2(g): all below kLuxPowers while the
  // stream has fewer than 2^kLuxPowers blocks.  Longer ones (10^11 draws a stream
  // and up) stay whole.
  sp.cut = longest > 1ull << sp.lgb && longest >> kLuxPowers == 0;
  return sp;
}

// Segments of 2^lgb blocks that a row of n draws is cut into, wherever its first
// block starts: an open block can leave one block fewer than n / 24, and a last
// segment that is then empty is skipped when it is filled.
PRNG_HD uint64_t lux_segments(uint64_t n, int lgb) {
  const uint64_t B = 1ull << lgb, segs = (n / 24 + B - 1) >> lgb;
  return segs > 0 ? segs : 1;
}

// Segments of the group that starts at segment seg.
PRNG_HD uint32_t lux_group_size(uint64_t segs, uint32_t seg) {
  return segs > (uint64_t)seg + kLuxGroup ? kLuxGroup : segs > seg ? (uint32_t)(segs - seg) : 1u;
}

// A single fill's items lie segment after segment, `warps` rows of 32 streams in
// each: the first item of its group g, and how many groups there are.
PRNG_HD uint32_t lux_first_item(uint32_t g, uint32_t warps) { return g / warps * kLuxGroup * warps + g % warps; }
PRNG_HD uint64_t lux_groups(uint64_t segs, uint64_t warps) { return (segs + kLuxGroup - 1) / kLuxGroup * warps; }

// Whether the tile engine can store rows x pitch words (a multiple of 4) in tiles
// of 32 x 32: its tile coordinates are signed 32-bit numbers.
constexpr uint64_t kLuxTileLimit = (1ull << 31) - 32;
PRNG_HD bool lux_tiles_reach(uint64_t pitch, uint64_t rows) {
  return pitch > 0 && (pitch & 3) == 0 && pitch <= kLuxTileLimit && rows > 0 && rows <= kLuxTileLimit;
}

}  // namespace prng
