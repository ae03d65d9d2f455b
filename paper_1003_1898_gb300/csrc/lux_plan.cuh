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

}  // namespace prng
