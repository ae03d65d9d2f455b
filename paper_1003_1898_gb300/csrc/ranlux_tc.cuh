// ranlux_tc.cuh -- entry points of the tensor-core RANLUX fills (k_ranlux_tc.cu).
#pragma once

#include <cuda.h>

#include "lux_plan.cuh"
#include "ranlux.cuh"

namespace prng {

// Lowest luxury p that the tensor-core form serves: its state of a fill that
// ends inside a block needs at least 24 discarded steps per cycle (p >= 48), and
// below p = 97 the borrow chain costs less than the carries of the product.
constexpr int kLuxTcMinP = 97;

// Fill the multiplier operands of the current device (idempotent; called when a
// RANLUX handle is created, before any of its fills).
cudaError_t lux_tables_init();

// Whether a kernel on device `dev` has given up waiting for its tensor core: its
// fill's output and handle are then not the ones asked for, and every later call
// on a RANLUX handle of the device says so.  Reads a word of host memory
// (lux_failed_word, nullptr before the device's first RANLUX handle).
bool lux_tc_failed(int dev);
uint32_t* lux_failed_word(int dev);

// The launch tile of a plain fill that leaves it to the library.
Tile ranlux_auto_tile(const FillDesc& d);

// A plain fill; with `segments` a few long streams may be cut into segments.
cudaError_t launch_fill_ranlux_tc(const FillDesc& d, bool segments, cudaStream_t s);

// Fills of one luxury level and output type as work items of 32 streams and one
// segment (BatchItem: req, row0, and the segment in `rows`).
struct LuxJob {
  CUtensorMap map;          // single fill: its output's, if tiles
  FillDesc one;             // single fill (reqs == nullptr): item = segment x warps + warp of 32 streams
  const BatchReq* reqs;
  const BatchItem* items;
  const CUtensorMap* maps;  // by request, valid where BatchReq::tiles
  uint32_t* counter;        // items are popped from it, or taken in turn when it is nullptr
  uint32_t* starts;         // lux_start_bytes(n_items)
  const uint32_t* firsts;   // batch: items whose segment is a multiple of kLuxGroup (nullptr: all are)
  uint32_t n_items, n_groups, warps, max_seg, tiles;
  int lgb;                  // segments of 2^lgb blocks; all of a stream when max_seg = 0
};
cudaError_t launch_lux_job(const LuxJob& job, int p, int mode, cudaStream_t s);
uint64_t lux_start_bytes(uint64_t items);

// The split on the current device.
LuxSplit lux_split(uint64_t warp_blocks, uint64_t longest);

// The tensor map of an output as a rows x pitch array of words in tiles of 32 x
// 32; false when it has none (unaligned, not this device's memory, more than 2^31 - 32
// words in a row or rows: lux_tiles_reach).
bool lux_out_map(void* out, uint64_t pitch, uint64_t rows, CUtensorMap* map);

}  // namespace prng
