// ranlux_tc.cuh -- entry points of the tensor-core RANLUX fill (k_ranlux_tc.cu).
#pragma once

#include "ranlux.cuh"

namespace prng {

// Lowest luxury p that the tensor-core form serves: its state of a fill that
// ends inside a block needs at least 24 discarded steps per cycle (p >= 48), and
// below p = 97 the borrow chain costs less than the carries of the product.
constexpr int kLuxTcMinP = 97;

// Fill the multiplier operands of the current device (idempotent; called when a
// RANLUX handle is created, before any of its fills).
cudaError_t lux_tables_init();

// Whether a kernel on the current device ever gave up waiting for its tensor
// core (its handle's state is then not the one after the fill).  Synchronises.
bool lux_tc_stuck();

// The launch tile of a plain fill that leaves it to the library.
Tile ranlux_auto_tile(const FillDesc& d);

cudaError_t launch_fill_ranlux_tc(const FillDesc& d, cudaStream_t s);

}  // namespace prng
