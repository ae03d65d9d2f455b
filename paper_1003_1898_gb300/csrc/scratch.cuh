// scratch.cuh -- stream-ordered scratch (the jump fills' chunk starts, the
// segments' starts of XOR128 and RANLUX fills), from a memory pool the library
// creates once per device and that keeps up to 1 GiB for reuse (the device's
// default pool would hand freed memory back at every synchronisation, so that
// each call allocated afresh).
#pragma once

#include <cstddef>
#include <cuda_runtime.h>

namespace prng {

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s);
cudaError_t scratch_free(void* p, cudaStream_t s);

// Whether the stream is being captured: a plain fill takes no scratch then, so
// that it stays a sequence of kernel nodes.
inline bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
    cudaGetLastError();
    return true;
  }
  return st != cudaStreamCaptureStatusNone;
}

}  // namespace prng
