// Scopes that keep streams in step when an error passes through.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace dfjk {

// Waits for a stream (0, the legacy default stream, included) on scope exit, error paths
// included, so that buffers the stream still uses are not returned to the cache under it:
// declared after them.
struct StreamDrain {
  cudaStream_t s;
  ~StreamDrain() { cudaStreamSynchronize(s); }
};

}  // namespace dfjk
