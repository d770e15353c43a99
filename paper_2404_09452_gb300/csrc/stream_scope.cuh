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

// Work on `side` beside `st` (nothing to do where they are the same): fork() makes `side`
// wait for what `st` has so far, join() makes `st` wait for `side`.  A fork that an
// error leaves open is joined at the scope's end: what `side` still writes (J, in the
// caller's memory) is then in order before anything the caller queues on `st`.
class SideScope {
  cudaStream_t st, side;
  cudaEvent_t ev_fork, ev_join;
  bool open = false;

 public:
  SideScope(cudaStream_t st, cudaStream_t side, cudaEvent_t ev_fork, cudaEvent_t ev_join)
      : st(st), side(side), ev_fork(ev_fork), ev_join(ev_join) {}
  void fork() {
    if (side == st) return;
    DFJK_CUDA_CHECK(cudaEventRecord(ev_fork, st));
    DFJK_CUDA_CHECK(cudaStreamWaitEvent(side, ev_fork, 0));
    open = true;
  }
  void join() {
    if (!open) return;
    DFJK_CUDA_CHECK(cudaEventRecord(ev_join, side));
    DFJK_CUDA_CHECK(cudaStreamWaitEvent(st, ev_join, 0));
    open = false;
  }
  ~SideScope() {
    if (!open) return;
    cudaEventRecord(ev_join, side);
    cudaStreamWaitEvent(st, ev_join, 0);
  }
};

}  // namespace dfjk
