// Two chains of launches that meet at the end.
#pragma once

#include <cuda_runtime_api.h>

// Runs body, which puts work on the caller's stream st and, between its own events, on
// `side`, and which waits for the side's work on st before it ends well.  Where it ends in an
// error it may be between the two: what the side has begun still writes the call's buffers, so
// st waits for it here (event `done`), or this thread does.
template <class Body>
cudaError_t run_with_side(cudaStream_t st, cudaStream_t side, cudaEvent_t done, Body body) {
  const cudaError_t e = body();
  if (e != cudaSuccess &&
      (cudaEventRecord(done, side) != cudaSuccess || cudaStreamWaitEvent(st, done, 0) != cudaSuccess))
    cudaStreamSynchronize(side);
  return e;
}
