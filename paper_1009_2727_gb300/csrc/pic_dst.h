// Device destinations of the field accessors: memory that the caller owns and that a context's stream writes.
#pragma once

#include <cuda_runtime.h>

namespace picgb {

class DeviceDst {
 public:
  ~DeviceDst() {
    if (ready) cudaEventDestroy(ready);
  }
  // Work queued on s from here on starts after the work already queued on the default stream, where the caller's earlier
  // use of the destination may still run (memory that an allocator hands out again in stream order). False: no event.
  bool order(cudaStream_t s) {
    if (!s) return true;
    if (!ready && cudaEventCreateWithFlags(&ready, cudaEventDisableTiming) != cudaSuccess) return false;
    return cudaEventRecord(ready, nullptr) == cudaSuccess && cudaStreamWaitEvent(s, ready, 0) == cudaSuccess;
  }

 private:
  cudaEvent_t ready = nullptr;
};

}  // namespace picgb
