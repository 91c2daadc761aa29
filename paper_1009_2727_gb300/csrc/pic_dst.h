// Device destinations of the field accessors: memory that the caller owns and that a context's stream writes.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace picgb {

// May a kernel on `device` write doubles at p? Only where p is that device's own memory and aligned to them. Everything
// else that a copy reaches (another GPU's memory without a peer mapping, managed or pinned host memory, an odd address) or
// refuses (pageable host memory) is left to a copy from the context's scratch.
inline bool writable_in_place(const void* p, const cudaPointerAttributes& a, int device) {
  return a.type == cudaMemoryTypeDevice && a.device == device && reinterpret_cast<uintptr_t>(p) % sizeof(double) == 0;
}

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

  static bool in_place(const void* p) {
    cudaPointerAttributes a{};
    int dev = -1;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaPointerGetAttributes(&a, p) == cudaSuccess)
      return writable_in_place(p, a, dev);
    cudaGetLastError();   // (a pointer that CUDA does not know is for the copy to refuse)
    return false;
  }

 private:
  cudaEvent_t ready = nullptr;
};

}  // namespace picgb
