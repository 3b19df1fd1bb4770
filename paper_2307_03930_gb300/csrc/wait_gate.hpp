// Bounded waits of one role of a kernel, one after another.  No CUDA headers:
// the tests compile it for the host alone.
#pragma once

#ifdef __CUDACC__
#define ROSKO_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define ROSKO_HOST_DEVICE inline
#endif

namespace rosko {

// Once a wait has run out its role waits for nothing more: an error return
// takes one limit, however many waits the role still had before it.
struct WaitGate {
  bool open = true;
  template <class Wait>
  ROSKO_HOST_DEVICE bool operator()(Wait wait) {
    if (open) open = wait();
    return open;
  }
};

}  // namespace rosko
