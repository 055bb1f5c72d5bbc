// The stream of a call and how its kernels are launched on it. Internal.
#pragma once
#include <cuda_runtime.h>

namespace ecmoe {

// overlap: launch each kernel with programmatic stream serialisation, so that its CTAs start
// while the kernel before it finishes (see pdl_begin in common.cuh). Converts to and from a plain
// stream (no overlap).
struct LaunchStream {
  cudaStream_t s;
  bool overlap;
  LaunchStream(cudaStream_t st, bool o = false) : s(st), overlap(o) {}
  operator cudaStream_t() const { return s; }
};

}  // namespace ecmoe
