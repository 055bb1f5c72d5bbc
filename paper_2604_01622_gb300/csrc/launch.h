// The stream of a call and how its kernels are launched on it. Internal.
#pragma once
#include <cuda_runtime.h>

namespace ecmoe {

// SMs of a GB300, for caps on grids and for splits whose summands lie in the workspace: its size
// is asked for before any call, also where there is no device, so it cannot come from one.
constexpr int kSms = 152;

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
