// Shared device helpers of the EC-MoE library (sm_103a).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <utility>

#include "launch.h"

namespace ecmoe {

// Device status word codes (first word of the workspace).
// DEV_BAD_CAPACITY: a capacity update read from device memory was rejected (the previous
// capacities stay in force).
enum : int { DEV_OK = 0, DEV_TIMEOUT = 1, DEV_BAD_CAPACITY = 2 };

// Element type tags.
typedef __nv_bfloat16 bf16;

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<bf16>(bf16 v) { return __bfloat162float(v); }

template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f32<bf16>(float v) { return __float2bfloat16_rn(v); }

// 16-byte vector of T: 4 floats or 8 bf16.
template <typename T> struct Vec16 { static constexpr int n = 16 / sizeof(T); };

__device__ __forceinline__ void unpack16(const uint4& u, float* f, float) {
  f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y);
  f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
}
__device__ __forceinline__ void unpack16(const uint4& u, float* f, bf16) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ uint4 pack16(const float* f, float) {
  return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]),
                    __float_as_uint(f[3]));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ uint4 pack16(const float* f, bf16) {
  return make_uint4(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3]), pack_bf16x2(f[4], f[5]),
                    pack_bf16x2(f[6], f[7]));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------------------ overlapped launches
// Small calls launch every kernel with programmatic stream serialisation (LaunchStream::overlap):
// its CTAs may start while the kernel before it still runs, and each waits in pdl_begin for that
// kernel's end (and its memory) before it touches global memory. Only what comes before
// pdl_begin overlaps: the launch itself, barrier and TMEM set-up, tensor-map fetches. The next
// kernel is let in after the wait, so when a kernel starts, everything before its predecessor has
// completed. Launched without it, both instructions do nothing.
// The pointers named in pdl_begin come out of an opaque step behind the wait, so no load through
// them, read-only loads included, can be moved above it.
template <typename P>
__device__ __forceinline__ P* after_wait(P* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}
template <typename... P>
__device__ __forceinline__ void pdl_begin(P&... ptrs) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  (([&] { asm volatile("" : "+l"(ptrs)::"memory"); }()), ...);
}

template <typename... K, typename... A>
cudaError_t launch_kernel(void (*kern)(K...), dim3 grid, dim3 block, size_t smem, LaunchStream st,
                          int cluster, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  unsigned n = 0;
  if (st.overlap) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = (unsigned)cluster;
    at[n].val.clusterDim.y = 1;
    at[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

// silu(a) = a * sigmoid(a); sigmoid evaluated with the CUDA math library's expf.
__device__ __forceinline__ float sigmoidf_(float a) { return 1.0f / (1.0f + expf(-a)); }

}  // namespace ecmoe
