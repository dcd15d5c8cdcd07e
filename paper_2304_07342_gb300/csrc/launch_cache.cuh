// launch_cache.cuh -- per-device cache of a kernel's launch shape: the
// dynamic shared-memory opt-in and the resident blocks per SM.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>

namespace glz {

// Launch-shape cache for one kernel instance, one entry per device: the
// shared-memory opt-in (cudaFuncSetAttribute acts on the current device's
// context only), which is only ever raised -- another thread may be about to
// launch the instance with the larger size -- and the resident blocks of the
// last few shapes.
constexpr int kMaxDevices = 64;
constexpr int kShapes = 4;

struct LaunchCache {
  struct Shape {
    int block = -1, per_sm = 0;
    size_t smem = 0;
  };
  struct Entry {
    int sms = 0, next = 0;
    size_t granted = 0;
    Shape shapes[kShapes];
  };
  std::mutex mu;
  Entry dev[kMaxDevices];
};

// Blocks of `kern` resident per SM on the current device for this block and
// smem size.
template <typename K>
static cudaError_t resident_blocks(LaunchCache &lc, K kern, int block,
                                   size_t smem, int *per_sm, int *sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(lc.mu);
  LaunchCache::Entry &c = lc.dev[dev];
  for (const LaunchCache::Shape &s : c.shapes)
    if (s.block == block && s.smem == smem) {
      *per_sm = s.per_sm;
      *sms = c.sms;
      return cudaSuccess;
    }
  if (smem > c.granted) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    c.granted = smem;
  }
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, block, smem);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  LaunchCache::Shape &s = c.shapes[c.next];
  c.next = (c.next + 1) % kShapes;
  s.block = block;
  s.smem = smem;
  s.per_sm = *per_sm;
  c.sms = *sms;
  return cudaSuccess;
}

// Launch that may begin while the kernel before it on the stream still runs
// (programmatic dependent launch): the kernel waits for that one itself
// (grid_wait) before it touches anything of it.
template <typename K, typename... Args>
static cudaError_t launch_dependent(K kern, unsigned grid, int block, size_t smem,
                                    cudaStream_t stream, const Args &...args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace glz
