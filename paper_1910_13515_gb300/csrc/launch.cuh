// launch.cuh -- launches of the kernels that solve (host side): their workspace
// is above the 48 KiB of dynamic shared memory a kernel may use without asking,
// so the first launch of each on a device raises its limit.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace lbm39 {

// The limit is a property of the function on a device; setting it twice (two
// threads at once) is harmless.  False where the runtime refuses.
template <auto Kernel>
bool allow_shared(size_t bytes) {
  static std::atomic<unsigned long long> done[4];  // one bit per device
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  const bool known = dev >= 0 && dev < 256;
  if (known && (done[dev >> 6].load(std::memory_order_relaxed) >> (dev & 63) & 1)) return true;
  if (cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) !=
      cudaSuccess)
    return false;
  if (known) done[dev >> 6].fetch_or(1ull << (dev & 63), std::memory_order_relaxed);
  return true;
}

// On a refusal the launch itself fails and leaves its error to the caller's check.
template <auto Kernel, class... Args>
void launch_ws(unsigned grid, int blk, size_t bytes, cudaStream_t stream, Args... args) {
  allow_shared<Kernel>(bytes);
  Kernel<<<grid, blk, bytes, stream>>>(args...);
}

// The same for a kernel that calls cudaGridDependencySynchronize before it touches what another has
// written: its blocks are set up while the kernel before it on the stream ends.  With the step's two
// kernels launched so, 20 steps of a 105 x 105 lattice take 0.91 ms; with only the second 0.96, and
// 0.92 where the step was one kernel.
template <auto Kernel, class... Args>
void launch_ws_early(unsigned grid, int blk, size_t bytes, cudaStream_t stream, Args... args) {
  allow_shared<Kernel>(bytes);
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = blk;
  c.dynamicSmemBytes = bytes;
  c.stream = stream;
  c.attrs = &a;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, Kernel, args...);
}

}  // namespace lbm39
