// Early starts of dependent kernels (programmatic stream serialization), and
// launch parameters that belong to a device.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace gsr {

// A positive number per device, made at the first use there. cudaFuncSetAttribute
// and the occupancy queries act on the current device, so what they set or return
// is not another device's. Threads whose first uses coincide each make it, and
// store the same.
class PerDevice {
 public:
  template <typename F>
  int get(F make) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return make();
    int x = v_[dev].load(std::memory_order_acquire);
    if (x == 0) {
      x = make();
      v_[dev].store(x, std::memory_order_release);
    }
    return x;
  }

 private:
  static constexpr int kDevices = 64;  // above: made at every use
  std::atomic<int> v_[kDevices] = {};
};

// A kernel launched by launch_dependent may start (its blocks become resident)
// before the kernel in front of it on the stream has ended, once all blocks of
// that one have called pdl_trigger or exited; it calls pdl_wait before anything
// else, which returns when that kernel has completed. So the launch and the
// block scheduling of one kernel of a chain hide behind the last blocks of the
// kernel before. Without `early` it is an ordinary launch. Every kernel launched
// this way waits on every path, so the completion of one implies that of all
// kernels before it.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
cudaError_t launch_dependent(bool early, void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st,
                             A... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
cudaError_t launch_dependent(bool early, void (*kernel)(P...), int grid, int block, cudaStream_t st, A... args) {
  return launch_dependent(early, kernel, dim3((unsigned)grid), block, (size_t)0, st, args...);
}

}  // namespace gsr
