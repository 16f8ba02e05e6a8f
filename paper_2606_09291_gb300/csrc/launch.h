// launch.h - every kernel launch of libmlsgd goes through launch(): it counts the
// launch and, when profiling is enabled for the kernel's class, brackets it with
// CUDA events on the launching stream and accumulates its algorithmic bytes
// (each input read once, each output written once).
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>
#include <utility>

namespace mlsgd {

void prof_begin(const char* cls, cudaStream_t st);
void prof_end(const char* cls, cudaStream_t st, double bytes, double flops);

// A kernel's opt-in to more dynamic shared memory than the default: once per device (and
// again when a call needs more, never to less), from any thread; no call on every enqueue.
// A refusal is returned and tried again by the next call.
struct SmemOptIn {
  static constexpr int kDevices = 64;
  std::atomic<int> bytes[kDevices];  // static storage: 0
  std::mutex m;
  template <typename... KArgs>
  cudaError_t operator()(void (*kern)(KArgs...), size_t need, bool carveout = false) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kDevices) return cudaErrorInvalidDevice;
    if (bytes[dev].load(std::memory_order_acquire) >= (int)need) return cudaSuccess;
    std::lock_guard<std::mutex> lock(m);
    if (bytes[dev].load(std::memory_order_relaxed) >= (int)need) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
    if (e == cudaSuccess && carveout)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) bytes[dev].store((int)need, std::memory_order_release);
    return e;
  }
};

// Launches `kern` in clusters of `cluster` consecutive blocks (0: none), as a
// programmatic dependent of the work before it in the stream: its blocks may start while
// the kernel before drains (every kernel begins with pdl_entry or pdl_wait, which wait for it).
// !early: not before that kernel has ended (a kernel whose time is that of the fullest SM
// wants its blocks spread over idle SMs, not placed where the kernel before leaves room).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 unsigned cluster, bool early, Args&&... args) {
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = cluster ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
inline void launch_flops(const char* cls, double bytes, double flops, void (*kern)(KArgs...), dim3 grid, dim3 block,
                         size_t smem, cudaStream_t st, Args&&... args) {
  prof_begin(cls, st);
  (void)launch_kernel(kern, grid, block, smem, st, 0, true, std::forward<Args>(args)...);  // checked by the callers
  prof_end(cls, st, bytes, flops);
}

template <typename... KArgs, typename... Args>
inline void launch(const char* cls, double bytes, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                   cudaStream_t st, Args&&... args) {
  launch_flops(cls, bytes, 0.0, kern, grid, block, smem, st, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
inline void launch_after(const char* cls, double bytes, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                         cudaStream_t st, Args&&... args) {
  prof_begin(cls, st);
  (void)launch_kernel(kern, grid, block, smem, st, 0, false, std::forward<Args>(args)...);  // checked by the callers
  prof_end(cls, st, bytes, 0.0);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_cluster(const char* cls, double bytes, void (*kern)(KArgs...), dim3 grid, dim3 block,
                                  unsigned cluster, size_t smem, cudaStream_t st, Args&&... args) {
  prof_begin(cls, st);
  const cudaError_t e = launch_kernel(kern, grid, block, smem, st, cluster, true, std::forward<Args>(args)...);
  prof_end(cls, st, bytes, 0.0);
  return e;
}

}  // namespace mlsgd
