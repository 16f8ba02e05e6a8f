// launch.h - every kernel launch of libmlsgd goes through launch(): it counts the
// launch and, when profiling is enabled for the kernel's class, brackets it with
// CUDA events on the launching stream and accumulates its algorithmic bytes
// (each input read once, each output written once).
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace mlsgd {

void prof_begin(const char* cls, cudaStream_t st);
void prof_end(const char* cls, cudaStream_t st, double bytes, double flops);

// Launches `kern` in clusters of `cluster` consecutive blocks (0: none), as a
// programmatic dependent of the work before it in the stream: its blocks may start while
// the kernel before drains (every kernel begins with pdl_entry, which waits for it).
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
