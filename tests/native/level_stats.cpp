// level_stats.cpp - launch_level_stats on a caller's device arrays, for tests of the statistics
// kernels with chosen nodal values.
#include <cuda_runtime.h>

#include "kernels.h"

extern "C" int level_stats(const double* qf, const double* phif, int Nf, const double* qc, const double* phic, int S, int Nc,
                           double theta, double* field, double* scalars, int qf_pairs, int qc_pairs) {
  double *work, *partial, *nodes;
  if (cudaMalloc(&work, (4 + 4 * (size_t)S) * 8) != cudaSuccess ||
      cudaMalloc(&partial, mlsgd::level_partial_cap(Nc, Nf) * 8) != cudaSuccess ||
      cudaMalloc(&nodes, mlsgd::nodes_of(Nf) * 8) != cudaSuccess)
    return 1;
  mlsgd::launch_level_stats(qf, phif, Nf, qc, phic, Nf / 2, S, Nc, theta, field, scalars, work, partial, nullptr, nullptr,
                            nullptr, qf_pairs != 0, qc_pairs != 0, nodes);
  const cudaError_t e = cudaDeviceSynchronize();
  cudaFree(work);
  cudaFree(partial);
  cudaFree(nodes);
  return e == cudaSuccess ? 0 : 2;
}
