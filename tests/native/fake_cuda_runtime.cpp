// fake_cuda_runtime.cpp - the CUDA runtime calls that the library makes, on host memory and
// without a GPU, for tests of the code that prepares and launches the kernels: no kernel
// runs, every launch is checked as the runtime checks it and recorded, and a call can be
// made to fail.  Linked with the library's object files in place of libcudart.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <utility>
#include <vector>

#include "kernels.h"
#include "mlsgd.h"

namespace {
struct Launch {
  std::string name;
  unsigned v[8];  // grid, block, dynamic shared memory, device
};
struct State {
  std::map<const void*, std::string> names;
  std::map<std::pair<const void*, int>, int> smem;  // opt-in per kernel and device
  std::vector<Launch> launches;
  std::string fail;     // kernels whose opt-in is refused
  bool no_occupancy = false;
  int device = 0;
  cudaError_t last = cudaSuccess;
};
State& S() {
  static State* s = new State;  // kernels register before this file's own statics exist
  return *s;
}
cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) S().last = e;
  return e;
}
cudaError_t record(const void* f, dim3 g, dim3 b, size_t smem) {
  const auto it = S().names.find(f);
  if (it == S().names.end()) return set(cudaErrorInvalidDeviceFunction);
  if (g.x < 1 || g.x > 0x7fffffffu || g.y < 1 || g.y > 65535u || g.z < 1 || g.z > 65535u || b.x * b.y * b.z < 1 ||
      b.x * b.y * b.z > 1024)
    return set(cudaErrorInvalidConfiguration);
  const auto o = S().smem.find({f, S().device});
  if (smem > 48 * 1024 && (o == S().smem.end() || smem > (size_t)o->second)) return set(cudaErrorInvalidValue);
  S().launches.push_back({it->second, {g.x, g.y, g.z, b.x, b.y, b.z, (unsigned)smem, (unsigned)S().device}});
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- for the tests
int fake_launches() { return (int)S().launches.size(); }
const char* fake_launch(int i, unsigned v[8]) {
  memcpy(v, S().launches[i].v, sizeof(Launch::v));
  return S().launches[i].name.c_str();
}
void fake_reset() { S().launches.clear(); }
void fake_refuse_opt_in(const char* kernel) { S().fail = kernel; }
void fake_refuse_occupancy(int on) { S().no_occupancy = on != 0; }
void fake_set_last_error(int e) { S().last = (cudaError_t)e; }
// 0 when the vectors of a solve on an N^3 grid lie side by side within solver_bytes
int fake_check_carve(int N, int S, int elem) {
  mlsgd::SolverBufs B;
  char* const base = (char*)4096;
  char* p = base;
  mlsgd::carve_solver(B, N, S, elem, p);
  if (p < base || (size_t)(p - base) > mlsgd::solver_bytes(N, S, elem)) return 1;
  std::vector<std::pair<char*, size_t>> v;
  const auto add = [&](void* q, long long n) { if (q) v.push_back({(char*)q, (size_t)n}); };
  const size_t e = (size_t)elem * S;
  for (void* q : {B.x, B.r, B.r2, B.p, B.q}) add(q, e * mlsgd::nodes_of(N));
  for (int j = 0; j <= B.J; ++j) {
    const int M = N >> j;
    for (void* q : {B.vx[j], B.vt[j], B.vr[j], B.dinv[j]}) add(q, e * mlsgd::nodes_of(M));
    add(B.acoef[j], e * mlsgd::cells_of(M));
  }
  std::sort(v.begin(), v.end());
  for (size_t i = 0; i < v.size(); ++i) {
    char* const end = i + 1 < v.size() ? v[i + 1].first : (char*)B.partial;
    if (v[i].first < base || v[i].first + v[i].second > end) return 2;
  }
  return 0;
}
long long fake_level_partial_cap(int Nc, int Nf) { return mlsgd::level_partial_cap(Nc, Nf); }

// ---- the runtime
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  S().names[host] = name;
}
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaErrorUnknown; }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaErrorUnknown; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return record(f, c->gridDim, c->blockDim, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (!S().fail.empty() && S().names[f].find(S().fail) != std::string::npos) return set(cudaErrorInvalidValue);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) S().smem[{f, S().device}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  if (S().no_occupancy) return set(cudaErrorUnknown);
  *n = 16;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(1, n); return *p ? cudaSuccess : set(cudaErrorMemoryAllocation); }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = S().device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { S().device = d; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = S().last; S().last = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError() { return S().last; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static char* a = (char*)calloc(1, MLSGD_NOALLOC_SCRATCH_BYTES);
  *p = a;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* r) {
  *f = nullptr;
  if (r) *r = cudaDriverEntryPointSymbolNotFound;
  return set(cudaErrorSymbolNotFound);
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}
