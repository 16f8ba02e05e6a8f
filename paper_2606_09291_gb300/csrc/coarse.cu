// coarse.cu - the coarse end of the V-cycle (rows a4, a6) in one launch: the levels
// 16^3, 8^3, 4^3 and 2^3 of a sample's hierarchy in the shared memory of one block.
//
// Below the fused fine-grid passes the V-cycle's levels are small (17^3 nodes and
// less): run level by level, each of the dozen steps (pre-smoothing and residual,
// restriction, the 2^3 solve, prolongation, post-smoothing, per level) is a launch
// whose grid is a few blocks per sample and whose time is mostly launch latency and
// tail.  Here one block per launched sample loads the restricted residual r and the
// four coefficient levels once, runs the whole V(1,1)-cycle below the 32^3 level with
// a block barrier between steps, and writes the correction z of the 16^3 level.
//
// The arithmetic is the V-cycle's (Sec. 5, the preconditioner of the PCG): at every
// level damped Jacobi with x0 = 0 (x = omega D^-1 r), the residual t = r - A x,
// restriction P^T t, recursion, x += P e, post-smoothing z = x + omega D^-1 (r - A x);
// on 2^3 the single interior unknown is solved exactly.  D = (h/3) sum_8 a: on the
// 16^3 level D^-1 is formed as the solver's D^-1 pass forms it (the four-cell sums of
// the planes below and above, then the reciprocal), on 8^3 and 4^3 the smoother
// divides by D as the level-by-level kernels do, and pre- and post-smoothing take
// the same D, so the preconditioner stays symmetric.  Boundary nodes hold 0 in every
// array.  The operator rows are those of the assembled Q1 stiffness (q1_row).
#include "internal.cuh"
#include "kernels.h"
#include "launch.h"
#include "levels.cuh"

namespace mlsgd {

namespace {

constexpr int kCT = 768;  // threads per block (24 warps: two blocks per SM hide the shared-memory latency)

// shared-memory layout (floats)
struct CoarseSmem {
  using L16 = Lv<16>;
  using L8 = Lv<8>;
  using L4 = Lv<4>;
  using L2 = Lv<2>;
  static constexpr int r16 = 0, x16 = r16 + L16::nodes, t16 = x16 + L16::nodes, d16 = t16 + L16::nodes,
                       a16 = d16 + L16::nodes;
  static constexpr int r8 = a16 + L16::cells, x8 = r8 + L8::nodes, t8 = x8 + L8::nodes, a8 = t8 + L8::nodes;
  static constexpr int r4 = a8 + L8::cells, x4 = r4 + L4::nodes, t4 = x4 + L4::nodes, a4 = t4 + L4::nodes;
  static constexpr int r2 = a4 + L4::cells, x2 = r2 + L2::nodes, a2 = x2 + L2::nodes;
  static constexpr int total = a2 + L2::cells;
  static constexpr size_t bytes = sizeof(float) * (size_t)total;
};

// asynchronous element copy into shared memory (the thread waits for its own copies, a block
// barrier then publishes them)
__device__ __forceinline__ void cp_async_elem(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(sizeof(float))
               : "memory");
}

struct CoarseArgs {
  const float* r;     // restricted residual on the 16^3 level, [S][17^3]
  const float* a[4];  // cell coefficient of the levels 16^3, 8^3, 4^3, 2^3, [S][cells]
  float* z;           // the V-cycle's correction on the 16^3 level, [S][17^3]
  const SolveScalars* sc;
  const int* act;
  float omega;
};

__global__ void __launch_bounds__(kCT, 2) k_coarse_vcycle(CoarseArgs A) {
  pdl_entry();
  using M = CoarseSmem;
  const int s = A.act != nullptr ? A.act[blockIdx.x] : (int)blockIdx.x;
  if (A.sc != nullptr && !A.sc[s].active) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  float* sm = reinterpret_cast<float*>(smraw);
  const float omega = A.omega;
  // r and the four coefficient levels, all copies in flight at once
  const float* rg = A.r + (long long)s * Lv<16>::nodes;
  for (int n = threadIdx.x; n < Lv<16>::nodes; n += kCT) cp_async_elem(sm + M::r16 + n, rg + n);
  const int aoff[4] = {M::a16, M::a8, M::a4, M::a2};
  const int acnt[4] = {Lv<16>::cells, Lv<8>::cells, Lv<4>::cells, Lv<2>::cells};
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const float* ag = A.a[l] + (long long)s * acnt[l];
    for (int n = threadIdx.x; n < acnt[l]; n += kCT) cp_async_elem(sm + aoff[l] + n, ag + n);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  dinv_level<kCT, float>(sm + M::a16, sm + M::d16);
  __syncthreads();
  // down: 16^3, 8^3, 4^3
  pre_level<kCT, 16, true, float>(sm + M::r16, sm + M::a16, sm + M::d16, sm + M::x16, sm + M::t16, omega);
  __syncthreads();
  restrict_level<kCT, 8, float>(sm + M::t16, sm + M::r8);
  __syncthreads();
  pre_level<kCT, 8, false, float>(sm + M::r8, sm + M::a8, nullptr, sm + M::x8, sm + M::t8, omega);
  __syncthreads();
  restrict_level<kCT, 4, float>(sm + M::t8, sm + M::r4);
  __syncthreads();
  pre_level<kCT, 4, false, float>(sm + M::r4, sm + M::a4, nullptr, sm + M::x4, sm + M::t4, omega);
  __syncthreads();
  restrict_level<kCT, 2, float>(sm + M::t4, sm + M::r2);
  __syncthreads();
  // 2^3: the single interior unknown (node 13), x = r / D
  for (int n = threadIdx.x; n < Lv<2>::nodes; n += kCT) {
    float v = 0.f;
    if (n == 13) {
      Cells8<float, float> C;
      cells8(C, sm + M::a2, 1, 1, 1, 2);
      v = sm[M::r2 + 13] / (float(1.0 / 6.0) * C.sum);
    }
    sm[M::x2 + n] = v;
  }
  __syncthreads();
  // up: 4^3, 8^3 (the smoothed corrections overwrite the dead residuals t), then 16^3
  prolong_level<kCT, 4, float>(sm + M::x4, sm + M::x2);
  __syncthreads();
  post_level<kCT, 4, false, float>(sm + M::r4, sm + M::a4, nullptr, sm + M::x4, sm + M::t4, omega);
  __syncthreads();
  prolong_level<kCT, 8, float>(sm + M::x8, sm + M::t4);
  __syncthreads();
  post_level<kCT, 8, false, float>(sm + M::r8, sm + M::a8, nullptr, sm + M::x8, sm + M::t8, omega);
  __syncthreads();
  prolong_level<kCT, 16, float>(sm + M::x16, sm + M::t8);
  __syncthreads();
  post_level<kCT, 16, true, float>(sm + M::r16, sm + M::a16, sm + M::d16, sm + M::x16,
                          A.z + (long long)s * Lv<16>::nodes, omega);
}

}  // namespace

bool coarse_vcycle_applies(int N, int j) { return j >= 1 && (N >> j) == 16; }

void coarse_vcycle(const float* r16, const float* const a[4], float* z16, const SolveScalars* sc, const Batch& bt,
                   double omega, cudaStream_t st) {
  using M = CoarseSmem;
  static SmemOptIn opt_in;
  (void)opt_in(k_coarse_vcycle, M::bytes);  // a launch without it is refused
  CoarseArgs A{};
  A.r = r16;
  for (int l = 0; l < 4; ++l) A.a[l] = a[l];
  A.z = z16;
  A.sc = sc;
  A.act = bt.act;
  A.omega = (float)omega;
  // per sample: r and z on 17^3 nodes, the four coefficient levels
  const double bytes = (double)bt.n * sizeof(float) *
                       (2.0 * Lv<16>::nodes + Lv<16>::cells + Lv<8>::cells + Lv<4>::cells + Lv<2>::cells);
  launch("coarse_f32", bytes, k_coarse_vcycle, dim3((unsigned)bt.n), dim3(kCT), M::bytes, st, A);
}

}  // namespace mlsgd
