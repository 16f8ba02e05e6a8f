// onchip.cuh - pieces shared by the solves that keep a sample on chip (small.cu,
// cluster32.cu): the V-cycle from an 8^3 level down and the scalar updates.
#pragma once
#include "internal.cuh"
#include "kernels.h"
#include "levels.cuh"

namespace mlsgd {

// The refinement loop's per-sample state, held by lane 0 of warp 0.
struct Outer {
  double bb, rr, rz;
  int iters, status, pad;
};

// x = 8^3 level and below: the V(1,1)-cycle with the level's residual r8 in shared memory,
// correction left in z8 (block of CT threads, thread n < 729 owns node n of the level).
// The levels 4^3 and 2^3 (27 and 1 interior nodes) are one warp's work.
struct CoarseLevels {
  float *r8, *x8, *t8;              // [729]; t8 also receives the correction
  const float* a8;                  // [512]
  float *x4, *t4;                   // [125]
  const float *a4, *a2;             // [64], [8]
};
constexpr int kCoarse8Floats = 3 * 729 + 512 + 2 * 125 + 64 + 8;
constexpr int kCoarse8Own = 2 * 729 + 2 * 125 + 64 + 8;  // without r8 and a8

template <int N>
__device__ __forceinline__ float diag_of(const float* a, int i, int j, int k) {  // D = (h/3) sum_8 a
  Cells8<float, float> C;
  cells8(C, a, i, j, k, N);
  return float(1.0 / (3.0 * N)) * C.sum;
}

// levels 4^3 and 2^3 by one warp: restricts t8, leaves the 4^3 correction in L.t4
__device__ __forceinline__ void coarse4(const CoarseLevels& L, float omega) {
  const int lane = threadIdx.x & 31;
  const int I = 1 + lane % 3, J = 1 + (lane / 3) % 3, K = 1 + lane / 9;  // lane < 27
  const int n = I + 5 * (J + 5 * K);
  const bool own = lane < 27;
  float r = 0.f, D = 1.f;
  if (own) {
    const float* f = L.t8 + 2 * I + 9 * (2 * J) + 81 * (2 * K);
    float v = 0.f;
#pragma unroll
    for (int w = -1; w <= 1; ++w)
#pragma unroll
      for (int u = -1; u <= 1; ++u)
#pragma unroll
        for (int q = -1; q <= 1; ++q) {
          const float wt = float((q == 0 ? 1.0 : 0.5) * (u == 0 ? 1.0 : 0.5) * (w == 0 ? 1.0 : 0.5));
          v += wt * f[q + 9 * u + 81 * w];
        }
    r = v;
    D = diag_of<4>(L.a4, I, J, K);
    L.x4[n] = omega * r / D;
  }
  __syncwarp();
  Cells8<float, float> C;
  if (own) {
    cells8(C, L.a4, I, J, K, 4);
    L.t4[n] = r - float(1.0 / 48.0) * q1_row(C, (const float*)L.x4, I, J, K, 5);
  }
  __syncwarp();
  // restriction to the single unknown of 2^3 and its exact solution (every lane the same)
  float e2;
  {
    const float* f = L.t4 + 62;
    float v = 0.f;
#pragma unroll
    for (int w = -1; w <= 1; ++w)
#pragma unroll
      for (int u = -1; u <= 1; ++u)
#pragma unroll
        for (int q = -1; q <= 1; ++q) {
          const float wt = float((q == 0 ? 1.0 : 0.5) * (u == 0 ? 1.0 : 0.5) * (w == 0 ? 1.0 : 0.5));
          v += wt * f[q + 5 * u + 25 * w];
        }
    Cells8<float, float> C2;
    cells8(C2, L.a2, 1, 1, 1, 2);
    e2 = v / (float(1.0 / 6.0) * C2.sum);
  }
  if (own) {  // trilinear: the one coarse node, weight 1/2 per odd index (I, J, K in 1..3)
    const float w = ((I & 1) ? 0.5f : 1.f) * ((J & 1) ? 0.5f : 1.f) * ((K & 1) ? 0.5f : 1.f);
    L.x4[n] += w * e2;
  }
  __syncwarp();
  if (own) {
    const float res = r - float(1.0 / 48.0) * q1_row(C, (const float*)L.x4, I, J, K, 5);
    L.t4[n] = L.x4[n] + omega * res / D;
  }
}

// V-cycle from the 8^3 level; r8 is complete (barrier passed), z in L.t8 after the return
// of all threads and one more barrier.  own: this thread's node of the level; D its
// diagonal.  Returns the correction at the own node.
template <int CT>
__device__ __forceinline__ float vcycle8(const CoarseLevels& L, int n, int i, int j, int k, bool in, float D,
                                         float omega) {
  constexpr float sc = float(1.0 / 96.0);
  const float r = n < 729 ? L.r8[n] : 0.f;
  if (in) L.x8[n] = omega * r / D;
  __syncthreads();
  if (in) {
    Cells8<float, float> C;
    cells8(C, L.a8, i, j, k, 8);
    L.t8[n] = r - sc * q1_row(C, (const float*)L.x8, i, j, k, 9);
  }
  __syncthreads();
  if (threadIdx.x < 32) coarse4(L, omega);
  __syncthreads();
  if (in) {
    const int i0 = i >> 1, j0 = j >> 1, k0 = k >> 1;
    const int i1 = i0 + (i & 1), j1 = j0 + (j & 1), k1 = k0 + (k & 1);
    const float wi = (i & 1) ? 0.5f : 1.f, wj = (j & 1) ? 0.5f : 1.f, wk = (k & 1) ? 0.5f : 1.f;
    const float* ec = L.t4;
    auto at = [&](int a, int b, int c) { return ec[a + 5 * b + 25 * c]; };
    float v;
    if ((i & 1) == 0 && (j & 1) == 0 && (k & 1) == 0) {
      v = at(i0, j0, k0);
    } else {
      v = wi * wj * wk *
          (at(i0, j0, k0) + ((i & 1) ? at(i1, j0, k0) : 0.f) + ((j & 1) ? at(i0, j1, k0) : 0.f) +
           ((k & 1) ? at(i0, j0, k1) : 0.f) + (((i & 1) && (j & 1)) ? at(i1, j1, k0) : 0.f) +
           (((i & 1) && (k & 1)) ? at(i1, j0, k1) : 0.f) + (((j & 1) && (k & 1)) ? at(i0, j1, k1) : 0.f) +
           (((i & 1) && (j & 1) && (k & 1)) ? at(i1, j1, k1) : 0.f));
    }
    L.x8[n] += v;
  }
  __syncthreads();
  float z = 0.f;
  if (in) {
    Cells8<float, float> C;
    cells8(C, L.a8, i, j, k, 8);
    const float res = r - sc * q1_row(C, (const float*)L.x8, i, j, k, 9);
    z = L.x8[n] + omega * res / D;
    L.t8[n] = z;
  }
  return z;
}

// scalar updates of the PCG (see SM_ALPHA, SM_BETA in solver.cu)
__device__ __forceinline__ float pcg_alpha(const Outer& o, double v) {
  return (float)((v > 0.0 && o.rz != 0.0) ? o.rz / v : 0.0);
}
__device__ __forceinline__ float pcg_beta(Outer& o, double v) {
  const double b = o.rz != 0.0 ? v / o.rz : 0.0;
  o.rz = v;
  return (float)b;
}
// the refinement's stop test (SM_OUTER_CONV): true while the sample goes on
__device__ __forceinline__ bool outer_go(Outer& o, double v, double tol2, int cap) {
  o.rr = v;
  if (v <= tol2 * o.bb) return false;
  if (!(v < INFINITY)) { o.status = 2; return false; }
  if (o.iters >= cap) { o.status = 1; return false; }
  return true;
}
__device__ __forceinline__ void store_scalars(SolveScalars* sc, const Outer& o) {
  SolveScalars c;
  c.bb = o.bb; c.rz = o.rz; c.alpha = 0.0; c.beta = 0.0; c.rr = o.rr;
  c.active = 0; c.iters = o.iters; c.status = o.status; c.pad = o.pad;
  *sc = c;
}

}  // namespace mlsgd
