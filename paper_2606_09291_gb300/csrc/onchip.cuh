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
  float *g4, *s4;                   // with MATRIX: the matrix [27 x 27], u and omega/D [2 x 27]
};
constexpr int kCoarse8Floats = 3 * 729 + 512 + 2 * 125 + 64 + 8;

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

// The V(1,1)-cycle from 4^3 down is a fixed linear map of the restricted residual r: with
// w = omega/D, p the interpolation of the 2^3 node to 4^3 (and its transpose the
// restriction), d the 2^3 diagonal and u = p - w A p,
//   z4 = w ((2 - omega) r + Off (w r)) + u (u . r) / d = G r   (A = D - Off),
// so the 27 x 27 matrix G is formed once per sample and every cycle is one product with it.
// Step by step the two levels were 4100 of the 12000 clocks of an 8^3 iteration: one warp's
// chain of two restrictions, three operator rows and three divisions.  Only the one-block
// solves use it: on grids of 32^3 and up its other rounding moves the results of the mixed
// path more (256^3: by 1e-7) than the passes' time gains.
// Needs a4, a2 (a barrier passed) and t4 = 0; the matrix is complete after the next barrier.
template <int CT>
__device__ __forceinline__ void coarse4_build(const CoarseLevels& L, float omega) {
  const int tid = threadIdx.x;
  constexpr float sc = float(1.0 / 48.0);
  const int I = 1 + tid % 3, J = 1 + (tid / 3) % 3, K = 1 + tid / 9, n = I + 5 * (J + 5 * K);
  const float p = ((I & 1) ? 0.5f : 1.f) * ((J & 1) ? 0.5f : 1.f) * ((K & 1) ? 0.5f : 1.f);
  if (tid < 27) L.t4[n] = p;
  __syncthreads();
  if (tid < 27) {
    Cells8<float, float> C;
    cells8(C, L.a4, I, J, K, 4);
    const float w = omega / (float(1.0 / 12.0) * C.sum);
    L.s4[27 + tid] = w;
    L.s4[tid] = p - w * (sc * q1_row(C, (const float*)L.t4, I, J, K, 5));
  }
  __syncthreads();
  if (tid < 27 * 27) {
    float s8 = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) s8 += L.a2[e];
    const float inv = 6.f / s8;
    for (int e = tid; e < 27 * 27; e += CT) {  // G[j][i]: a lane takes a row i
      const int i = e % 27, j = e / 27;
      const int xi = 1 + i % 3, yi = 1 + (i / 3) % 3, zi = 1 + i / 9;
      const int du = 1 + j % 3 - xi, dv = 1 + (j / 3) % 3 - yi, dw = 1 + j / 9 - zi;
      const float wi = L.s4[27 + i];
      float g = L.s4[i] * (L.s4[j] * inv);
      if (i == j) g = fmaf(wi, 2.f - omega, g);
      const int zeros = (du == 0) + (dv == 0) + (dw == 0);
      if (zeros <= 1 && abs(du) <= 1 && abs(dv) <= 1 && abs(dw) <= 1) {  // across a face or body diagonal
        const int c0 = (du > 0 ? xi : xi - 1) + 4 * ((dv > 0 ? yi : yi - 1) + 4 * (dw > 0 ? zi : zi - 1));
        float a = L.a4[c0];
        if (zeros) a += L.a4[c0 + (du == 0 ? 1 : dv == 0 ? 4 : 16)];
        g = fmaf(wi * (sc * a), L.s4[27 + j], g);
      }
      L.g4[e] = g;
    }
  }
}
// by one warp: restricts t8, leaves the 4^3 correction in L.t4
__device__ __forceinline__ void coarse4_matrix(const CoarseLevels& L) {
  const int lane = threadIdx.x & 31, row = lane < 27 ? lane : 26;
  const int I = 1 + row % 3, J = 1 + (row / 3) % 3, K = 1 + row / 9;
  const float* f = L.t8 + 2 * I + 9 * (2 * J) + 81 * (2 * K);
  float a[3];
#pragma unroll
  for (int w = -1; w <= 1; ++w) {
    float b[3];
#pragma unroll
    for (int u = -1; u <= 1; ++u) {
      const float* q = f + 9 * u + 81 * w;
      b[u + 1] = fmaf(0.5f, q[-1] + q[1], q[0]);
    }
    a[w + 1] = fmaf(0.5f, b[0] + b[2], b[1]);
  }
  const float r = fmaf(0.5f, a[0] + a[2], a[1]);
  float z[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < 27; ++j) z[j % 3] = fmaf(L.g4[27 * j + row], __shfl_sync(0xffffffffu, r, j), z[j % 3]);
  if (lane < 27) L.t4[I + 5 * (J + 5 * K)] = z[0] + (z[1] + z[2]);
}

// V-cycle from the 8^3 level; r8 is complete (barrier passed), z in L.t8 after the return
// of all threads and one more barrier.  own: this thread's node of the level; D its
// diagonal, or omega/D with MATRIX (4^3 and below as one matrix, see coarse4_build).
// Returns the correction at the own node.
template <int CT, bool MATRIX = false>
__device__ __forceinline__ float vcycle8(const CoarseLevels& L, int n, int i, int j, int k, bool in, float D,
                                         float omega) {
  constexpr float sc = float(1.0 / 96.0);
  const float r = n < 729 ? L.r8[n] : 0.f;
  if (in) L.x8[n] = MATRIX ? D * r : omega * r / D;
  __syncthreads();
  if (in) {
    Cells8<float, float> C;
    cells8(C, L.a8, i, j, k, 8);
    L.t8[n] = r - sc * q1_row(C, (const float*)L.x8, i, j, k, 9);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    if constexpr (MATRIX) coarse4_matrix(L);
    else coarse4(L, omega);
  }
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
    z = MATRIX ? fmaf(res, D, L.x8[n]) : L.x8[n] + omega * res / D;
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
