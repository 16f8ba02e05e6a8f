// levels.cuh - the steps of a V(1,1)-cycle on small levels held in the shared memory of
// one block of CT threads (used by the fused coarse V-cycle and by the one-block solves).
// Boundary nodes hold 0 in every array; the operator rows are those of the assembled Q1
// stiffness (q1_row).
#pragma once
#include "internal.cuh"
#include "kernels.h"

namespace mlsgd {

template <int N>
struct Lv {
  static constexpr int n1 = N + 1, nodes = n1 * n1 * n1, cells = N * N * N;
};

// the eight cells around interior node (i, j, k) of an N^3 level held in shared memory
template <typename T>
__device__ __forceinline__ void cells8(Cells8<T, T>& C, const T* a, int i, int j, int k, int N) {
  C.sum = T(0);
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const T v = a[(i - 1 + p) + N * ((j - 1 + q) + N * (k - 1 + r))];
        C.c[p][q][r] = v;
        C.sum += v;
      }
}

__device__ __forceinline__ float rcp(float x) { return __fdividef(1.0f, x); }

// D^-1 of the 16^3 level at every node (0 on the boundary)
template <int CT, typename T>
__device__ void dinv_level(const T* a, T* d) {
  constexpr int N = 16, n1 = N + 1;
  const T h3 = T(1.0 / (3.0 * N));
  for (int n = threadIdx.x; n < Lv<N>::nodes; n += CT) {
    int i, j, k;
    node_ijk(n, n1, i, j, k);
    T v = T(0);
    if (interior(i, j, k, N)) {
      auto sum4 = [&](int c) {
        const T* p = a + (i - 1) + N * (j - 1) + N * N * c;
        return (p[0] + p[1]) + (p[N] + p[N + 1]);
      };
      v = rcp(h3 * (sum4(k - 1) + sum4(k)));
    }
    d[n] = v;
  }
}

// pre-smoothing from 0 and the residual: x = omega D^-1 r (from d, or dividing by D),
// t = r - A x
template <int CT, int N, bool DTAB, typename T>
__device__ void pre_level(const T* r, const T* a, const T* d, T* x, T* t, T omega) {
  constexpr int n1 = N + 1;
  const T h3 = T(1.0 / (3.0 * N)), sc = T(1.0 / (12.0 * N));
  for (int n = threadIdx.x; n < Lv<N>::nodes; n += CT) {
    int i, j, k;
    node_ijk(n, n1, i, j, k);
    T v = T(0);
    if (interior(i, j, k, N)) {
      if (DTAB) {
        v = omega * r[n] * d[n];
      } else {
        Cells8<T, T> C;
        cells8(C, a, i, j, k, N);
        v = omega * r[n] / (h3 * C.sum);
      }
    }
    x[n] = v;
  }
  __syncthreads();
  for (int n = threadIdx.x; n < Lv<N>::nodes; n += CT) {
    int i, j, k;
    node_ijk(n, n1, i, j, k);
    T v = T(0);
    if (interior(i, j, k, N)) {
      Cells8<T, T> C;
      cells8(C, a, i, j, k, N);
      v = r[n] - sc * q1_row(C, x, i, j, k, n1);
    }
    t[n] = v;
  }
}

// rc = P^T tf (coarse level Nc, weights 1 and 1/2 per axis around the even fine node)
template <int CT, int NC, typename T>
__device__ void restrict_level(const T* tf, T* rc) {
  constexpr int n1c = NC + 1, n1f = 2 * NC + 1;
  for (int n = threadIdx.x; n < Lv<NC>::nodes; n += CT) {
    int I, J, K;
    node_ijk(n, n1c, I, J, K);
    T v = T(0);
    if (interior(I, J, K, NC)) {
      const T* f = tf + 2 * I + n1f * (2 * J) + n1f * n1f * (2 * K);
#pragma unroll
      for (int w = -1; w <= 1; ++w)
#pragma unroll
        for (int u = -1; u <= 1; ++u)
#pragma unroll
          for (int q = -1; q <= 1; ++q) {
            const T wt = T((q == 0 ? 1.0 : 0.5) * (u == 0 ? 1.0 : 0.5) * (w == 0 ? 1.0 : 0.5));
            v += wt * f[q + n1f * u + n1f * n1f * w];
          }
    }
    rc[n] = v;
  }
}

// xf += P ec (trilinear; ec holds 0 on its boundary)
template <int CT, int NF, typename T>
__device__ void prolong_level(T* xf, const T* ec) {
  constexpr int n1f = NF + 1, n1c = NF / 2 + 1;
  for (int n = threadIdx.x; n < Lv<NF>::nodes; n += CT) {
    int i, j, k;
    node_ijk(n, n1f, i, j, k);
    if (!interior(i, j, k, NF)) continue;
    const int i0 = i >> 1, j0 = j >> 1, k0 = k >> 1;
    const int i1 = i0 + (i & 1), j1 = j0 + (j & 1), k1 = k0 + (k & 1);
    const T wi = (i & 1) ? T(0.5) : T(1), wj = (j & 1) ? T(0.5) : T(1), wk = (k & 1) ? T(0.5) : T(1);
    auto at = [&](int a, int b, int c) { return ec[a + n1c * b + n1c * n1c * c]; };
    T v;
    if ((i & 1) == 0 && (j & 1) == 0 && (k & 1) == 0) {
      v = at(i0, j0, k0);
    } else {
      v = wi * wj * wk *
          (at(i0, j0, k0) + ((i & 1) ? at(i1, j0, k0) : T(0)) + ((j & 1) ? at(i0, j1, k0) : T(0)) +
           ((k & 1) ? at(i0, j0, k1) : T(0)) + (((i & 1) && (j & 1)) ? at(i1, j1, k0) : T(0)) +
           (((i & 1) && (k & 1)) ? at(i1, j0, k1) : T(0)) + (((j & 1) && (k & 1)) ? at(i0, j1, k1) : T(0)) +
           (((i & 1) && (j & 1) && (k & 1)) ? at(i1, j1, k1) : T(0)));
    }
    xf[n] += v;
  }
}

// post-smoothing z = x + omega D^-1 (r - A x), written to z (shared or global)
template <int CT, int N, bool DTAB, typename T>
__device__ void post_level(const T* r, const T* a, const T* d, const T* x, T* z, T omega) {
  constexpr int n1 = N + 1;
  const T h3 = T(1.0 / (3.0 * N)), sc = T(1.0 / (12.0 * N));
  for (int n = threadIdx.x; n < Lv<N>::nodes; n += CT) {
    int i, j, k;
    node_ijk(n, n1, i, j, k);
    T v = T(0);
    if (interior(i, j, k, N)) {
      Cells8<T, T> C;
      cells8(C, a, i, j, k, N);
      const T res = r[n] - sc * q1_row(C, x, i, j, k, n1);
      v = DTAB ? x[n] + omega * res * d[n] : x[n] + omega * res / (h3 * C.sum);
    }
    z[n] = v;
  }
}

}  // namespace mlsgd
