// small64.cu - FP64 work on 8^3 and 16^3 levels, one thread-block cluster per sample: the
// whole PCG solve on those grids, and the V-cycle below a 32^3 level (rows a4, a6).
//
// FP64 issues at 2 operations per clock and SM here, so a 16^3 sample on one SM is bound
// by its FP64 pipe (a V-cycle alone took 142 us), while as single passes over the whole
// GPU a solve is some 200 dependent launches.  A cluster gives a sample several pipes and
// still keeps it on chip: block c of the cluster owns the node planes 2c + 1 and 2c + 2
// (8 blocks on 16^3, 4 on 8^3; a thread owns the column (x, y) of both), holds its planes
// and one halo plane on either side in shared memory, and the blocks exchange through
// distributed shared memory: the residual restricted to the next level (each coarse plane
// is completed by two blocks), the next level's residual, the boundary planes of z and of
// q = A p, and the partial sums.  A PCG iteration has four cluster barriers (three on
// 8^3): r, p and the operands are updated on the halo planes too, so they need none.
//
// Operations.  The cells are scaled by h/12 once, and the sums of the two cells that share
// a face diagonal are formed once per solve, so with A = D - Off (D the diagonal, Off the
// 20 neighbours) every application is 20 FMAs and the smoother needs no diagonal:
//   x1 = w r, w = omega / D:   t = r - A x1 = (1 - omega) r + Off x1
//   x2 = w r + P e:            z = x2 + w (r - A x2) = (1 - omega) x2 + w (r + Off x2)
//   q = D p - Off p
// about 83 operations per node and iteration, of which the level-by-level kernels took
// some 140.  The levels 4^3 and 2^3 are one 27 x 27 matrix per sample, formed once.
// What is left is latency: a warp alone issues one FP64 operation in 64 clocks, so every
// step's length is the operations of its busiest warp, and three to four cluster barriers.
// Measured: state and adjoint solves of 4 samples of 8^3 at rtol 1e-12 2.92 ms in passes,
// 0.54 ms with the coarse levels run step by step, two nodes per thread and clusters packed
// onto SMs, 0.32 ms now; 64 samples 3.85, 0.68, 0.44; 16 samples of 16^3 with their 8^3
// partners at 1e-10 10.1, 1.78, 1.45 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "internal.cuh"
#include "kernels.h"
#include "launch.h"

namespace cg = cooperative_groups;

namespace mlsgd {

namespace {

template <int N>
struct Cfg {
  static constexpr int C = N / 2;               // blocks per sample (planes 2c + 1, 2c + 2)
  static constexpr int M = N - 1;               // interior nodes per side
  static constexpr int U = N == 16 ? 2 : 1;      // own nodes per thread: both planes of a column, or one
  static constexpr int NT = N == 16 ? 256 : 128;  // threads: M^2 columns (8^3: for each of the two planes)
  static constexpr int n1 = N + 1, PL = n1 * n1, CP = N * N;
};

// shared memory of one block (doubles); node planes 2c .. 2c + 3 at local planes 0 .. 3
template <int N>
struct Smem {
  using K = Cfg<N>;
  double r[4 * K::PL], op[4 * K::PL], wd[4 * K::PL];
  double c[3 * K::CP], fxy[2 * K::CP], fxz[3 * K::CP], fyz[3 * K::CP];  // scaled cells, face sums
  double t8[729], z4[125], a4[64], wd4[125], a2[8];
  double g4[27 * 27], inv4, part4[4 * 27];  // the V-cycle from 4^3 down as a matrix (coarse4_setup)
  double red[K::NT];
  double slot[3][K::C];  // partial sums of the blocks: r.r, r.z, p.q
  double bc;             // alpha or beta
  int go;
};
template <int N>
struct SmemSolve : Smem<N> {
  using K = Cfg<N>;
  double p[4 * K::PL], zh[2 * K::PL], qh[2 * K::PL];  // halo planes from the neighbours
};
template <int N, typename B>
struct With8 : B {};
template <typename B>
struct With8<16, B> : B {  // the 8^3 level below a 16^3 one
  double r8a[729], wd8[729], a8[512];
  union { double r8b[729], x8[729]; };  // x8 once r8b has been added to r8a
  double fxy8[3 * 64], fxz8[4 * 64], fyz8[4 * 64];  // face sums of the cell layers rank - 1 .. rank + 2
};

// Off x at an interior node: xq = &x[node], cq = &cells[lowest cell]; F: face sums
template <int S1, int S2, int CN>
__device__ __forceinline__ double off_row(double acc, const double* x, const double* c, const double* fxy,
                                          const double* fxz, const double* fyz) {
  // fxy at the node plane: cells (i-1+p, j-1+q); fxz at cell plane r: cells i-1+p, node row j;
  // fyz at cell plane r: node column i, cells j-1+q
  double a0 = acc, a1 = 0.0;  // two chains
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int p = 0; p < 2; ++p) a0 = fma(fxy[p + CN * q], x[(2 * p - 1) + S1 * (2 * q - 1)], a0);
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const double* xp = x + S2 * (2 * r - 1);
    const int o = CN * CN * r;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      a1 = fma(fxz[o + p], xp[2 * p - 1], a1);
      a0 = fma(fyz[o + CN * p], xp[S1 * (2 * p - 1)], a0);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const double v = xp[(2 * p - 1) + S1 * (2 * q - 1)];
        if (q) a1 = fma(c[o + p + CN * q], v, a1);
        else a0 = fma(c[o + p + CN * q], v, a0);
      }
  }
  return a0 + a1;
}
// the same from cells alone (levels whose face sums are not kept)
template <int CN>
__device__ __forceinline__ double off_cells(double acc, const double* x, const double* c) {
  constexpr int S1 = CN + 1, S2 = S1 * S1;
  double C[2][2][2];  // [r][q][p]
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) C[r][q][p] = c[p + CN * q + CN * CN * r];
  double a0 = acc, a1 = 0.0, a2 = 0.0;
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int u = 2 * p - 1, v = 2 * q - 1;
      a0 = fma(C[0][q][p] + C[1][q][p], x[u + S1 * v], a0);
      a1 = fma(C[q][0][p] + C[q][1][p], x[u + S2 * v], a1);
      a2 = fma(C[q][p][0] + C[q][p][1], x[S1 * u + S2 * v], a2);
      a0 = fma(C[0][q][p], x[u + S1 * v - S2], a0);
      a1 = fma(C[1][q][p], x[u + S1 * v + S2], a1);
    }
  return a0 + (a1 + a2);
}
// trilinear interpolation of the coarse vector e (row CS1, plane CS2 strides) at fine node (i, j, k)
template <int CS1, int CS2>
__device__ __forceinline__ double interp(const double* e, int i, int j, int k) {
  const double* q = e + (i >> 1) + CS1 * (j >> 1) + CS2 * (k >> 1);
  const int di = i & 1, dj = (j & 1) ? CS1 : 0, dk = (k & 1) ? CS2 : 0;
  auto line = [&](const double* s) { return di ? s[0] + s[1] : s[0]; };
  auto face = [&](const double* s) { return dj ? line(s) + line(s + dj) : line(s); };
  const double v = dk ? face(q) + face(q + dk) : face(q);
  const double w = (di ? 0.5 : 1.0) * (dj ? 0.5 : 1.0) * (dk ? 0.5 : 1.0);
  return w * v;
}
// (1, 2, 1)/2 weighted sum over the 3 x 3 x 3 nodes around f, three chains
template <int S1, int S2>
__device__ __forceinline__ double restrict27(const double* f) {
  double a[3];
#pragma unroll
  for (int w = -1; w <= 1; ++w) {
    double v = 0.0;
#pragma unroll
    for (int u = -1; u <= 1; ++u) {
      const double* s = f + S1 * u + S2 * w;
      v = fma(u == 0 ? 1.0 : 0.5, fma(0.5, s[-1] + s[1], s[0]), v);
    }
    a[w + 1] = v;
  }
  return fma(0.5, a[0] + a[2], a[1]);
}

// The V(1,1)-cycle from 4^3 down is a fixed linear map of the restricted residual r: with
// w = omega/D, p the interpolation of the 2^3 node to 4^3 (and its transpose the
// restriction), d the 2^3 diagonal and u = (1 - omega) p + w Off p,
//   z4 = w ((2 - omega) r + Off (w r)) + u (u . r) / d = G r,
// so the 27 x 27 matrix G is formed once and every cycle is one product with it: run step
// by step the level took a third of an 8^3 iteration (11070 of 33800 clocks: 170
// operations in a row in one warp, which alone issues one FP64 operation in 64 clocks).
// a4 holds h/12 a of the 4^3 cells, wd4 omega/D, a2 the 2^3 cells; z4 is 0 on entry.
template <typename SM>
__device__ void coarse4_setup(SM& M, double omega, int nt) {
  const int tid = threadIdx.x;
  const int I = 1 + tid % 3, J = 1 + (tid / 3) % 3, K = 1 + tid / 9, n = I + 5 * (J + 5 * K);
  const double p = ((I & 1) ? 0.5 : 1.0) * ((J & 1) ? 0.5 : 1.0) * ((K & 1) ? 0.5 : 1.0);
  if (tid < 27) M.z4[n] = p;
  if (tid == 32) {
    double s8 = 0.0;
#pragma unroll
    for (int e = 0; e < 8; ++e) s8 += M.a2[e];
    M.inv4 = 6.0 / s8;
  }
  __syncthreads();
  if (tid < 27)
    M.part4[tid] = fma(M.wd4[n], off_cells<4>(0.0, M.z4 + n, M.a4 + (I - 1) + 4 * ((J - 1) + 4 * (K - 1))), (1.0 - omega) * p);
  __syncthreads();
  for (int e = tid; e < 27 * 27; e += nt) {  // G[j][i]: a lane takes a row i
    const int i = e % 27, j = e / 27;
    const int xi = 1 + i % 3, yi = 1 + (i / 3) % 3, zi = 1 + i / 9;
    const int du = 1 + j % 3 - xi, dv = 1 + (j / 3) % 3 - yi, dw = 1 + j / 9 - zi;
    const double wi = M.wd4[xi + 5 * (yi + 5 * zi)], wj = M.wd4[(xi + du) + 5 * ((yi + dv) + 5 * (zi + dw))];
    double g = M.part4[i] * (M.part4[j] * M.inv4);
    if (i == j) g = fma(wi, 2.0 - omega, g);
    const int zeros = (du == 0) + (dv == 0) + (dw == 0);
    if (zeros <= 1 && abs(du) <= 1 && abs(dv) <= 1 && abs(dw) <= 1) {  // neighbours across a face or body diagonal
      const int c0 = (du > 0 ? xi : xi - 1) + 4 * ((dv > 0 ? yi : yi - 1) + 4 * (dw > 0 ? zi : zi - 1));
      double a = M.a4[c0];
      if (zeros) a += M.a4[c0 + (du == 0 ? 1 : dv == 0 ? 4 : 16)];
      g = fma(wi * a, wj, g);
    }
    M.g4[e] = g;
  }
}
// restricts M.t8, leaves the correction in M.z4 (complete after the next block barrier);
// called by every thread.  Four warps (one per quarter of the SM) share the sums.
template <typename SM>
__device__ __forceinline__ void coarse4(SM& M) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int I = 1 + lane % 3, J = 1 + (lane / 3) % 3, K = 1 + lane / 9;
  const bool own = lane < 27;
  if (own && w < 3) {  // the restriction's three planes
    const double* f = M.t8 + 2 * I + 18 * J + 81 * (2 * K + w - 1);
    double v = 0.0;
#pragma unroll
    for (int u = -1; u <= 1; ++u) {
      const double* q = f + 9 * u;
      v = fma(u == 0 ? 1.0 : 0.5, fma(0.5, q[-1] + q[1], q[0]), v);
    }
    M.part4[27 * w + lane] = v;
  }
  __syncthreads();
  double z = 0.0;
  if (w < 4) {  // columns 7 w .. 7 w + 6 of G
    const double r = own ? fma(0.5, M.part4[lane] + M.part4[54 + lane], M.part4[27 + lane]) : 0.0;
    const double* g = M.g4 + 7 * 27 * w + (own ? lane : 0);
#pragma unroll
    for (int jj = 0; jj < 7; ++jj) {
      const double rj = __shfl_sync(0xffffffffu, r, (7 * w + jj) & 31);
      if (7 * w + jj < 27) z = fma(g[27 * jj], rj, z);
    }
  }
  __syncthreads();
  if (own && w < 4) M.part4[27 * w + lane] = z;
  __syncthreads();
  if (own && w == 0)
    M.z4[I + 5 * (J + 5 * K)] = (M.part4[lane] + M.part4[27 + lane]) + (M.part4[54 + lane] + M.part4[81 + lane]);
}

// One V(1,1)-cycle on M.r (own and halo planes): z of the thread's own nodes, planes
// 2 rank + 1 + u0 + (0 .. U - 1) of its column.
// after_t runs between the barrier that publishes the restricted residual and the rest
// (false: the cluster stops here).
template <int N, typename SM, typename F>
__device__ __forceinline__ bool vcycle(SM& M, cg::cluster_group& cl, int rank, bool col, int i, int j, double omega,
                                       int u0, double (&z)[Cfg<N>::U], F&& after_t) {
  using K = Cfg<N>;
  constexpr int S1 = K::n1, S2 = K::PL, C = K::C, U = K::U;
  const int tid = threadIdx.x, nb = i + S1 * j, cb = (i - 1) + N * (j - 1);
  const double om1 = 1.0 - omega;
  const int l0 = 2 * u0;  // the thread's staged planes l0 .. l0 + 2 U - 1
  if (col) {
#pragma unroll
    for (int l = l0; l < l0 + 2 * U; ++l) M.op[l * S2 + nb] = M.r[l * S2 + nb] * M.wd[l * S2 + nb];
  }
  __syncthreads();
  auto off = [&](double acc, const double* v, int u) {  // node plane 2 rank + 1 + u
    return off_row<S1, S2, N>(acc, v + (u + 1) * S2 + nb, M.c + u * K::CP + cb, M.fxy + u * K::CP + cb,
                              M.fxz + u * K::CP + (i - 1) + N * j, M.fyz + u * K::CP + i + N * (j - 1));
  };
  const int nown = 2 * rank + 2 < N ? 2 : 1;  // the last block's second plane is the boundary
  double t[U] = {};
  if (col) {
#pragma unroll
    for (int v = 0; v < U; ++v)
      if (u0 + v < nown) t[v] = off(om1 * M.r[(u0 + v + 1) * S2 + nb], M.op, u0 + v);
  }
  if constexpr (N == 16) {
    __syncthreads();  // op has been read: t takes its first two planes
    if (col) {
      M.op[nb] = t[0];
      M.op[S2 + nb] = t[U - 1];
    }
    __syncthreads();
    if (tid < 49) {  // coarse planes rank + 1 (planes 2 rank + 1, 2 rank + 2) and rank (half of plane 2 rank + 1)
      const int I = 1 + tid % 7, J = 1 + tid / 7;
      const double* f = M.op + 2 * I + 17 * (2 * J);
      double a[3], b[3];
#pragma unroll
      for (int u = -1; u <= 1; ++u) {
        const double* s = f + 17 * u;
        b[u + 1] = fma(0.5, s[-1] + s[1], s[0]);
        a[u + 1] = fma(0.5, s[288] + s[290], s[289]);
      }
      const double lo = 0.5 * fma(0.5, b[0] + b[2], b[1]);
      const double up = fma(0.5, a[0] + a[2], a[1]) + lo;
      const int e = I + 9 * J;
      for (int q = 0; q < C; ++q) {
        SM* R = cl.map_shared_rank(&M, q);
        if (rank + 1 < 8) R->r8a[e + 81 * (rank + 1)] = up;
        if (rank > 0) R->r8b[e + 81 * rank] = lo;
      }
    }
  } else {
    if (col && u0 < nown) {
      for (int q = 0; q < C; ++q) cl.map_shared_rank(&M, q)->t8[nb + 81 * (2 * rank + 1 + u0)] = t[0];
    }
  }
  // Off x8 at node (a, b, k) of the 8^3 level, k = rank .. rank + 2
  auto off8 = [&](double acc, int a, int b, int k) {
    if constexpr (N == 16) {
      const int l = k - rank;
      return off_row<9, 81, 8>(acc, M.x8 + a + 9 * b + 81 * k, M.a8 + (a - 1) + 8 * (b - 1) + 64 * (k - 1),
                               M.fxy8 + 64 * l + (a - 1) + 8 * (b - 1), M.fxz8 + 64 * l + (a - 1) + 8 * b,
                               M.fyz8 + 64 * l + a + 8 * (b - 1));
    }
    return acc;
  };
  cl.sync();
  if (!after_t()) return false;
  if constexpr (N == 16) {
    for (int e = tid; e < 729; e += K::NT) {
      const double v = M.r8a[e] + M.r8b[e];
      M.r8a[e] = v;
      M.x8[e] = M.wd8[e] * v;  // 0 on the boundary
    }
    __syncthreads();
    const int kt = rank + 1;  // the block's plane of the 8^3 residual
    if (kt < 8 && tid < 49) {
      const int a = 1 + tid % 7, b = 1 + tid / 7, n = a + 9 * b + 81 * kt;
      const double v = off8(om1 * M.r8a[n], a, b, kt);
      for (int q = 0; q < C; ++q) cl.map_shared_rank(&M, q)->t8[n] = v;
    }
    cl.sync();
  }
  coarse4(M);
  __syncthreads();
  if constexpr (N == 16) {
    // corrected x8 on the planes the stencils of planes rank .. rank + 2 read, then z8 there
    const int p0 = rank > 1 ? rank - 1 : 1, p1 = rank + 3 < 7 ? rank + 3 : 7;
    for (int e = tid; e < 49 * (p1 - p0 + 1); e += K::NT) {
      const int a = 1 + e % 7, b = 1 + (e / 7) % 7, k = p0 + e / 49, n = a + 9 * b + 81 * k;
      M.x8[n] += interp<5, 25>(M.z4, a, b, k);
    }
    __syncthreads();
    const int q0 = rank > 0 ? rank : 1, q1 = rank + 2 < 7 ? rank + 2 : 7;
    for (int e = tid; e < 49 * (q1 - q0 + 1); e += K::NT) {
      const int a = 1 + e % 7, b = 1 + (e / 7) % 7, k = q0 + e / 49, n = a + 9 * b + 81 * k;
      M.t8[n] = fma(M.wd8[n], off8(M.r8a[n], a, b, k), om1 * M.x8[n]);
    }
    __syncthreads();
  }
  double x2[2 * U];
  if (col) {
    // staged plane l is node plane 2 rank + l: an even l takes coarse plane rank + l/2, an odd
    // one the mean of it and the next; the sums over x and y are shared, weights come last
    const double* e = N == 16 ? M.t8 : M.z4;
    constexpr int E1 = N / 2 + 1, E2 = E1 * E1;
    auto face = [&](int kc) {
      if (kc > N / 2) return 0.0;
      const double* q = e + (i >> 1) + E1 * (j >> 1) + E2 * kc;
      double v = q[0];
      if (i & 1) v += q[1];
      if (j & 1) v += (i & 1) ? q[E1] + q[E1 + 1] : q[E1];
      return v;
    };
    const double wf = ((i & 1) ? 0.5 : 1.0) * ((j & 1) ? 0.5 : 1.0);
    double f = face(rank + u0);
#pragma unroll
    for (int h = 0; h < U; ++h) {
      const int l = l0 + 2 * h;
      const double fn = face(rank + u0 + h + 1);
      x2[2 * h] = fma(wf, f, M.wd[l * S2 + nb] * M.r[l * S2 + nb]);
      x2[2 * h + 1] = fma(0.5 * wf, f + fn, M.wd[(l + 1) * S2 + nb] * M.r[(l + 1) * S2 + nb]);
      if (2 * rank + l + 1 > N) x2[2 * h + 1] = 0.0;
      M.op[l * S2 + nb] = x2[2 * h];
      M.op[(l + 1) * S2 + nb] = x2[2 * h + 1];
      f = fn;
    }
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < U; ++v) {
    z[v] = 0.0;
    const int l = u0 + v + 1;
    if (col && u0 + v < nown)
      z[v] = fma(M.wd[l * S2 + nb], off(M.r[l * S2 + nb], M.op, u0 + v), om1 * x2[l - l0]);
  }
  return true;
}

// scaled cells of the block's three cell planes (2 rank .. 2 rank + 2) and their face sums;
// a: the sample's cells.  Planes outside the grid hold 0.
template <int N, typename SM>
__device__ void load_cells(SM& M, const double* a, int rank) {
  using K = Cfg<N>;
  const double s = 1.0 / (12.0 * N);
  for (int e = threadIdx.x; e < 3 * K::CP; e += K::NT) {
    const int k = 2 * rank + e / K::CP;
    M.c[e] = k < N ? s * a[(long long)k * K::CP + e % K::CP] : 0.0;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 3 * K::CP; e += K::NT) {
    const int i = e % N, j = (e / N) % N;
    if (e < 2 * K::CP) M.fxy[e] = M.c[e] + M.c[e + K::CP];
    M.fxz[e] = j > 0 ? M.c[e - N] + M.c[e] : 0.0;
    M.fyz[e] = i > 0 ? M.c[e - 1] + M.c[e] : 0.0;
  }
}
// face sums of the 8^3 level around planes rank .. rank + 2 from M.a8 (scaled)
template <typename SM>
__device__ void faces8(SM& M, int rank) {
  for (int e = threadIdx.x; e < 4 * 64; e += 256) {
    const int L = rank - 1 + e / 64, q = e & 63, i = q & 7, j = q >> 3;  // cell layer L at local layer e / 64
    const bool in = L >= 0 && L < 8;
    const double* c = M.a8 + 64 * (in ? L : 0) + q;
    M.fxz8[e] = in && j > 0 ? c[-8] + c[0] : 0.0;
    M.fyz8[e] = in && i > 0 ? c[-1] + c[0] : 0.0;
    if (e < 3 * 64) M.fxy8[e] = in && L + 1 < 8 ? c[0] + c[64] : 0.0;
  }
}
// zero what the passes never write (boundary nodes)
template <typename SM>
__device__ void clear_all(SM& M, int nt) {
  double* d = reinterpret_cast<double*>(&M);
  for (unsigned e = threadIdx.x; e < sizeof(SM) / 8; e += nt) d[e] = 0.0;
}

// ---------------------------------------------------------------- the V-cycle below 32^3
struct CoarseArgs64 {
  const double* r;      // restricted residual of the 16^3 level [S][17^3]
  const double* a[4];   // cells of 16^3 .. 2^3
  const double* wd[3];  // omega D^-1 of 16^3, 8^3, 4^3
  double* z;            // correction [S][17^3]
  const SolveScalars* sc;
  const int* act;
  double omega;
};
using SmemV = With8<16, Smem<16>>;

__global__ void __launch_bounds__(256, 2) k_vcycle64(CoarseArgs64 A) {
  pdl_entry();
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), t = blockIdx.x / 8;
  const int s = A.act != nullptr ? A.act[t] : t;
  if (A.sc != nullptr && !A.sc[s].active) return;  // the whole cluster
  extern __shared__ __align__(16) unsigned char smraw[];
  SmemV& M = *reinterpret_cast<SmemV*>(smraw);
  const int tid = threadIdx.x;
  clear_all(M, 256);
  __syncthreads();
  load_cells<16>(M, A.a[0] + (long long)s * 4096, rank);
  const double* rg = A.r + (long long)s * 4913 + 2 * rank * 289;
  const double* wg = A.wd[0] + (long long)s * 4913 + 2 * rank * 289;
  const int planes = 2 * rank + 3 > 16 ? 3 : 4;
  for (int e = tid; e < planes * 289; e += 256) {
    M.r[e] = rg[e];
    M.wd[e] = wg[e];
  }
  for (int e = tid; e < 512; e += 256) M.a8[e] = (1.0 / 96.0) * A.a[1][(long long)s * 512 + e];
  for (int e = tid; e < 729; e += 256) M.wd8[e] = A.wd[1][(long long)s * 729 + e];
  if (tid < 64) M.a4[tid] = (1.0 / 48.0) * A.a[2][(long long)s * 64 + tid];
  if (tid < 125) M.wd4[tid] = A.wd[2][(long long)s * 125 + tid];
  if (tid < 8) M.a2[tid] = A.a[3][(long long)s * 8 + tid];
  __syncthreads();
  faces8(M, rank);
  coarse4_setup(M, A.omega, 256);
  cl.sync();  // every block's memory is ready for its neighbours' writes
  const int i = 1 + tid % 15, j = 1 + tid / 15;
  const bool col = tid < 225;
  double z[2];
  vcycle<16>(M, cl, rank, col, i, j, A.omega, 0, z, [] { return true; });
  double* zo = A.z + (long long)s * 4913 + (2 * rank + 1) * 289;
  if (col) {
    zo[i + 17 * j] = z[0];
    if (rank < 7) zo[289 + i + 17 * j] = z[1];
  }
  cl.sync();  // no block leaves while others may still write to it
}

// ---------------------------------------------------------------- the whole solve
struct SolveArgs64 {
  const double* a;    // cells [S][N^3]
  const double* b;    // right-hand side, bstride 0: one for every sample
  long long bstride;
  double* x;          // solution [S][(N+1)^3]
  SolveScalars* sc;
  double tol2, omega;
  int max_iter;
};

__device__ __forceinline__ double mean8(const double* f, int Nf) {
  double v = 0.0;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) v += f[p + Nf * (q + Nf * r)];
  return 0.125 * v;
}
// omega / D at interior node (i, j, k) of an NN^3 level with scaled cells (h a / 12) c
template <int NN>
__device__ __forceinline__ double omega_over_d(const double* c, int i, int j, int k, double omega) {
  const double* q = c + (i - 1) + NN * ((j - 1) + NN * (k - 1));
  double v = 0.0;
#pragma unroll
  for (int e = 0; e < 8; ++e) v += q[(e & 1) + NN * ((e >> 1) & 1) + NN * NN * (e >> 2)];
  return omega / (4.0 * v);
}

template <int N>
__global__ void __launch_bounds__(Cfg<N>::NT, N == 16 ? 2 : 5) k_small64(SolveArgs64 A) {
  pdl_entry();
  using K = Cfg<N>;
  using SM = With8<N, SmemSolve<N>>;
  constexpr int S1 = K::n1, S2 = K::PL, C = K::C, NT = K::NT, U = K::U;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), s = blockIdx.x / C;
  extern __shared__ __align__(16) unsigned char smraw[];
  SM& M = *reinterpret_cast<SM*>(smraw);
  const int tid = threadIdx.x, lane = tid & 31;
  const double* as = A.a + (long long)s * K::CP * N;
  const long long nodes = (long long)S2 * S1;
  const double* bs = A.b + s * A.bstride;
  clear_all(M, NT);
  __syncthreads();
  load_cells<N>(M, as, rank);
  __syncthreads();
  // coarse coefficients (means of the eight children; scaled by h/12 once all are formed)
  if constexpr (N == 16) {
    for (int e = tid; e < 512; e += NT) {
      const int x = e & 7, y = (e >> 3) & 7, zc = e >> 6;
      M.a8[e] = mean8(as + 2 * x + 16 * (2 * y) + 256 * (2 * zc), 16);
    }
    __syncthreads();
    for (int e = tid; e < 64; e += NT) M.a4[e] = mean8(M.a8 + 2 * (e & 3) + 8 * (2 * ((e >> 2) & 3)) + 64 * (2 * (e >> 4)), 8);
  } else {
    for (int e = tid; e < 64; e += NT) M.a4[e] = mean8(as + 2 * (e & 3) + 8 * (2 * ((e >> 2) & 3)) + 64 * (2 * (e >> 4)), 8);
  }
  __syncthreads();
  if (tid < 8) M.a2[tid] = mean8(M.a4 + 2 * (tid & 1) + 4 * (2 * ((tid >> 1) & 1)) + 16 * (2 * (tid >> 2)), 4);
  __syncthreads();
  if constexpr (N == 16)
    for (int e = tid; e < 512; e += NT) M.a8[e] *= 1.0 / 96.0;
  for (int e = tid; e < 64; e += NT) M.a4[e] *= 1.0 / 48.0;
  __syncthreads();
  if (tid < 27) {
    const int I = 1 + tid % 3, J = 1 + (tid / 3) % 3, Kc = 1 + tid / 9;
    M.wd4[I + 5 * (J + 5 * Kc)] = omega_over_d<4>(M.a4, I, J, Kc, A.omega);
  }
  if constexpr (N == 16) {
    for (int e = tid; e < 343; e += NT) {
      const int a = 1 + e % 7, b = 1 + (e / 7) % 7, k = 1 + e / 49;
      M.wd8[a + 9 * b + 81 * k] = omega_over_d<8>(M.a8, a, b, k, A.omega);
    }
  }
  __syncthreads();
  if constexpr (N == 16) faces8(M, rank);
  coarse4_setup(M, A.omega, NT);
  // this thread's column, its own planes u0 .. u0 + U - 1, their diagonal and right-hand side
  const int u0 = U == 2 ? 0 : tid >> 6, tc = U == 2 ? tid : tid & 63;
  const int i = 1 + tc % K::M, j = 1 + tc / K::M, nb = i + S1 * j, cb = (i - 1) + N * (j - 1);
  const bool col = tc < K::M * K::M;
  const int nown = 2 * rank + 2 < N ? 2 : 1;
  double D[U] = {}, x[U] = {};
  double bb = 0.0;
  if (col) {
    auto sum4 = [&](const double* q) { return (q[0] + q[1]) + (q[N] + q[N + 1]); };
#pragma unroll
    for (int h = 0; h < U; ++h) {
      const int u = u0 + h;
      if (u < nown) {
        D[h] = 4.0 * sum4(M.fxy + u * K::CP + cb);
        const double v = bs[(2 * rank + 1 + u) * S2 + nb];
        M.r[(u + 1) * S2 + nb] = v;
        bb = fma(v, v, bb);
        M.wd[(u + 1) * S2 + nb] = A.omega / D[h];
      }
    }
    // halo planes: their diagonal from the cells in memory (one plane beyond the block's)
    const double h12 = 1.0 / (12.0 * N);
    auto halo = [&](int k, int l) {
      if (k <= 0 || k >= N) return;
      const double* q = as + (long long)(k - 1) * K::CP + cb;
      M.wd[l * S2 + nb] = A.omega / (4.0 * (h12 * (sum4(q) + sum4(q + K::CP))));
      M.r[l * S2 + nb] = bs[k * S2 + nb];
    };
    if (u0 == 0) halo(2 * rank, 0);
    if (u0 == 2 - U) halo(2 * rank + 3, 3);
  }
  // block sum to every block's slot (complete after the next cluster barrier)
  auto push_sum = [&](double v, int which) {
    M.red[tid] = v;
    __syncthreads();
    if (tid < 32) {
      double a = M.red[lane];
#pragma unroll
      for (int q = 1; q < NT / 32; ++q) a += M.red[lane + 32 * q];
      a = warp_sum(a);
      if (lane < C) cl.map_shared_rank(&M, lane)->slot[which][rank] = a;
    }
  };
  auto slot_sum = [&](int which) {  // warp 0
    double v = lane < C ? M.slot[which][lane] : 0.0;
#pragma unroll
    for (int o = C / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return __shfl_sync(0xffffffffu, v, 0);
  };
  cl.sync();  // every block's memory is ready for its neighbours' writes
  push_sum(bb, 0);
  cl.sync();
  // scalars of the sample, the same in thread 0 of every block
  double bbs = 0.0, rr = 0.0, rz = 0.0;
  int iters = 0, status = 0;
  if (tid < 32) {
    const double v = slot_sum(0);
    if (tid == 0) {
      bbs = rr = v;
      M.go = v > 0.0 && v < INFINITY;
      if (!(v < INFINITY)) status = 2;
    }
  }
  cl.sync();  // slot 0 has been read by every block
  bool go = M.go != 0;
  double rsum = 0.0;  // r.r of the own nodes
  for (int it = 0; go; ++it) {
    if (it > 0) push_sum(rsum, 0);
    double z[U];
    const bool on = vcycle<N>(M, cl, rank, col, i, j, A.omega, u0, z, [&] {
      if (it == 0) return true;
      // stop test of the iterate before this V-cycle
      if (tid < 32) {
        const double v = slot_sum(0);
        if (tid == 0) {
          rr = v;
          iters += 1;
          int g = 1;
          if (v <= A.tol2 * bbs) g = 0;
          else if (!(v < INFINITY)) { g = 0; status = 2; }
          else if (iters >= A.max_iter) { g = 0; status = 1; }
          M.go = g;
        }
      }
      __syncthreads();
      return M.go != 0;
    });
    if (!on) break;
    // r.z, and z on the neighbours' halo planes
    double v = 0.0;
    if (col) {
#pragma unroll
      for (int h = 0; h < U; ++h)
        if (u0 + h < nown) v = fma(M.r[(u0 + h + 1) * S2 + nb], z[h], v);
      if (u0 == 0 && rank > 0) cl.map_shared_rank(&M, rank - 1)->zh[S2 + nb] = z[0];
      if (u0 == 2 - U && rank + 1 < C) cl.map_shared_rank(&M, rank + 1)->zh[nb] = z[U - 1];
    }
    push_sum(v, 1);
    cl.sync();
    if (tid < 32) {
      const double w = slot_sum(1);
      if (tid == 0) {
        M.bc = (it > 0 && rz != 0.0) ? w / rz : 0.0;
        rz = w;
      }
    }
    __syncthreads();
    const double beta = M.bc;
    if (col) {  // p = z + beta p on the own and the halo planes
      double zl[2 * U];  // the thread's staged planes 2 u0 .. 2 u0 + 2 U - 1
      if constexpr (U == 2) {
        zl[0] = M.zh[nb]; zl[1] = z[0]; zl[2] = z[1]; zl[3] = M.zh[S2 + nb];
      } else {
        zl[0] = u0 ? z[0] : M.zh[nb];
        zl[1] = u0 ? M.zh[S2 + nb] : z[0];
      }
#pragma unroll
      for (int h = 0; h < 2 * U; ++h) {
        double* pl = M.p + (2 * u0 + h) * S2 + nb;
        *pl = it == 0 ? zl[h] : fma(beta, *pl, zl[h]);
      }
    }
    __syncthreads();
    double q[U] = {};
    v = 0.0;
    if (col) {
#pragma unroll
      for (int h = 0; h < U; ++h) {
        const int u = u0 + h;
        if (u < nown) {
          const double pv = M.p[(u + 1) * S2 + nb];
          const double o = off_row<S1, S2, N>(0.0, M.p + (u + 1) * S2 + nb, M.c + u * K::CP + cb,
                                              M.fxy + u * K::CP + cb, M.fxz + u * K::CP + (i - 1) + N * j,
                                              M.fyz + u * K::CP + i + N * (j - 1));
          q[h] = fma(D[h], pv, -o);
          v = fma(pv, q[h], v);
        }
      }
      if (u0 == 0 && rank > 0) cl.map_shared_rank(&M, rank - 1)->qh[S2 + nb] = q[0];
      if (u0 == 2 - U && rank + 1 < C) cl.map_shared_rank(&M, rank + 1)->qh[nb] = q[U - 1];
    }
    push_sum(v, 2);
    cl.sync();
    if (tid < 32) {
      const double w = slot_sum(2);
      if (tid == 0) M.bc = (w > 0.0 && rz != 0.0) ? rz / w : 0.0;
    }
    __syncthreads();
    const double alpha = M.bc;
    rsum = 0.0;
    if (col) {
      double ql[2 * U];
      if constexpr (U == 2) {
        ql[0] = M.qh[nb]; ql[1] = q[0]; ql[2] = q[1]; ql[3] = M.qh[S2 + nb];
      } else {
        ql[0] = u0 ? q[0] : M.qh[nb];
        ql[1] = u0 ? M.qh[S2 + nb] : q[0];
      }
#pragma unroll
      for (int h = 0; h < 2 * U; ++h) {
        double* rl = M.r + (2 * u0 + h) * S2 + nb;
        *rl = fma(-alpha, ql[h], *rl);
      }
#pragma unroll
      for (int h = 0; h < U; ++h) {
        const int u = u0 + h;
        x[h] = fma(alpha, M.p[(u + 1) * S2 + nb], x[h]);
        const double rv = M.r[(u + 1) * S2 + nb];
        if (u < nown) rsum = fma(rv, rv, rsum);
      }
    }
  }
  // the own planes of the solution, boundary nodes 0 (the first and the last block: planes 0 and N)
  double* xo = A.x + s * nodes;
  for (int e = tid; e < 2 * S2; e += NT) {
    const int k = 2 * rank + 1 + e / S2, n = e % S2;
    const int xx = n % S1, yy = n / S1;
    if (xx == 0 || yy == 0 || xx == N || yy == N || k == N) xo[(long long)k * S2 + n] = 0.0;
    if (rank == 0 && e < S2) xo[e] = 0.0;
  }
  if (col) {
#pragma unroll
    for (int h = 0; h < U; ++h)
      if (u0 + h < nown) xo[(long long)(2 * rank + 1 + u0 + h) * S2 + nb] = x[h];
  }
  if (rank == 0 && tid == 0) {
    SolveScalars c;
    c.bb = bbs; c.rz = rz; c.alpha = 0.0; c.beta = 0.0; c.rr = rr;
    c.active = 0; c.iters = iters; c.status = status; c.pad = 0;
    A.sc[s] = c;
  }
  cl.sync();  // no block leaves while others may still write to it
}

static_assert(sizeof(SmemV) <= 113 * 1024 && sizeof(With8<16, SmemSolve<16>>) <= 113 * 1024, "two blocks per SM");

// Launches one cluster per sample, spread over as many SMs as one wave allows: blocks that
// share an SM share its FP64 pipe, and the hardware fills an SM before it takes the next
// (16 clusters of eight blocks went to 64 SMs).  The shared memory that is asked for sets
// how many blocks an SM takes: the fewest with which every sample's cluster is resident.
struct Spread {  // of one device
  std::mutex m;
  int n = 0;  // 0: not set up (again after a failure)
  size_t smem[8];
  int clusters[8];  // resident with at most i + 1 blocks per SM
};
template <typename Args>
cudaError_t launch_spread(Spread (&spreads)[SmemOptIn::kDevices], const char* cls, double bytes, void (*k)(Args), int threads, int cluster,
                          size_t smem, int most, int samples, cudaStream_t st, const Args& A) {
  int dev = 0;
  const cudaError_t ed = cudaGetDevice(&dev);
  if (ed != cudaSuccess) return ed;
  if (dev < 0 || dev >= SmemOptIn::kDevices) return cudaErrorInvalidDevice;
  Spread& sp = spreads[dev];
  {
    std::lock_guard<std::mutex> lock(sp.m);
    if (sp.n == 0) {
      constexpr size_t kSm = 228 * 1024, kBlock = 1024;  // of an SM; reserved per block
      const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)std::max(smem, kSm / 2 - kBlock + 16));
      if (e != cudaSuccess) return e;
      for (int occ = 1; occ <= most; ++occ) {
        const size_t want = std::max(smem, kSm / (occ + 1) - kBlock + 16);  // occ + 1 blocks don't fit
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)cluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)cluster);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = want;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int c = 0;  // without an answer the least shared memory is taken
        const bool clean = cudaPeekAtLastError() == cudaSuccess;
        if (cudaOccupancyMaxActiveClusters(&c, k, &cfg) != cudaSuccess) {
          if (clean) (void)cudaGetLastError();  // an earlier call's error stays
          c = 0;
        }
        sp.smem[occ - 1] = want;
        sp.clusters[occ - 1] = c;
      }
      sp.n = most;
    }
  }
  size_t use = smem;
  for (int i = 0; i < sp.n; ++i)
    if (sp.clusters[i] >= samples) {
      use = sp.smem[i];
      break;
    }
  return launch_cluster(cls, bytes, k, dim3((unsigned)(samples * cluster)), dim3((unsigned)threads), (unsigned)cluster,
                        use, st, A);
}

}  // namespace

cudaError_t coarse_vcycle64(const double* r16, const double* const a[4], const double* const wd[3], double* z16,
                            const SolveScalars* sc, const Batch& bt, double omega, cudaStream_t st) {
  static Spread sp[SmemOptIn::kDevices];
  CoarseArgs64 A{};
  A.r = r16;
  for (int l = 0; l < 4; ++l) A.a[l] = a[l];
  for (int l = 0; l < 3; ++l) A.wd[l] = wd[l];
  A.z = z16; A.sc = sc; A.act = bt.act; A.omega = omega;
  // per sample: r, z and omega D^-1 of 16^3, the coefficient levels, omega D^-1 of 8^3 and 4^3
  const double bytes = (double)bt.n * 8 * (3.0 * 4913 + 4096 + 512 + 64 + 8 + 729 + 125);
  return launch_spread(sp, "coarse_f64", bytes, k_vcycle64, 256, 8, sizeof(SmemV), 2, bt.n, st, A);
}

cudaError_t small_fp64(SolverBufs& B, const double* a64, const double* b, long long bstride, double* x_out,
                       const PcgParams& prm, cudaStream_t st) {
  const int N = B.N, S = B.S;
  SolveArgs64 A{a64, b, bstride, x_out, B.sc, prm.rtol * prm.rtol, prm.omega, prm.max_iter};
  const double bytes = (bstride ? S : 1) * (double)nodes_of(N) * 8 + (double)S * 8 * (nodes_of(N) + cells_of(N));
  static Spread sp8[SmemOptIn::kDevices], sp16[SmemOptIn::kDevices];
  if (N == 16)
    return launch_spread(sp16, "small_f64", bytes, k_small64<16>, 256, 8, sizeof(With8<16, SmemSolve<16>>), 2, S, st, A);
  return launch_spread(sp8, "small_f64", bytes, k_small64<8>, 128, 4, sizeof(With8<8, SmemSolve<8>>), 5, S, st, A);
}

}  // namespace mlsgd
