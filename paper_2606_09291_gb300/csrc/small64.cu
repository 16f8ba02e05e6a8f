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
// some 140.  The levels 4^3 and 2^3 are one warp's work in every block.
// What is left is latency: barriers, dependent FMAs and the scalars' divisions.
// Measured: state and adjoint solves of 4 samples of 8^3 at rtol 1e-12 2.92 ms in passes,
// 0.57 ms now; 16 samples of 16^3 with their 8^3 partners at 1e-10 10.1 -> 2.1 ms; with the
// V-cycle below 32^3 9 samples of 64^3 and partners 36.2 -> 29.2 ms.
#include <cooperative_groups.h>

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
  static constexpr int NT = N == 16 ? 256 : 64;  // threads: M^2 columns
  static constexpr int n1 = N + 1, PL = n1 * n1, CP = N * N;
};

// shared memory of one block (doubles); node planes 2c .. 2c + 3 at local planes 0 .. 3
template <int N>
struct Smem {
  using K = Cfg<N>;
  double r[4 * K::PL], op[4 * K::PL], wd[4 * K::PL];
  double c[3 * K::CP], fxy[2 * K::CP], fxz[3 * K::CP], fyz[3 * K::CP];  // scaled cells, face sums
  double t8[729], x4[125], t4[125], z4[125], a4[64], wd4[125], a2[8];
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
  double t[2 * 289];
  double r8a[729], r8b[729], x8[729], wd8[729], a8[512];
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

// levels 4^3 and 2^3 by warp 0 of every block: restricts M.t8, leaves the correction in M.z4
template <typename SM>
__device__ __forceinline__ void coarse4(SM& M, double omega) {
  const int lane = threadIdx.x;
  const int I = 1 + lane % 3, J = 1 + (lane / 3) % 3, K = 1 + lane / 9;
  const int n = I + 5 * (J + 5 * K), c = (I - 1) + 4 * ((J - 1) + 4 * (K - 1));
  const bool own = lane < 27;
  double r = 0.0, w = 0.0, x = 0.0;
  if (own) {
    r = restrict27<9, 81>(M.t8 + 2 * I + 18 * J + 162 * K);
    w = M.wd4[n];
    x = w * r;
    M.x4[n] = x;
  }
  __syncwarp();
  if (own) M.t4[n] = off_cells<4>((1.0 - omega) * r, M.x4 + n, M.a4 + c);
  __syncwarp();
  const double r2 = restrict27<5, 25>(M.t4 + 62);
  double s8 = 0.0;
#pragma unroll
  for (int e = 0; e < 8; ++e) s8 += M.a2[e];
  const double e2 = r2 / ((1.0 / 6.0) * s8);
  if (own) {
    x = fma(((I & 1) ? 0.5 : 1.0) * ((J & 1) ? 0.5 : 1.0) * ((K & 1) ? 0.5 : 1.0), e2, x);
    M.x4[n] = x;
  }
  __syncwarp();
  if (own) M.z4[n] = fma(w, off_cells<4>(r, M.x4 + n, M.a4 + c), (1.0 - omega) * x);
}

// One V(1,1)-cycle on M.r (own and halo planes): z of the own column's two nodes.
// after_t runs between the barrier that publishes the restricted residual and the rest
// (false: the cluster stops here).
template <int N, typename SM, typename F>
__device__ __forceinline__ bool vcycle(SM& M, cg::cluster_group& cl, int rank, bool col, int i, int j, double omega,
                                       double z[2], F&& after_t) {
  using K = Cfg<N>;
  constexpr int S1 = K::n1, S2 = K::PL, C = K::C;
  const int tid = threadIdx.x, nb = i + S1 * j, cb = (i - 1) + N * (j - 1);
  const double om1 = 1.0 - omega;
  if (col) {
#pragma unroll
    for (int l = 0; l < 4; ++l) M.op[l * S2 + nb] = M.r[l * S2 + nb] * M.wd[l * S2 + nb];
  }
  __syncthreads();
  auto off = [&](double acc, const double* v, int u) {  // node plane 2 rank + 1 + u
    return off_row<S1, S2, N>(acc, v + (u + 1) * S2 + nb, M.c + u * K::CP + cb, M.fxy + u * K::CP + cb,
                              M.fxz + u * K::CP + (i - 1) + N * j, M.fyz + u * K::CP + i + N * (j - 1));
  };
  const int nown = 2 * rank + 2 < N ? 2 : 1;  // the last block's second plane is the boundary
  double t[2] = {0.0, 0.0};
  if (col) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < nown) t[u] = off(om1 * M.r[(u + 1) * S2 + nb], M.op, u);
  }
  if constexpr (N == 16) {
    if (col) {
      M.t[nb] = t[0];
      M.t[S2 + nb] = t[1];
    }
    __syncthreads();
    if (tid < 49) {  // coarse planes rank + 1 (planes 2 rank + 1, 2 rank + 2) and rank (half of plane 2 rank + 1)
      const int I = 1 + tid % 7, J = 1 + tid / 7;
      const double* f = M.t + 2 * I + 17 * (2 * J);
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
    if (col) {
      for (int q = 0; q < C; ++q) {
        SM* R = cl.map_shared_rank(&M, q);
        R->t8[nb + 81 * (2 * rank + 1)] = t[0];
        if (nown == 2) R->t8[nb + 81 * (2 * rank + 2)] = t[1];
      }
    }
  }
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
      const double v = off_cells<8>(om1 * M.r8a[n], M.x8 + n, M.a8 + (a - 1) + 8 * (b - 1) + 64 * (kt - 1));
      for (int q = 0; q < C; ++q) cl.map_shared_rank(&M, q)->t8[n] = v;
    }
    cl.sync();
  }
  if (tid < 32) coarse4(M, omega);
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
      const double s = off_cells<8>(M.r8a[n], M.x8 + n, M.a8 + (a - 1) + 8 * (b - 1) + 64 * (k - 1));
      M.t8[n] = fma(M.wd8[n], s, om1 * M.x8[n]);
    }
    __syncthreads();
  }
  double x2[4];
  if (col) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int k = 2 * rank + l;
      double e = 0.0;
      if (k > 0 && k < N) {
        if constexpr (N == 16) e = interp<9, 81>(M.t8, i, j, k);
        else e = interp<5, 25>(M.z4, i, j, k);
      }
      x2[l] = fma(M.wd[l * S2 + nb], M.r[l * S2 + nb], e);
      M.op[l * S2 + nb] = x2[l];
    }
  }
  __syncthreads();
  z[0] = z[1] = 0.0;
  if (col) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < nown)
        z[u] = fma(M.wd[(u + 1) * S2 + nb], off(M.r[(u + 1) * S2 + nb], M.op, u), om1 * x2[u + 1]);
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
  cl.sync();  // every block's memory is ready for its neighbours' writes
  const int i = 1 + tid % 15, j = 1 + tid / 15;
  const bool col = tid < 225;
  double z[2];
  vcycle<16>(M, cl, rank, col, i, j, A.omega, z, [] { return true; });
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
__global__ void __launch_bounds__(Cfg<N>::NT, N == 16 ? 2 : 8) k_small64(SolveArgs64 A) {
  pdl_entry();
  using K = Cfg<N>;
  using SM = With8<N, SmemSolve<N>>;
  constexpr int S1 = K::n1, S2 = K::PL, C = K::C, NT = K::NT;
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
  // this thread's column, its diagonal and right-hand side
  const int i = 1 + tid % K::M, j = 1 + tid / K::M, nb = i + S1 * j, cb = (i - 1) + N * (j - 1);
  const bool col = tid < K::M * K::M;
  const int nown = 2 * rank + 2 < N ? 2 : 1;
  double D[2] = {0.0, 0.0}, x[2] = {0.0, 0.0};
  double bb = 0.0;
  if (col) {
    auto sum4 = [&](const double* q) { return (q[0] + q[1]) + (q[N] + q[N + 1]); };
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < nown) {
        D[u] = 4.0 * sum4(M.fxy + u * K::CP + cb);
        const double v = bs[(2 * rank + 1 + u) * S2 + nb];
        M.r[(u + 1) * S2 + nb] = v;
        bb = fma(v, v, bb);
        M.wd[(u + 1) * S2 + nb] = A.omega / D[u];
      }
    // halo planes: their diagonal from the cells in memory (one plane beyond the block's)
    const double h12 = 1.0 / (12.0 * N);
    auto halo = [&](int k, int l) {
      if (k <= 0 || k >= N) return;
      const double* q = as + (long long)(k - 1) * K::CP + cb;
      M.wd[l * S2 + nb] = A.omega / (4.0 * (h12 * (sum4(q) + sum4(q + K::CP))));
      M.r[l * S2 + nb] = bs[k * S2 + nb];
    };
    halo(2 * rank, 0);
    halo(2 * rank + 3, 3);
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
    double z[2];
    const bool on = vcycle<N>(M, cl, rank, col, i, j, A.omega, z, [&] {
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
      v = M.r[S2 + nb] * z[0];
      if (nown == 2) v = fma(M.r[2 * S2 + nb], z[1], v);
      if (rank > 0) cl.map_shared_rank(&M, rank - 1)->zh[S2 + nb] = z[0];
      if (rank + 1 < C) cl.map_shared_rank(&M, rank + 1)->zh[nb] = z[1];
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
      const double zl[4] = {M.zh[nb], z[0], z[1], M.zh[S2 + nb]};
#pragma unroll
      for (int l = 0; l < 4; ++l) M.p[l * S2 + nb] = it == 0 ? zl[l] : fma(beta, M.p[l * S2 + nb], zl[l]);
    }
    __syncthreads();
    double q[2] = {0.0, 0.0};
    v = 0.0;
    if (col) {
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (u < nown) {
          const double pv = M.p[(u + 1) * S2 + nb];
          const double o = off_row<S1, S2, N>(0.0, M.p + (u + 1) * S2 + nb, M.c + u * K::CP + cb,
                                              M.fxy + u * K::CP + cb, M.fxz + u * K::CP + (i - 1) + N * j,
                                              M.fyz + u * K::CP + i + N * (j - 1));
          q[u] = fma(D[u], pv, -o);
          v = fma(pv, q[u], v);
        }
      if (rank > 0) cl.map_shared_rank(&M, rank - 1)->qh[S2 + nb] = q[0];
      if (rank + 1 < C) cl.map_shared_rank(&M, rank + 1)->qh[nb] = q[1];
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
      const double ql[4] = {M.qh[nb], q[0], q[1], M.qh[S2 + nb]};
#pragma unroll
      for (int l = 0; l < 4; ++l) M.r[l * S2 + nb] = fma(-alpha, ql[l], M.r[l * S2 + nb]);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        x[u] = fma(alpha, M.p[(u + 1) * S2 + nb], x[u]);
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
    xo[(long long)(2 * rank + 1) * S2 + nb] = x[0];
    if (nown == 2) xo[(long long)(2 * rank + 2) * S2 + nb] = x[1];
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

template <typename Kern>
cudaError_t allow_smem(Kern* k, size_t bytes, bool& done) {
  if (done) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  done = e == cudaSuccess;
  return e;
}

}  // namespace

cudaError_t coarse_vcycle64(const double* r16, const double* const a[4], const double* const wd[3], double* z16,
                            const SolveScalars* sc, const Batch& bt, double omega, cudaStream_t st) {
  static bool smem_set = false;  // once (capture-friendly)
  const cudaError_t e = allow_smem(k_vcycle64, sizeof(SmemV), smem_set);
  if (e != cudaSuccess) return e;
  CoarseArgs64 A{};
  A.r = r16;
  for (int l = 0; l < 4; ++l) A.a[l] = a[l];
  for (int l = 0; l < 3; ++l) A.wd[l] = wd[l];
  A.z = z16; A.sc = sc; A.act = bt.act; A.omega = omega;
  // per sample: r, z and omega D^-1 of 16^3, the coefficient levels, omega D^-1 of 8^3 and 4^3
  const double bytes = (double)bt.n * 8 * (3.0 * 4913 + 4096 + 512 + 64 + 8 + 729 + 125);
  return launch_cluster("coarse_f64", bytes, k_vcycle64, dim3((unsigned)bt.n * 8), dim3(256), 8, sizeof(SmemV), st, A);
}

cudaError_t small_fp64(SolverBufs& B, const double* a64, const double* b, long long bstride, double* x_out,
                       const PcgParams& prm, cudaStream_t st) {
  const int N = B.N, S = B.S;
  SolveArgs64 A{a64, b, bstride, x_out, B.sc, prm.rtol * prm.rtol, prm.omega, prm.max_iter};
  const double bytes = (bstride ? S : 1) * (double)nodes_of(N) * 8 + (double)S * 8 * (nodes_of(N) + cells_of(N));
  if (N == 16) {
    using SM = With8<16, SmemSolve<16>>;
    static bool smem_set = false;
    const cudaError_t e = allow_smem(k_small64<16>, sizeof(SM), smem_set);
    if (e != cudaSuccess) return e;
    return launch_cluster("small_f64", bytes, k_small64<16>, dim3((unsigned)S * 8), dim3(256), 8, sizeof(SM), st, A);
  }
  using SM = With8<8, SmemSolve<8>>;
  static bool smem_set8 = false;
  const cudaError_t e = allow_smem(k_small64<8>, sizeof(SM), smem_set8);
  if (e != cudaSuccess) return e;
  return launch_cluster("small_f64", bytes, k_small64<8>, dim3((unsigned)S * 4), dim3(64), 4, sizeof(SM), st, A);
}

}  // namespace mlsgd
