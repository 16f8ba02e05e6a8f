// cluster32.cu - FP32 work on 32^3 levels with a cluster of four blocks per sample: the
// whole mixed-precision solve on a 32^3 grid, and the V-cycle from a coarse 32^3 level
// down (rows a4, a6).
//
// Run pass by pass, a PCG iteration on 32^3 is six dependent launches (pre-smoothing, the
// V-cycle below, post-smoothing, A p and two scalar updates) of 10 to 15 us each, most
// of it launch latency, partial sums through memory and too few blocks: one 32^3 sample
// is four blocks.  Here block c of a cluster keeps the node planes 8c + 1 .. 8c + 8 of
// its sample (one segment of the passes' partial sums) with one halo plane on either side
// in shared memory, and the blocks exchange boundary planes and partial sums through
// distributed shared memory: seven cluster barriers per iteration.  The 16^3 level is
// split the same way (four planes each), 8^3 and below is every block's own work.  The
// vectors a thread reads only at its own nodes (r, p, the correction) stay in global
// memory (L2); their halo planes are updated along with the own ones.
//
// What bounds it (ncu, 16 samples): the latency of barriers and of the vectors in L2 (6.4 and
// 5.6 of 24 cycles per instruction of a warp); a block of 1024 threads has one SM to
// itself and issues in 33% of its cycles.  It wins while the clusters make few waves (kCluster32Max in solver.cu).
//
// Arithmetic: that of the slab passes (slab.cu), the fused coarse V-cycle (coarse.cu) and
// the refinement step on the same level, operation by operation, with the order of their
// sums: a thread owns four rows of two planes; the dot products run as one chain per
// (lane, row group) through the eight planes, handed from the threads of two planes to
// the next.
#include <cooperative_groups.h>

#include "internal.cuh"
#include "kernels.h"
#include "launch.h"
#include "onchip.cuh"
#include "refine.cuh"

namespace cg = cooperative_groups;

namespace mlsgd {

namespace {

constexpr int kC = 4;            // blocks per sample
constexpr int kNT = 1024;
constexpr int n1 = 33, PL = n1 * n1, kNodes = PL * n1;  // 32^3 grid
constexpr int CPL = 32 * 32;
constexpr int P16 = 17 * 17;

struct Smem {
  float op[10 * PL];     // operand, local plane l = plane 8c + l
  float t[8 * PL];       // residual to restrict; between V-cycles: z and q from the neighbours
  float rh[2 * PL];      // r on the halo planes 8c and 8c + 9
  float sv[225];         // the next block's first residual plane, restricted in x and y
  float r16[6 * P16], x16[6 * P16], t16[6 * P16], z16[6 * P16], d16[6 * P16];  // local plane l: plane 4c + l
  float a16[7 * 256];    // cell plane 4c - 1 + l
  float lv[kCoarse8Floats];
  float chain[8][32];
  float red8[8];
  double slot[2][kC];
  float bc;
  int go;
};
template <typename TA>
struct SmemV : Smem {
  TA cells[9 * CPL];     // V-cycle coefficient, cell plane 8c + l
};
struct SmemS : SmemV<__nv_bfloat16> {
  float a32[9 * CPL];    // operator coefficient
  float ph[2 * PL], dh[2 * PL];  // p and the correction on the halo planes
};
static_assert(sizeof(SmemS) <= 227 * 1024 && sizeof(SmemV<float>) <= 227 * 1024, "shared memory");

__device__ __forceinline__ float cell_f(float c) { return c; }
__device__ __forceinline__ float cell_f(__nv_bfloat16 c) { return __bfloat162float(c); }

// where a thread works
struct Own {
  int rank, lane, ws, kq;  // row group 4 ws + 1 .. 4 ws + 4, planes l = 1 + 2 kq, 2 + 2 kq
  int x, y0;
  __device__ bool row_ok(int t) const { return lane < 31 && y0 + t < 32; }
  __device__ bool ok(int u, int t) const { return row_ok(t) && 8 * rank + 1 + 2 * kq + u < 32; }
  __device__ int l(int u) const { return 1 + 2 * kq + u; }
  __device__ int at(int l, int t) const { return l * PL + (y0 + t) * n1 + x; }           // local
  __device__ int node(int l, int t) const { return (8 * rank + l) * PL + (y0 + t) * n1 + x; }  // of the sample
};

// the 3 x 6 operand window of local plane l and the 2 x 5 cells of local cell plane c
using Win = float[3][6];
using Cel = float[2][5];
__device__ __forceinline__ void load_win(const float* op, const Own& w, int l, Win& W) {
  const float* p = op + l * PL + (w.y0 - 1) * n1 + w.x - 1;
#pragma unroll
  for (int r = 0; r < 6; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) W[c][r] = p[(w.y0 - 1 + r < n1 ? r : 0) * n1 + c];  // row 33 does not exist
}
template <typename TA>
__device__ __forceinline__ void load_cel(const TA* a, const Own& w, int c, Cel& C) {
  const TA* p = a + c * CPL + (w.y0 - 1) * 32 + w.x - 1;
#pragma unroll
  for (int r = 0; r < 5; ++r)
#pragma unroll
    for (int q = 0; q < 2; ++q) C[q][r] = cell_f(p[(w.y0 - 1 + r < 32 ? r : 0) * 32 + (w.x - 1 + q < 32 ? q : 0)]);
}
__device__ __forceinline__ void off_term(float (&acc)[4], const Win& W, const Cel& C) {
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    float a2 = acc[t];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      a2 -= (C[u][t] + C[u][t + 1]) * W[2 * u][t + 1];
      a2 -= (C[0][t + u] + C[1][t + u]) * W[1][t + 2 * u];
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) a2 -= C[p][t + q] * W[2 * p][t + 2 * q];
    acc[t] = a2;
  }
}
__device__ __forceinline__ void centre_term(float (&acc)[4], const Win& W, const Cel& Cl, const Cel& Ch) {
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    float pxy[2][2];
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
      for (int u = 0; u < 2; ++u) pxy[v][u] = Cl[u][t + v] + Ch[u][t + v];
    const float sum8 = (pxy[0][0] + pxy[0][1]) + (pxy[1][0] + pxy[1][1]);
    float a1 = fmaf(4.f * sum8, W[1][t + 1], acc[t]);
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
      for (int u = 0; u < 2; ++u) a1 -= pxy[v][u] * W[2 * u][t + 2 * v];
    acc[t] = a1;
  }
}
// (A op) / (h / 12) at the thread's nodes of its two planes, and the operand there: four
// operand windows and three cell planes serve both
template <typename TA>
__device__ __forceinline__ void apply_rows(const float* op, const TA* a, const Own& w, float (&acc)[2][4],
                                           float (&ctr)[2][4]) {
  const int l = w.l(0);
  Win W;
  Cel C0, C1;
#pragma unroll
  for (int t = 0; t < 4; ++t) acc[0][t] = acc[1][t] = 0.f;
  load_cel(a, w, l - 1, C0);
  load_win(op, w, l - 1, W);
  off_term(acc[0], W, C0);
  load_cel(a, w, l, C1);
  load_win(op, w, l, W);
  centre_term(acc[0], W, C0, C1);
  off_term(acc[1], W, C1);
#pragma unroll
  for (int t = 0; t < 4; ++t) ctr[0][t] = W[1][t + 1];
  load_win(op, w, l + 1, W);
  off_term(acc[0], W, C1);
  load_cel(a, w, l + 1 < 9 ? l + 1 : 8, C0);
  centre_term(acc[1], W, C1, C0);
#pragma unroll
  for (int t = 0; t < 4; ++t) ctr[1][t] = W[1][t + 1];
  load_win(op, w, l + 2, W);
  off_term(acc[1], W, C0);
}

// The V-cycle's static data below 32^3
struct Levels {
  CoarseLevels c8;
  int i8, j8, k8;
  bool in8;
  float D8;
};
// loads the coefficient levels below 32^3 (global arrays of the sample) and zeroes what no
// pass writes; ends with a block barrier
template <typename SM>
__device__ void load_levels(SM& M, Levels& L, int rank, const float* a16, const float* a8, const float* a4,
                            const float* a2) {
  const int tid = threadIdx.x;
  for (int e = tid; e < 10 * PL; e += kNT) M.op[e] = 0.f;
  for (int e = tid; e < 2 * PL; e += kNT) M.rh[e] = 0.f;
  for (int e = tid; e < 6 * P16; e += kNT) M.r16[e] = M.x16[e] = M.t16[e] = M.z16[e] = M.d16[e] = 0.f;
  for (int e = tid; e < 225; e += kNT) M.sv[e] = 0.f;
  for (int e = tid; e < 7 * 256; e += kNT) {
    const int cz = 4 * rank - 1 + e / 256;
    M.a16[e] = cz >= 0 && cz < 16 ? a16[cz * 256 + e % 256] : 0.f;
  }
  for (int e = tid; e < kCoarse8Floats; e += kNT) M.lv[e] = 0.f;
  __syncthreads();
  CoarseLevels& c = L.c8;
  c.r8 = M.lv; c.x8 = c.r8 + 729; c.t8 = c.x8 + 729;
  float* s8 = c.t8 + 729;
  c.x4 = s8 + 512; c.t4 = c.x4 + 125;
  float* s4 = c.t4 + 125;
  float* s2 = s4 + 64;
  c.a8 = s8; c.a4 = s4; c.a2 = s2;
  for (int e = tid; e < 512; e += kNT) s8[e] = a8[e];
  if (tid < 64) s4[tid] = a4[tid];
  if (tid < 8) s2[tid] = a2[tid];
  // D^-1 of the 16^3 level on the own and halo planes
  for (int e = tid; e < 6 * 225; e += kNT) {
    const int l = e / 225, j = 1 + (e / 15) % 15, i = 1 + e % 15, k = 4 * rank + l;
    if (k <= 0 || k >= 16) continue;
    auto sum4 = [&](int cl) {
      const float* p = M.a16 + (i - 1) + 16 * (j - 1) + 256 * cl;
      return (p[0] + p[1]) + (p[16] + p[17]);
    };
    M.d16[l * P16 + j * 17 + i] = __fdividef(1.0f, float(1.0 / 48.0) * (sum4(l) + sum4(l + 1)));
  }
  __syncthreads();
  L.i8 = L.j8 = L.k8 = 0;
  if (tid < 729) node_ijk(tid, 9, L.i8, L.j8, L.k8);
  L.in8 = tid < 729 && interior(L.i8, L.j8, L.k8, 8);
  L.D8 = L.in8 ? diag_of<8>(s8, L.i8, L.j8, L.k8) : 1.f;
}

// One V(1,1)-cycle on r (global, own nodes; M.rh on the halo planes): z at the own nodes.
// rv: r at the own nodes (loaded here).
template <typename SM>
__device__ __forceinline__ void vcycle32(SM& M, cg::cluster_group& cl, const Own& w, const Levels& L, const float* r,
                                         const float* dinv, float omega, float (&z)[2][4], float (&rv)[2][4]) {
  const int tid = threadIdx.x, rank = w.rank;
  constexpr float scale = float(1.0 / (12.0 * 32)), sc16 = float(1.0 / (12.0 * 16));
  // x1 = omega D^-1 r on the own and halo planes
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      rv[u][t] = 0.f;
      if (w.ok(u, t)) {
        const int g = w.node(w.l(u), t);
        rv[u][t] = r[g];
        M.op[w.at(w.l(u), t)] = rv[u][t] * dinv[g];
      }
    }
  const int hl = w.kq == 0 ? 0 : 9, hk = 8 * rank + hl;  // halo plane of this row group's first and last threads
  const bool hplane = (w.kq == 0 || w.kq == 3) && hk > 0 && hk < 32;
  const float* rh = M.rh + (w.kq == 0 ? 0 : PL);
  if (hplane) {
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (w.row_ok(t)) M.op[w.at(hl, t)] = rh[w.at(0, t)] * dinv[w.node(hl, t)];
  }
  __syncthreads();
  {
    float acc[2][4], ctr[2][4];
    apply_rows(M.op, M.cells, w, acc, ctr);
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (w.row_ok(t)) M.t[w.at(w.l(u) - 1, t)] = w.ok(u, t) ? fmaf(-scale, acc[u][t], rv[u][t]) : 0.f;
  }
  __syncthreads();
  // restriction to 16^3: planes 4c + 1 .. 4c + 4; the last one needs the next block's first plane
  auto xy = [&](int X, int Y, int lt) {  // residual plane lt restricted in x and y
    const float* p = M.t + lt * PL + 2 * Y * n1 + 2 * X;
    auto row = [&](int o) { return fmaf(0.5f, p[o - 1] + p[o + 1], p[o]); };
    return fmaf(0.5f, row(-n1) + row(n1), row(0));
  };
  const int X = 1 + tid % 15, Y = 1 + (tid / 15) % 15, l16 = 1 + tid / 225;
  const bool own16 = tid < 900 && 4 * rank + l16 < 16;
  const int n16 = l16 * P16 + Y * 17 + X;
  float r16 = 0.f;
  if (own16) {
    const int lt = 2 * l16 - 1;  // local residual plane (t index) of fine plane 2Z: 8c + 2 l16
    r16 = 0.5f * xy(X, Y, lt - 1);
    r16 = r16 + xy(X, Y, lt);
    if (l16 < 4) r16 = fmaf(0.5f, xy(X, Y, lt + 1), r16);
  }
  if (rank > 0 && tid < 225) cl.map_shared_rank(&M, rank - 1)->sv[tid] = xy(1 + tid % 15, 1 + tid / 15, 0);
  cl.sync();
  if (own16) {
    if (l16 == 4) r16 = fmaf(0.5f, M.sv[tid - 675], r16);
    M.r16[n16] = r16;
    if (l16 == 1 && rank > 0) cl.map_shared_rank(&M, rank - 1)->r16[n16 + 4 * P16] = r16;
    if (l16 == 4 && rank + 1 < kC) cl.map_shared_rank(&M, rank + 1)->r16[n16 - 4 * P16] = r16;
  }
  cl.sync();
  for (int e = tid; e < 6 * P16; e += kNT) M.x16[e] = omega * M.r16[e] * M.d16[e];  // d16 is 0 on the boundary
  __syncthreads();
  Cells8<float, float> C;
  if (own16) {
    cells8(C, (const float*)M.a16, X, Y, l16 + 1, 16);
    const float v = r16 - sc16 * q1_row(C, (const float*)M.x16, X, Y, l16, 17);
    M.t16[n16] = v;
    if (l16 == 1 && rank > 0) cl.map_shared_rank(&M, rank - 1)->t16[n16 + 4 * P16] = v;
  }
  cl.sync();
  if (tid < 98) {  // 8^3 planes 2c + 1, 2c + 2
    const int a = 1 + tid % 7, b = 1 + (tid / 7) % 7, h = tid / 49, K = 2 * rank + 1 + h;
    if (K < 8) {
      const float* f = M.t16 + 2 * a + 17 * (2 * b) + P16 * (2 + 2 * h);
      float v = 0.f;
#pragma unroll
      for (int k = -1; k <= 1; ++k)
#pragma unroll
        for (int j = -1; j <= 1; ++j)
#pragma unroll
          for (int i = -1; i <= 1; ++i) {
            const float wt = float((i == 0 ? 1.0 : 0.5) * (j == 0 ? 1.0 : 0.5) * (k == 0 ? 1.0 : 0.5));
            v += wt * f[i + 17 * j + P16 * k];
          }
      for (int q = 0; q < kC; ++q) cl.map_shared_rank(&M, q)->lv[a + 9 * b + 81 * K] = v;  // r8
    }
  }
  cl.sync();
  (void)vcycle8<kNT>(L.c8, tid, L.i8, L.j8, L.k8, L.in8, L.D8, omega);
  __syncthreads();
  // x16 += P z8 on the own and halo planes
  for (int e = tid; e < 6 * 225; e += kNT) {
    const int l = e / 225, j = 1 + (e / 15) % 15, i = 1 + e % 15, k = 4 * rank + l;
    if (k <= 0 || k >= 16) continue;
    const int i0 = i >> 1, j0 = j >> 1, k0 = k >> 1;
    const int i1 = i0 + (i & 1), j1 = j0 + (j & 1), k1 = k0 + (k & 1);
    const float wi = (i & 1) ? 0.5f : 1.f, wj = (j & 1) ? 0.5f : 1.f, wk = (k & 1) ? 0.5f : 1.f;
    auto at = [&](int a, int b, int c) { return L.c8.t8[a + 9 * b + 81 * c]; };
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
    M.x16[l * P16 + j * 17 + i] += v;
  }
  __syncthreads();
  if (own16) {
    const float res = r16 - sc16 * q1_row(C, (const float*)M.x16, X, Y, l16, 17);
    const float v = M.x16[n16] + omega * res * M.d16[n16];
    M.z16[n16] = v;
    if (l16 == 1 && rank > 0) cl.map_shared_rank(&M, rank - 1)->z16[n16 + 4 * P16] = v;
    if (l16 == 4 && rank + 1 < kC) cl.map_shared_rank(&M, rank + 1)->z16[n16 - 4 * P16] = v;
  }
  cl.sync();
  // x2 = omega D^-1 r + P z16 on the own and halo planes
  auto corr = [&](int l, int t) {  // P z16 at the thread's node of local plane l
    const int yy = w.y0 + t;
    const float* e = M.z16 + (l >> 1) * P16 + (yy >> 1) * 17 + (w.x >> 1);
    const bool px = w.x & 1, py = yy & 1;
    auto plane = [&](const float* q) {
      if (!px && !py) return q[0];
      if (!py) return 0.5f * (q[0] + q[1]);
      if (!px) return 0.5f * (q[0] + q[17]);
      return 0.5f * (0.5f * (q[0] + q[1]) + 0.5f * (q[17] + q[18]));
    };
    return (l & 1) ? 0.5f * (plane(e) + plane(e + P16)) : plane(e);
  };
  float dv[2][4];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      dv[u][t] = 0.f;
      if (w.ok(u, t)) {
        dv[u][t] = dinv[w.node(w.l(u), t)];
        M.op[w.at(w.l(u), t)] = fmaf(rv[u][t], dv[u][t], corr(w.l(u), t));
      }
    }
  if (hplane) {
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (w.row_ok(t)) M.op[w.at(hl, t)] = fmaf(rh[w.at(0, t)], dinv[w.node(hl, t)], corr(hl, t));
  }
  __syncthreads();
  float acc[2][4], ctr[2][4];
  apply_rows(M.op, M.cells, w, acc, ctr);
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int t = 0; t < 4; ++t)
      z[u][t] = w.ok(u, t) ? fmaf(fmaf(-scale, acc[u][t], rv[u][t]), dv[u][t], ctr[u][t]) : 0.f;
}

__device__ __forceinline__ Own own_of(int rank) {
  Own w;
  const int warp = threadIdx.x >> 5;
  w.rank = rank;
  w.lane = threadIdx.x & 31;
  w.ws = warp & 7;
  w.kq = warp >> 3;
  w.x = w.lane + 1;
  w.y0 = 1 + 4 * w.ws;
  return w;
}

// ---------------------------------------------------------------- the V-cycle from a coarse 32^3 level
struct VArgs {
  const float *r, *a, *dinv;                 // residual, cells and omega D^-1 of the 32^3 level
  const float *a16, *a8, *a4, *a2;           // cells below
  float* z;
  const SolveScalars* sc;
  const int* act;
  float omega;
};
__global__ void __launch_bounds__(kNT, 1) k_vcycle32(VArgs A) {
  pdl_entry();
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tb = blockIdx.x / kC;
  const int s = A.act != nullptr ? A.act[tb] : tb;
  if (A.sc != nullptr && !A.sc[s].active) return;  // the whole cluster
  extern __shared__ __align__(16) unsigned char smraw[];
  SmemV<float>& M = *reinterpret_cast<SmemV<float>*>(smraw);
  const Own w = own_of(rank);
  const float* r = A.r + (long long)s * kNodes;
  const float* dinv = A.dinv + (long long)s * kNodes;
  const float* a = A.a + (long long)s * 32768;
  for (int e = threadIdx.x; e < 9 * CPL; e += kNT) M.cells[e] = 8 * rank + e / CPL < 32 ? a[8 * rank * CPL + e] : 0.f;
  Levels L;
  load_levels(M, L, rank, A.a16 + (long long)s * 4096, A.a8 + (long long)s * 512, A.a4 + (long long)s * 64,
              A.a2 + (long long)s * 8);
  for (int e = threadIdx.x; e < PL; e += kNT) {
    if (rank > 0) M.rh[e] = r[8 * rank * PL + e];
    if (rank + 1 < kC) M.rh[PL + e] = r[(8 * rank + 9) * PL + e];
  }
  cl.sync();  // every block's memory is ready for its neighbours' writes
  float z[2][4], rv[2][4];
  vcycle32(M, cl, w, L, r, dinv, A.omega, z, rv);
  float* zo = A.z + (long long)s * kNodes;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (w.ok(u, t)) zo[w.node(w.l(u), t)] = z[u][t];
  cl.sync();  // no block leaves while others may still write to it
}

// ---------------------------------------------------------------- the whole solve on a 32^3 grid
struct SArgs {
  const float *a32, *dinv;
  const __nv_bfloat16* abf;
  const float *a16, *a8, *a4, *a2;
  float *r, *p, *d;          // own-node vectors; r holds b rounded
  const float2* rr_in;       // b as pairs, rr_stride 0: one for every sample
  long long rr_stride;
  float2 *rr, *x;            // residual pairs after a step, solution pairs
  SolveScalars* sc;          // bb, active, status from the init pass
  double tol2;
  float omega;
  int fixed, cap, inner, inner_next;
};

__global__ void __launch_bounds__(kNT, 1) k_solve32(SArgs A) {
  pdl_entry();
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), s = blockIdx.x / kC, tid = threadIdx.x;
  extern __shared__ __align__(16) unsigned char smraw[];
  SmemS& M = *reinterpret_cast<SmemS*>(smraw);
  const Own w = own_of(rank);
  constexpr float scale = float(1.0 / (12.0 * 32));
  const long long base = (long long)s * kNodes;
  float2* x = A.x + base;
  // the solution's boundary nodes, and all of it for a sample that takes no step
  const bool active = A.sc[s].active != 0;
  for (int e = tid; e < 9 * PL; e += kNT) {
    const int k = 8 * rank + e / PL, i = e % n1, j = (e / n1) % n1;
    if (k > 32 || (rank > 0 && e < PL)) continue;  // plane 8c belongs to the block before
    if (!active || k == 0 || k == 32 || i == 0 || i == 32 || j == 0 || j == 32) x[k * PL + e % PL] = make_float2(0.f, 0.f);
  }
  if (!active) return;  // the whole cluster
  float* r = A.r + base;
  float* p = A.p + base;
  float* d = A.d + base;
  const float* dinv = A.dinv + base;
  for (int e = tid; e < 9 * CPL; e += kNT) {
    const bool in = 8 * rank + e / CPL < 32;
    const long long g = (long long)s * 32768 + 8 * rank * CPL + e;
    M.cells[e] = in ? A.abf[g] : __float2bfloat16_rn(0.f);
    M.a32[e] = in ? A.a32[g] : 0.f;
  }
  for (int e = tid; e < 2 * PL; e += kNT) M.ph[e] = M.dh[e] = 0.f;
  Levels L;
  load_levels(M, L, rank, A.a16 + (long long)s * 4096, A.a8 + (long long)s * 512, A.a4 + (long long)s * 64,
              A.a2 + (long long)s * 8);
  auto load_rh = [&] {
    for (int e = tid; e < PL; e += kNT) {
      if (rank > 0) M.rh[e] = __ldcg(r + 8 * rank * PL + e);
      if (rank + 1 < kC) M.rh[PL + e] = __ldcg(r + (8 * rank + 9) * PL + e);
    }
  };
  load_rh();
  Outer o{A.sc[s].bb, A.sc[s].bb, 0.0, 0, A.sc[s].status, 0};
  // sum over the sample of u v in the order of the slab passes; result in warp 0 after the
  // cluster barrier
  auto dot = [&](const float (&u)[2][4], const float (&v)[2][4], int which) {
    float red = 0.f;
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {  // the chain of eight planes, two by two
      if (w.kq == q) {
        red = q ? M.chain[w.ws][w.lane] : 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int t = 0; t < 4; ++t) red = fmaf(u[k][t], v[k][t], red);  // 0 off the interior
        if (q < 3) M.chain[w.ws][w.lane] = red;
      }
      if (q < 3) __syncthreads();
    }
    if (w.kq == 3) {
      red = warp_sum(red);
      if (w.lane == 0) M.red8[w.ws] = red;
    }
    __syncthreads();
    if (tid < 32) {
      float b = w.lane < 8 ? M.red8[w.lane] : 0.f;
#pragma unroll
      for (int h = 4; h > 0; h >>= 1) b += __shfl_xor_sync(0xffffffffu, b, h);
      if (w.lane < kC) cl.map_shared_rank(&M, w.lane)->slot[which][rank] = (double)b;
    }
    cl.sync();
    double t = 0.0;
    if (tid < 32) {
      t = w.lane < kC ? M.slot[which][w.lane] : 0.0;
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      t += __shfl_xor_sync(0xffffffffu, t, 1);
    }
    return t;  // lane 0
  };
  // own boundary planes of v into the neighbours' halo buffers at M.t + o
  auto push = [&](const float (&v)[2][4], int off) {
    if (w.kq == 0 && rank > 0) {
      float* h = cl.map_shared_rank(&M, rank - 1)->t + off + PL;
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (w.row_ok(t)) h[w.at(0, t)] = v[0][t];
    }
    if (w.kq == 3 && rank + 1 < kC) {
      float* h = cl.map_shared_rank(&M, rank + 1)->t + off;
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (w.row_ok(t)) h[w.at(0, t)] = v[1][t];
    }
  };
  const int hl = w.kq == 0 ? 0 : 9, hk = 8 * rank + hl, ho = w.kq == 0 ? 0 : PL;
  const bool hplane = (w.kq == 0 || w.kq == 3) && hk > 0 && hk < 32;
  cl.sync();  // every block's memory is ready for its neighbours' writes
  float al = 0.f;
  int last = A.inner;
  for (int step = 0;; ++step) {
    float rv[2][4], z[2][4];
    if (step > 0) {  // refinement step: inc = d + alpha p, rr -= A inc, r = rr rounded, x (+)= inc
      const bool dzero = last <= 1;
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (w.ok(u, t)) {
            const int g = w.node(w.l(u), t);
            M.op[w.at(w.l(u), t)] = dzero ? al * p[g] : fmaf(al, p[g], d[g]);
          }
      if (hplane) {
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (w.row_ok(t)) {
            const int e = ho + w.at(0, t);
            M.op[w.at(hl, t)] = dzero ? al * M.ph[e] : fmaf(al, M.ph[e], M.dh[e]);
          }
      }
      __syncthreads();
      const float2* rin = step == 1 ? A.rr_in + s * A.rr_stride : A.rr + base;
      constexpr double kH12 = 1.0 / (12.0 * 32);
      const float sch = (float)kH12, scl = (float)(kH12 - (double)(float)kH12);  // h/12 as an FP32 pair
#pragma unroll 1
      for (int u = 0; u < 2; ++u) {
        const int l = w.l(u);
        float S[4], cmp[4], ctr[4];
        Cel Cl, Ch;
        Win W;
        load_cel(M.a32, w, l - 1, Cl);
        load_cel(M.a32, w, l, Ch);
        load_win(M.op, w, l, W);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          F2 pxy[2][2];
#pragma unroll
          for (int v = 0; v < 2; ++v)
#pragma unroll
            for (int q = 0; q < 2; ++q) pxy[v][q] = two_sum(Cl[q][t + v], Ch[q][t + v]);
          float S8 = pxy[0][0].h, E8 = pxy[0][0].l;
#pragma unroll
          for (int v = 0; v < 2; ++v)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              if (v == 0 && q == 0) continue;
              const F2 f = two_sum(S8, pxy[v][q].h);
              S8 = f.h;
              E8 += f.l + pxy[v][q].l;
            }
          ctr[t] = W[1][t + 1];
          const float c8h = 4.f * S8, c8l = 4.f * E8;
          S[t] = __fmul_rn(c8h, W[1][t + 1]);
          cmp[t] = __fmaf_rn(c8l, W[1][t + 1], __fmaf_rn(c8h, W[1][t + 1], -S[t]));
#pragma unroll
          for (int v = 0; v < 2; ++v)
#pragma unroll
            for (int q = 0; q < 2; ++q) res_term<true>(S[t], cmp[t], pxy[v][q], W[2 * q][t + 2 * v]);
        }
        auto side = [&](const Cel& C) {
#pragma unroll
          for (int t = 0; t < 4; ++t) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              res_term<true>(S[t], cmp[t], two_sum(C[q][t], C[q][t + 1]), W[2 * q][t + 1]);
              res_term<true>(S[t], cmp[t], two_sum(C[0][t + q], C[1][t + q]), W[1][t + 2 * q]);
            }
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
              for (int a = 0; a < 2; ++a) res_term1<true>(S[t], cmp[t], C[a][t + b], W[2 * a][t + 2 * b]);
          }
        };
        load_win(M.op, w, l - 1, W);
        side(Cl);
        load_win(M.op, w, l + 1, W);
        side(Ch);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float rn = 0.f;
          if (w.ok(u, t)) {
            const int g = w.node(l, t);
            const F2 axs = two_sum(S[t], cmp[t]);
            const float pp = __fmul_rn(axs.h, sch);
            const float pe = __fmaf_rn(axs.h, scl, __fmaf_rn(axs.l, sch, __fmaf_rn(axs.h, sch, -pp)));
            const float2 bv = rin[g];
            const F2 dd = two_sum(bv.x, -pp);
            const float e = dd.l + (bv.y - pe);
            rn = dd.h + e;
            A.rr[base + g] = make_float2(rn, e - (rn - dd.h));
            r[g] = rn;
            x[g] = step == 1 ? make_float2(ctr[t], 0.f) : pair_add(x[g], ctr[t]);
          }
          if (u == 0) rv[0][t] = rn;
          else rv[1][t] = rn;
        }
      }
      const double v = dot(rv, rv, 0);
      if (tid == 0) M.go = outer_go(o, v, A.tol2, A.cap);
      __syncthreads();
      if (M.go == 0) break;
      load_rh();
      __syncthreads();
    }
    if (A.fixed > 0 && step == A.fixed) break;
    const int inner = step == 0 ? A.inner : A.inner_next;
    last = inner;
    for (int it = 0;; ++it) {
      vcycle32(M, cl, w, L, r, dinv, A.omega, z, rv);
      push(z, 0);
      double v = dot(rv, z, 0);
      if (tid == 0) {
        if (it == 0) o.rz = v;
        M.bc = it == 0 ? 0.f : pcg_beta(o, v);
      }
      __syncthreads();
      const float be = M.bc;
      // p = z + beta p on the own and halo planes
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (w.ok(u, t)) {
            const int g = w.node(w.l(u), t);
            const float pv = it == 0 ? z[u][t] : fmaf(be, p[g], z[u][t]);
            p[g] = pv;
            M.op[w.at(w.l(u), t)] = pv;
          }
      if (hplane) {
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (w.row_ok(t)) {
            const int e = ho + w.at(0, t);
            const float pv = it == 0 ? M.t[e] : fmaf(be, M.ph[e], M.t[e]);
            M.ph[e] = pv;
            M.op[w.at(hl, t)] = pv;
          }
      }
      __syncthreads();
      float q[2][4];
      {
        float acc[2][4], ctr[2][4];
        apply_rows(M.op, M.a32, w, acc, ctr);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            q[u][t] = w.ok(u, t) ? scale * acc[u][t] : 0.f;
            z[u][t] = w.ok(u, t) ? ctr[u][t] : 0.f;  // p
          }
      }
      push(q, 2 * PL);
      v = dot(z, q, 1);
      if (tid == 0) M.bc = pcg_alpha(o, v);
      __syncthreads();
      al = M.bc;
      if (it == inner - 1) break;
      // d += alpha p, r -= alpha q
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (w.ok(u, t)) {
            const int g = w.node(w.l(u), t);
            d[g] = it == 0 ? al * z[u][t] : fmaf(al, z[u][t], d[g]);
            r[g] = fmaf(-al, q[u][t], r[g]);
          }
      if (hplane) {
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (w.row_ok(t)) {
            const int e = ho + w.at(0, t);
            M.dh[e] = it == 0 ? al * M.ph[e] : fmaf(al, M.ph[e], M.dh[e]);
            M.rh[e] = fmaf(-al, M.t[2 * PL + e], M.rh[e]);
          }
      }
      __syncthreads();
    }
    if (tid == 0) { o.iters += 1; o.pad += inner; }
  }
  if (rank == 0 && tid == 0) store_scalars(A.sc + s, o);
  cl.sync();  // no block leaves while others may still write to it
}

}  // namespace

cudaError_t vcycle32(const float* r, const float* a, const float* dinv, const float* const below[4], float* z,
                     const SolveScalars* sc, const Batch& bt, double omega, cudaStream_t st) {
  static SmemOptIn opt_in;
  const cudaError_t e = opt_in(k_vcycle32, sizeof(SmemV<float>));
  if (e != cudaSuccess) return e;
  VArgs A{r, a, dinv, below[0], below[1], below[2], below[3], z, sc, bt.act, (float)omega};
  const double bytes = (double)bt.n * 4 * (3.0 * kNodes + 32768 + 4096 + 512 + 64 + 8);
  return launch_cluster("vcycle32_f32", bytes, k_vcycle32, dim3((unsigned)bt.n * kC), dim3(kNT), kC, sizeof(SmemV<float>),
                        st, A);
}

cudaError_t solve32(SolverBufs& B, const float* a32, const __nv_bfloat16* abf, const float2* rr_in, long long rr_stride,
                    float2* x, const PcgParams& prm, int inner, int inner_next, int fixed_steps, cudaStream_t st) {
  static SmemOptIn opt_in;
  const cudaError_t e = opt_in(k_solve32, sizeof(SmemS));
  if (e != cudaSuccess) return e;
  SArgs A{};
  A.a32 = a32; A.abf = abf; A.dinv = (const float*)B.dinv[0];
  A.a16 = (const float*)B.acoef[1]; A.a8 = (const float*)B.acoef[2]; A.a4 = (const float*)B.acoef[3];
  A.a2 = (const float*)B.acoef[4];
  A.r = (float*)B.r; A.p = (float*)B.p; A.d = (float*)B.x;
  A.rr_in = rr_in; A.rr_stride = rr_stride; A.rr = B.bdf; A.x = x;
  A.sc = B.sc;
  A.tol2 = prm.rtol * prm.rtol;
  A.omega = (float)prm.omega;
  A.fixed = fixed_steps > 0 ? fixed_steps : 0;
  A.cap = fixed_steps > 0 ? fixed_steps : prm.max_iter;
  A.inner = inner;
  A.inner_next = inner_next;
  const double bytes = (double)B.S * (kNodes * (4.0 + 8 + 8) + 32768 * 6.0);
  return launch_cluster("solve32_f32", bytes, k_solve32, dim3((unsigned)B.S * kC), dim3(kNT), kC, sizeof(SmemS), st, A);
}

}  // namespace mlsgd
