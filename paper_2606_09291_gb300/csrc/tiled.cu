// tiled.cu - z-marching shared-memory kernels for the refinement residual on grids without
// a slab form and for Phi / the adjoint right-hand side (rows a4, a5), and the choice of
// the FP32 passes' family.
//
// Layout: a block of 32 x 8 threads owns a tile of interior nodes (x0 = 1 + 32 bx, y0 = 1 +
// (tile rows) by) and marches along z over a chunk of interior planes; each node plane is
// staged once into shared memory with a one-node halo by cp.async, so every value is read
// from HBM about once per pass (halos come from L2).  Node (lx, ly) of the staged plane is
// the global node (x0 - 1 + lx, y0 - 1 + ly).  Boundary nodes are zero-filled at staging
// (like nodes outside the grid) and not written.

#include "internal.cuh"
#include "kernels.h"
#include "launch.h"
#include "refine.cuh"

namespace mlsgd {

constexpr int TX = 32, TY = 8;
constexpr int NPX = TX + 2;                     // staged node row: 34 nodes
constexpr int NPY = TY + 2, NP = NPX * NPY;      // the Phi kernels' staged plane (one row per thread): 34 x 10
constexpr int NT = TX * TY;

// ---------------------------------------------------------------- async staging
// cp.async (4- or 8-byte, zero-filled when the source is outside the grid)
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem, bool valid) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int src = valid ? BYTES : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(sa), "l"(gmem), "n"(BYTES), "r"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Partial sums (dot products of the fused passes, Phi) are formed per segment of
// kZSeg interior planes, whatever z chunk the block marches: partial entry
// (seg * by + tile_y) * bx + tile_x of a sample holds the segment's block sum, so
// the reduction order, and with it every sample's iterates, is independent of the
// batch size that chose the z chunking.
constexpr int kZSeg = 8;

// The refinement residual on grids without a slab form: r = b - A x to FP64 accuracy with
// x = hi + lo and b as FP32 pairs and FP32 cells, error-free products and compensated sums
// (no FP64 instruction), rounded to FP32, and the partial r.r.  A tile of 32 x 16 nodes, two
// rows per thread; the window is read from the staged planes themselves (five of them: three
// in use, two in flight), so a plane takes one block barrier.  Bound by FP32 issue, some 400
// operations per node.
constexpr int kResRows = 2, kResTY = TY * kResRows, kResRing = 5;
constexpr int kResNP = NPX * (kResTY + 2);                         // staged nodes: 34 x 18
constexpr int kResCX = TX + 1, kResCP = kResCX * (kResTY + 1);     // staged cells: 33 x 17
constexpr size_t kResSmem = kResRing * (sizeof(float2) * kResNP + sizeof(float) * kResCP);
constexpr double kRes64OpsPerNode = 12 * 6 + 28 + 21 * 12 + 20;  // = 372 (see tiled_res64)

struct ResArgs {
  const float2 *x, *b;
  const float* a;
  float* r;
  double* partial;
  const SolveScalars* sc;
  const int* act;
  long long bstride;  // 0: one b for every sample
  int N, nzc, zc, nseg;
};

__global__ void __launch_bounds__(NT) k_res64(ResArgs A) {
  pdl_entry();
  constexpr int RY = kResRows;
  constexpr int MN = (kResNP + NT - 1) / NT, MC = (kResCP + NT - 1) / NT;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* xs = reinterpret_cast<float2*>(smraw);
  float* cs = reinterpret_cast<float*>(smraw + kResRing * sizeof(float2) * kResNP);
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int N = A.N, n1 = N + 1;
  const int chunk = blockIdx.z % A.nzc;
  const int s = A.act != nullptr ? A.act[blockIdx.z / A.nzc] : (int)(blockIdx.z / A.nzc);
  if (A.sc != nullptr && !A.sc[s].active) return;
  const int x0 = 1 + TX * blockIdx.x, y0 = 1 + kResTY * blockIdx.y;
  const long long pn = (long long)n1 * n1, pc = (long long)N * N, nodes = pn * n1;
  const int kbeg = 1 + chunk * A.zc, kend = min(N - 1, kbeg + A.zc - 1);
  const float2* xg = A.x + s * nodes;
  const float* ag = A.a + s * pc * N;
  int noff[MN], coff[MC];  // offsets in a plane, -1: zero-filled
#pragma unroll
  for (int j = 0; j < MN; ++j) {
    const int e = tid + j * NT, gi = x0 - 1 + e % NPX, gj = y0 - 1 + e / NPX;
    noff[j] = (gi > 0 && gj > 0 && gi < N && gj < N) ? gi + n1 * gj : -1;
  }
#pragma unroll
  for (int j = 0; j < MC; ++j) {
    const int e = tid + j * NT, gi = x0 - 1 + e % kResCX, gj = y0 - 1 + e / kResCX;
    coff[j] = (gi < N && gj < N) ? gi + N * gj : -1;
  }
  auto issue = [&](int m, int slot) {  // node plane m, cell plane m
    const bool mok = m > 0 && m < N, cok = m < N;
    const float2* xb = xg + (mok ? m * pn : 0);
    const float* ab = ag + (cok ? m * pc : 0);
#pragma unroll
    for (int j = 0; j < MN; ++j) {
      const int e = tid + j * NT;
      const bool ok = mok && noff[j] >= 0;
      if (j < MN - 1 || e < kResNP) cp_async<8>(xs + slot * kResNP + e, xb + (ok ? noff[j] : 0), ok);
    }
#pragma unroll
    for (int j = 0; j < MC; ++j) {
      const int e = tid + j * NT;
      const bool ok = cok && coff[j] >= 0;
      if (j < MC - 1 || e < kResCP) cp_async<4>(cs + slot * kResCP + e, ab + (ok ? coff[j] : 0), ok);
    }
    cp_async_commit();
  };
  for (int m = kbeg - 1; m <= kbeg + 2; ++m) issue(m, m % kResRing);  // planes past N are zero-filled
  const int gi = x0 + tx, gj0 = y0 + RY * ty;
  const bool colok = gi < N;
  const int xb = tx + NPX * RY * ty, cbn = tx + kResCX * RY * ty;
  const float2* bptr = A.b + s * A.bstride + gi + (long long)n1 * gj0;
  float* r32o = A.r + s * nodes + gi + (long long)n1 * gj0;
  float redf = 0.f;
  const double scd = 1.0 / (12.0 * N);
  const float sch = (float)scd, scl = (float)(scd - (double)sch);  // h/12 as an FP32 pair
  int sl[3] = {(kbeg - 1) % kResRing, kbeg % kResRing, (kbeg + 1) % kResRing};  // slots of planes k - 1, k, k + 1
  for (int k = kbeg; k <= kend; ++k) {
    float2 bv[RY];
#pragma unroll
    for (int t = 0; t < RY; ++t)
      bv[t] = (colok && gj0 + t < N) ? bptr[pn * k + n1 * t] : make_float2(0.f, 0.f);
    cp_async_wait<1>();  // plane k + 1 has landed
    __syncthreads();     // for every thread; plane k - 2 is no longer read
    issue(k + 3, sl[2] + 2 >= kResRing ? sl[2] + 2 - kResRing : sl[2] + 2);
    if (colok) {
      float2 X[3][3][RY + 2];
      float C[2][2][RY + 1];
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) {
        const float2* xp = xs + sl[pl] * kResNP + xb;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int rr = 0; rr < RY + 2; ++rr) X[pl][c][rr] = xp[c + NPX * rr];
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float* cp = cs + sl[r] * kResCP + cbn;
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
          for (int cr = 0; cr < RY + 1; ++cr) C[r][p][cr] = cp[p + kResCX * cr];
      }
#pragma unroll
      for (int t = 0; t < RY; ++t) {
        if (gj0 + t >= N) break;
        F2 pxy[2][2], pxz[2][2], pyz[2][2];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            pxy[v][u] = two_sum(C[0][u][t + v], C[1][u][t + v]);
            pxz[v][u] = two_sum(C[v][u][t], C[v][u][t + 1]);
            pyz[v][u] = two_sum(C[v][0][t + u], C[v][1][t + u]);
          }
        float S8 = 0.f, E8 = 0.f;
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const F2 q = two_sum(S8, pxy[v][u].h);
            S8 = q.h;
            E8 += q.l + pxy[v][u].l;
          }
        float S = 0.f, comp = 0.f;
        df_term<false>(S, comp, F2{4.f * S8, 4.f * E8}, X[1][1][t + 1]);
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int u = 0; u < 2; ++u) df_term<true>(S, comp, pxy[v][u], X[1][2 * u][t + 2 * v]);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int pl = 2 * r;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            df_term<true>(S, comp, pxz[r][u], X[pl][2 * u][t + 1]);
            df_term<true>(S, comp, pyz[r][u], X[pl][1][t + 2 * u]);
          }
#pragma unroll
          for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int p = 0; p < 2; ++p) df_term<true>(S, comp, F2{C[r][p][t + q], 0.f}, X[pl][2 * p][t + 2 * q]);
        }
        // ax = (S + comp) (sch + scl), a pair (p, pe)
        const F2 axs = two_sum(S, comp);
        const float p = __fmul_rn(axs.h, sch);
        const float pe = __fmaf_rn(axs.h, scl, __fmaf_rn(axs.l, sch, __fmaf_rn(axs.h, sch, -p)));
        const long long o = pn * k + n1 * t;
        const F2 d = two_sum(bv[t].x, -p);
        const float rv = d.h + (d.l + (bv[t].y - pe));
        r32o[o] = rv;  // the inner solve's FP32 residual
        redf = __fmaf_rn(rv, rv, redf);
      }
    }
    if (k == kend || (k - 1) % kZSeg == kZSeg - 1) {  // end of a partial-sum segment (block-uniform)
      const double b = block_sum((double)redf);
      if (tid == 0)
        A.partial[(long long)s * (gridDim.x * gridDim.y * A.nseg) +
                  (((k - 1) / kZSeg) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = b;
      redf = 0.f;
    }
    sl[0] = sl[1];
    sl[1] = sl[2];
    sl[2] = sl[2] == kResRing - 1 ? 0 : sl[2] + 1;
  }
  cp_async_wait<0>();
}

// Phi = 1/2 e^T M e and badj = M e on interior rows, e = y - g_h (row a5).
// The consistent Q1 mass is (h/6)^3 [1 4 1] x [1 4 1] x [1 4 1]: a staged plane of
// y is summed along x, then y, into the tile; three such planes combine along z.
// g_h = gx(i) gx(j) gx(k) and M g_h = mg(i) mg(j) mg(k) are separable, so they
// come from the 1D tables gtab[i] = sin(pi i / N) (0 at i = 0, N) and
// mgtab[i] = (h/6)(g[i-1] + 4 g[i] + g[i+1]).
__global__ void __launch_bounds__(NT) k_phi_tiled(const double* __restrict__ y, int N, const double* __restrict__ gtab,
                                                  const double* __restrict__ mgtab, double* __restrict__ badj,
                                                  double* __restrict__ partial, int nzc, int zc, int nseg) {
  pdl_entry();
  __shared__ double ys[NP];
  __shared__ double xsum[NPY][TX];
  __shared__ double mxy[3][NT];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int n1 = N + 1;
  const int s = blockIdx.z / nzc, chunk = blockIdx.z % nzc;
  const int x0 = 1 + TX * blockIdx.x, y0 = 1 + TY * blockIdx.y;
  const long long nodes = (long long)n1 * n1 * n1;
  const double* yb = y + s * nodes;
  const int kbeg = 1 + chunk * zc;
  const int kend = min(N - 1, kbeg + zc - 1);
  const int gi = x0 + tx, gj = y0 + ty;
  const bool mine = gi < N && gj < N;
  double ycen[3] = {0.0, 0.0, 0.0};
  auto advance = [&](int m) {
    for (int e = tid; e < NP; e += NT) {
      const int lx = e % NPX, ly = e / NPX;
      const int i = x0 - 1 + lx, j = y0 - 1 + ly;
      ys[e] = (m >= 0 && m <= N && i <= N && j <= N) ? yb[i + (long long)n1 * (j + (long long)n1 * m)] : 0.0;
    }
    __syncthreads();
    for (int e = tid; e < NPY * TX; e += NT) {
      const int ly = e / TX, lx = e % TX;
      const double* row = ys + NPX * ly + lx;
      xsum[ly][lx] = row[0] + 4.0 * row[1] + row[2];
    }
    ycen[(m + 3) % 3] = ys[(tx + 1) + NPX * (ty + 1)];
    __syncthreads();
    mxy[(m + 3) % 3][tid] = xsum[ty][tx] + 4.0 * xsum[ty + 1][tx] + xsum[ty + 2][tx];
    __syncthreads();
  };
  const double h6 = 1.0 / (6.0 * N), h63 = h6 * h6 * h6;
  double red = 0.0;
  advance(kbeg - 1);
  advance(kbeg);
  for (int k = kbeg; k <= kend; ++k) {
    advance(k + 1);
    if (mine) {
      const double my = mxy[(k + 2) % 3][tid] + 4.0 * mxy[k % 3][tid] + mxy[(k + 1) % 3][tid];
      const double me = h63 * my - mgtab[gi] * mgtab[gj] * mgtab[k];
      const double e = ycen[k % 3] - gtab[gi] * gtab[gj] * gtab[k];
      badj[s * nodes + gi + (long long)n1 * (gj + (long long)n1 * k)] = me;
      red += e * me;
    }
    if (k == kend || (k - 1) % kZSeg == kZSeg - 1) {  // end of a partial-sum segment
      const double b = block_sum(red);
      if (tid == 0)
        partial[(long long)s * (gridDim.x * gridDim.y * nseg) + (((k - 1) / kZSeg) * gridDim.y + blockIdx.y) * gridDim.x +
                blockIdx.x] = b;
      red = 0.0;
      __syncthreads();
    }
  }
}

// k_phi_tiled for a state given as FP32 (hi, lo) pairs (the mixed level gradient):
// the same separable sums in pair arithmetic (no FP64 instruction), the 1D tables as
// pairs, M e written as pairs (the adjoint solve's right-hand side), the partial
// e.M e of each block returned in FP64.  Each thread takes kPhiRows rows of a
// 32 x (8 kPhiRows) tile, so the three block barriers of a plane serve four nodes;
// the staged plane is double-buffered and plane m + 1 is copied asynchronously while
// plane m is summed.
constexpr int kPhiRows = 4;
constexpr int kPhiTY = TY * kPhiRows;                        // tile rows
constexpr int kPhiNPY = kPhiTY + 2, kPhiNP = NPX * kPhiNPY;  // staged plane with halo
constexpr size_t kPhiSmem = sizeof(float2) * (2 * kPhiNP + kPhiNPY * TX + 3 * kPhiTY * TX);
__global__ void __launch_bounds__(NT) k_phi_tiled_df(const float2* __restrict__ y, int N, const float2* __restrict__ gtab,
                                                     const float2* __restrict__ mgtab, float2* __restrict__ badj,
                                                     double* __restrict__ partial, int nzc, int zc, int nseg) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smp[];
  float2* ysb = reinterpret_cast<float2*>(smp);  // [2][kPhiNP]: plane m in buffer m & 1
  float2(*xsum)[TX] = reinterpret_cast<float2(*)[TX]>(ysb + 2 * kPhiNP);                   // [kPhiNPY][TX]
  float2(*mxy)[kPhiTY][TX] = reinterpret_cast<float2(*)[kPhiTY][TX]>(ysb + 2 * kPhiNP + kPhiNPY * TX);  // [3]
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int n1 = N + 1;
  const int s = blockIdx.z / nzc, chunk = blockIdx.z % nzc;
  const int x0 = 1 + TX * blockIdx.x, y0 = 1 + kPhiTY * blockIdx.y;
  const long long nodes = (long long)n1 * n1 * n1;
  const float2* yb = y + s * nodes;
  const int kbeg = 1 + chunk * zc;
  const int kend = min(N - 1, kbeg + zc - 1);
  const int gi = x0 + tx;
  const int ly0 = kPhiRows * ty;  // the thread's first tile row
  DF yc[kPhiRows], yn[kPhiRows];  // y at the thread's nodes of planes k and k + 1
  auto four = [](DF a) { return DF{4.f * a.h, 4.f * a.l}; };  // exact
  auto load = [&](int m) {  // plane m into buffer m & 1 (zeros outside the grid)
    float2* ys = ysb + (m & 1) * kPhiNP;
    for (int e = tid; e < kPhiNP; e += NT) {
      const int lx = e % NPX, ly = e / NPX;
      const int i = x0 - 1 + lx, j = y0 - 1 + ly;
      const bool ok = m >= 0 && m <= N && i <= N && j <= N;
      cp_async<8>(ys + e, ok ? yb + i + (long long)n1 * (j + (long long)n1 * m) : yb, ok);
    }
    cp_async_commit();
  };
  // plane m (copied by load(m)) into the x and xy sums; copies plane m + 1 meanwhile
  // (into the buffer of plane m - 1, whose last reads precede the first barrier)
  auto advance = [&](int m, DF* ycen) {
    const int r3 = (m + 3) % 3;
    const float2* ys = ysb + (m & 1) * kPhiNP;
    cp_async_wait<0>();
    __syncthreads();
    if (m + 1 <= kend + 1) load(m + 1);
    for (int e = tid; e < kPhiNPY * TX; e += NT) {
      const int ly = e / TX, lx = e % TX;
      const float2* row = ys + NPX * ly + lx;
      xsum[ly][lx] = df_f2(df_add(df_add(df_make(row[0]), df_make(row[2])), four(df_make(row[1]))));
    }
#pragma unroll
    for (int t = 0; t < kPhiRows; ++t) ycen[t] = df_make(ys[(tx + 1) + NPX * (ly0 + t + 1)]);
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kPhiRows; ++t) {
      const int ly = ly0 + t;
      mxy[r3][ly][tx] =
          df_f2(df_add(df_add(df_make(xsum[ly][tx]), df_make(xsum[ly + 2][tx])), four(df_make(xsum[ly + 1][tx]))));
    }
    __syncthreads();
  };
  const double h6 = 1.0 / (6.0 * N);
  const DF h63 = df_make(df_split(h6 * h6 * h6));
  DF red{0.f, 0.f};
  load(kbeg - 1);
  advance(kbeg - 1, yn);
  advance(kbeg, yc);
  const DF mgi = gi < N ? df_make(mgtab[gi]) : DF{0.f, 0.f}, ggi = gi < N ? df_make(gtab[gi]) : DF{0.f, 0.f};
  for (int k = kbeg; k <= kend; ++k) {
    advance(k + 1, yn);
    const DF mgk = df_make(mgtab[k]), ggk = df_make(gtab[k]);
#pragma unroll
    for (int t = 0; t < kPhiRows; ++t) {
      const int gj = y0 + ly0 + t;
      if (gi < N && gj < N) {
        const DF my = df_add(df_add(df_make(mxy[(k + 2) % 3][ly0 + t][tx]), df_make(mxy[(k + 1) % 3][ly0 + t][tx])),
                             four(df_make(mxy[k % 3][ly0 + t][tx])));
        const DF mg3 = df_mul(df_mul(mgi, df_make(mgtab[gj])), mgk);
        const DF g3 = df_mul(df_mul(ggi, df_make(gtab[gj])), ggk);
        const DF me = df_add(df_mul(h63, my), df_neg(mg3));
        const DF e = df_add(yc[t], df_neg(g3));
        badj[s * nodes + gi + (long long)n1 * (gj + (long long)n1 * k)] = df_f2(me);
        red = df_add(red, df_mul(e, me));
      }
    }
#pragma unroll
    for (int t = 0; t < kPhiRows; ++t) yc[t] = yn[t];
    if (k == kend || (k - 1) % kZSeg == kZSeg - 1) {  // end of a partial-sum segment
      const double b = block_sum(df_to_double(red));
      if (tid == 0)
        partial[(long long)s * (gridDim.x * gridDim.y * nseg) + (((k - 1) / kZSeg) * gridDim.y + blockIdx.y) * gridDim.x +
                blockIdx.x] = b;
      red = DF{0.f, 0.f};
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------- host side

TiledShape tiled_shape(int N, int S, int ry, int zchunks) {
  TiledShape t;
  t.bx = (N - 1 + TX - 1) / TX;
  t.by = (N - 1 + TY * ry - 1) / (TY * ry);
  // enough blocks to fill the GPU: split z into chunks of whole partial-sum segments
  // when the batch is small (the partial-sum layout does not depend on the split)
  const int nseg = (N - 1 + kZSeg - 1) / kZSeg;
  const long long base = (long long)t.bx * t.by * S;
  int nzc = 1;
  if (zchunks > 0) nzc = zchunks < nseg ? zchunks : nseg;
  else
    while (base * nzc < 4 * 152 * 4 && 2 * nzc <= nseg) nzc *= 2;
  const int spc = (nseg + nzc - 1) / nzc;  // segments per chunk
  t.nzc = (nseg + spc - 1) / spc;
  t.zc = spc * kZSeg;
  t.nseg = nseg;
  t.blocks_per_sample = t.bx * t.by * nseg;  // partial-sum entries per sample
  return t;
}

static double vbytes(int N, int S, double vec, double coef) {
  return (double)S * (vec * (double)nodes_of(N) * 4 + coef * (double)cells_of(N) * 4);
}

// p is double-buffered: neighbouring tiles read the old p in their halos while
// this tile writes the new one.
// FP32 vectors on 32^3 and 64^3 grids go to the whole-row slab passes (slab.cu)
static bool slab_pass(int N, const Batch& bt) { return bt.stencil == 0 && slab_supported(N); }
void tiled_apply(const float* z, const float* pold, float* pnew, const float* a, float* q, double* partial,
                 const SolveScalars* sc, int N, const Batch& bt, int first, cudaStream_t st) {
  if (slab_pass(N, bt)) slab_apply(z, pold, pnew, a, q, nullptr, partial, sc, N, bt, first != 0, false, false, st);
  else tile32_apply(z, pold, pnew, a, q, nullptr, partial, sc, N, bt, first != 0, false, st);
}
// fused variants of the mixed inner solve: x += alpha_prev p_old, and PREU
void tiled_apply_x(const float* z, const float* pold, float* pnew, const float* a, float* q, float* x, double* partial,
                   const SolveScalars* sc, int N, const Batch& bt, cudaStream_t st, bool x_first) {
  if (slab_pass(N, bt)) slab_apply(z, pold, pnew, a, q, x, partial, sc, N, bt, false, true, x_first, st);
  else tile32_apply(z, pold, pnew, a, q, x, partial, sc, N, bt, false, x_first, st);
}
bool tiled_pre_update(const float* r, const float* q, const __nv_bfloat16* a, const float* dinv, float* t,
                      float* rnew, float* rc, const SolveScalars* sc, int N, const Batch& bt, cudaStream_t st) {
  if (slab_pass(N, bt)) {
    slab_pre<__nv_bfloat16>(r, q, a, dinv, rnew, rc, sc, N, bt, st);
    return true;
  }
  tile32_pre<__nv_bfloat16>(r, q, a, dinv, t, rnew, sc, N, bt, st);
  return false;
}
template <typename TA>
bool tiled_pre(const float* r, const TA* a, const float* dinv, float* t, float* rc, const SolveScalars* sc, int N,
               const Batch& bt, cudaStream_t st) {
  if (slab_pass(N, bt)) {
    slab_pre<TA>(r, nullptr, a, dinv, nullptr, rc, sc, N, bt, st);
    return true;
  }
  tile32_pre<TA>(r, nullptr, a, dinv, t, nullptr, sc, N, bt, st);
  return false;
}
template <typename TA>
void tiled_post(const float* r, const TA* a, const float* dinv, const float* ec, float* z, double* partial,
                const SolveScalars* sc, int N, const Batch& bt, cudaStream_t st) {
  if (slab_pass(N, bt)) slab_post<TA>(r, a, dinv, ec, z, partial, sc, N, bt, st);
  else tile32_post<TA>(r, a, dinv, ec, z, partial, sc, N, bt, st);
}

// The z chunks follow the number of samples launched; the partial sums do not depend on them.
void tiled_res64(const float2* b, long long bstride, const float2* x, const float* a, float* r32, double* partial,
                 const SolveScalars* sc, int N, const Batch& bt, cudaStream_t st) {
  const TiledShape t = tiled_shape(N, bt.n, kResRows, bt.zchunks);
  const ResArgs A{x, b, a, r32, partial, sc, bt.act, bstride, N, t.nzc, t.zc, t.nseg};
  const double bb = (double)(bstride ? bt.n : 1) * nodes_of(N) * 8;
  // FP32 operations per interior node as written (no sharing between nodes): 12 exact
  // cell-pair sums (6 each), the 8-cell sum (28), 21 compensated product terms (12
  // each), the scaling, the subtraction from b and r.r (20)
  const double ops = (double)bt.n * (N - 1) * (N - 1) * (N - 1) * kRes64OpsPerNode;
  static_assert(kResSmem <= 48 * 1024, "no opt-in");
  launch_flops("resid64", bb + vbytes(N, bt.n, 3, 1), ops, k_res64, dim3(t.bx, t.by, (unsigned)(bt.n * t.nzc)),
               dim3(TX, TY), kResSmem, st, A);
}

int tiled_phi_df(const float2* y, int N, int S, const float2* gtab, const float2* mgtab, float2* badj,
                 double* partial, cudaStream_t st) {
  const TiledShape t = tiled_shape(N, S, kPhiRows);
  static SmemOptIn opt_in;
  (void)opt_in(k_phi_tiled_df, kPhiSmem);  // a launch without it is refused
  launch("phi_adjrhs", (double)S * nodes_of(N) * 16, k_phi_tiled_df, dim3(t.bx, t.by, (unsigned)(S * t.nzc)),
         dim3(TX, TY), kPhiSmem, st, y, N, gtab, mgtab, badj, partial, t.nzc, t.zc, t.nseg);
  return t.blocks_per_sample;
}

int tiled_phi(const double* y, int N, int S, const double* gtab, const double* mgtab, double* badj, double* partial,
              cudaStream_t st) {
  const TiledShape t = tiled_shape(N, S, 1);
  launch("phi_adjrhs", (double)S * nodes_of(N) * 16, k_phi_tiled, dim3(t.bx, t.by, (unsigned)(S * t.nzc)),
         dim3(TX, TY), 0, st, y, N, gtab, mgtab, badj, partial, t.nzc, t.zc, t.nseg);
  return t.blocks_per_sample;
}

template bool tiled_pre<__nv_bfloat16>(const float*, const __nv_bfloat16*, const float*, float*, float*,
                                       const SolveScalars*, int, const Batch&, cudaStream_t);
template bool tiled_pre<float>(const float*, const float*, const float*, float*, float*, const SolveScalars*, int,
                               const Batch&, cudaStream_t);
template void tiled_post<__nv_bfloat16>(const float*, const __nv_bfloat16*, const float*, const float*, float*, double*,
                                        const SolveScalars*, int, const Batch&, cudaStream_t);
template void tiled_post<float>(const float*, const float*, const float*, const float*, float*, double*,
                                const SolveScalars*, int, const Batch&, cudaStream_t);

int tiled_blocks_per_sample(int N, int S, bool slab) {
  return slab && slab_supported(N) ? slab_shape(N, S).blocks_per_sample : tiled_shape(N, S, 4).blocks_per_sample;
}
int res64_blocks_per_sample(int N, int S) { return tiled_shape(N, S, kResRows).blocks_per_sample; }

}  // namespace mlsgd
