// estimator.cu - right-hand sides, Phi, B*q, entropic weights, level
// differences, Chan statistics and the multilevel step (rows a3, a5, a7-a10).
#include <math.h>

#include <algorithm>

#include <type_traits>

#include "internal.cuh"
#include "kernels.h"
#include "launch.h"

namespace mlsgd {

// Passes over the control cells march over them with at most kCellBlocks blocks, so that
// what is the same for every cell, and the FP64 block reductions (five additions per
// warp, as much as the cell's own work), are paid once per block.
constexpr int kCellBlocks = 8 * 152;  // eight blocks of 256 threads per SM
static int cell_blocks(long long n) {
  const long long b = (n + kBlock - 1) / kBlock;
  return (int)(b < kCellBlocks ? b : kCellBlocks);
}

// (B z)_n = int z phi_n (<B u, v> = int u v, Sec. 5) for a cellwise-constant control
// z on the control grid Nc.
//
// Control coarser than the grid (N = r Nc): each of the 8 cells around node n lies in
// one control cell (its parent) and int_e phi_n = h^3 / 8.
__global__ void k_rhs_state(const double* __restrict__ z, int Nc, int N, double* __restrict__ b) {
  pdl_entry();
  const int n1 = N + 1;
  const long long nodes = (long long)n1 * n1 * n1;
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nodes) return;
  int i, j, k;
  node_ijk(n, n1, i, j, k);
  double acc = 0.0;
  if (interior(i, j, k, N)) {
    const int r = N / Nc;
    for (int dz = -1; dz <= 0; ++dz)
      for (int dy = -1; dy <= 0; ++dy)
        for (int dx = -1; dx <= 0; ++dx)
          acc += z[(i + dx) / r + (long long)Nc * ((j + dy) / r + (long long)Nc * ((k + dz) / r))];
    const double h = 1.0 / N;
    acc *= 0.125 * h * h * h;
  }
  b[n] = acc;
}

// Control grid at least as fine as the grid (Nc = r N): the midpoint rule on each
// control cell c is exact for the multilinear phi_n, so (B z)_n = h_c^3 sum_c z_c
// phi_n(x_c) over the (2r)^3 control cells of the support.  phi_n(x_c) is a product of
// one hat weight per axis: t = (m + 1/2) / r for the right and 1 - t for the left node of
// the level cell that holds the m-th control cell along the axis.
//
// Bound: FP64 issue, then one read of z.  Contracted axis by axis every control cell
// costs two FMAs (to the two nodes of its level cell along y), where contracting the
// (2r)^2 rows of each node row's support costs 4 (and reads z four times).
// k_rhs_xy: one block per (level cell row ey, control plane z0 + cz) contracts y, then x,
// into u[cz][ey][side][i]; k_rhs_z contracts z, slab after slab of the control planes that u
// has room for (the order of the sums does not depend on the slabs).  A 256^3 control onto
// 8^3: 615 us by node rows, about 105 us by axis; a whole FP64 state and adjoint solve of one
// 8^3 sample under it 862 and 343 us.
__global__ void __launch_bounds__(kBlock) k_rhs_xy(const double* __restrict__ z, int Nc, int N, int z0,
                                                   double* __restrict__ u) {
  pdl_entry();
  extern __shared__ double sm[];  // t[r], left and right sums [2][Nc]
  const int r = Nc / N, n1 = N + 1;
  double* t = sm;
  double* col = sm + r;
  const int ey = blockIdx.x, cz = blockIdx.y;
  const double inv_r = 1.0 / r;
  for (int m = threadIdx.x; m < r; m += blockDim.x) t[m] = (m + 0.5) * inv_r;
  __syncthreads();
  const double* zp = z + (long long)Nc * ((long long)r * ey + (long long)Nc * (z0 + cz));
  for (int cx = threadIdx.x; cx < Nc; cx += blockDim.x) {
    double all = 0.0, right = 0.0;
#pragma unroll 4
    for (int m = 0; m < r; ++m) {
      const double v = zp[(long long)Nc * m + cx];
      all += v;
      right = fma(t[m], v, right);
    }
    col[cx] = all - right;
    col[Nc + cx] = right;
  }
  __syncthreads();
  double* ub = u + ((long long)cz * N + ey) * 2 * n1;
  for (int e = threadIdx.x; e < 2 * n1; e += blockDim.x) {
    const int side = e / n1, i = e - side * n1;
    double v = 0.0;
    if (i > 0 && i < N) {
      const double* cp = col + side * Nc + r * (i - 1);
      for (int m = 0; m < r; ++m) v = fma(t[m], cp[m], fma(1.0 - t[m], cp[m + r], v));
    }
    ub[e] = v;
  }
}
// node (i, j, k): the right side of cell row j - 1 and the left side of row j, over those of
// its 2r control planes that are among z0 .. z0 + planes - 1; b holds the sum so far between
// two slabs.  One warp per block: a warp alone issues an FP64 operation in 64 clocks and eight
// of an SM share its pipe, so the few nodes of a coarse grid are spread over SMs (8^3 under
// 256^3: 15 us less than with 256 threads a block).
constexpr int kRhsZBlock = 32;
__global__ void __launch_bounds__(kRhsZBlock) k_rhs_z(const double* __restrict__ u, int Nc, int N, int z0, int planes,
                                                  double* __restrict__ b) {
  pdl_entry();
  const int n1 = N + 1, r = Nc / N;
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= n1 * n1 * n1) return;
  int i, j, k;
  node_ijk(n, n1, i, j, k);
  if (!interior(i, j, k, N)) {
    if (z0 == 0) b[n] = 0.0;
    return;
  }
  const int first = r * (k - 1), m0 = max(0, z0 - first), m1 = min(2 * r, z0 + planes - first);
  if (m0 >= m1) return;
  const long long plane = (long long)N * 2 * n1;
  const double* up = u + (long long)(first + m0 - z0) * plane + (long long)(2 * (j - 1) + 1) * n1 + i;
  const double inv_r = 1.0 / r;
  double v = m0 > 0 ? b[n] : 0.0;
#pragma unroll 8
  for (int m = m0; m < m1; ++m, up += plane) {
    const double w = m < r ? (m + 0.5) * inv_r : 2.0 - (m + 0.5) * inv_r;
    v = fma(w, up[0] + up[n1], v);
  }
  const double hc = 1.0 / Nc;
  if (m1 == 2 * r) v *= hc * hc * hc;
  b[n] = v;
}
// Control and level grid equal: (B z)_n = h^3 / 8 sum of the eight cells, summed along y,
// z and x in that order (the order of k_rhs_rows, whose weights are all 1/2 here).  One
// thread per node column marches over kRhsPlanes planes; a plane's sums serve two nodes.
constexpr int kRhsPlanes = 16;
__global__ void __launch_bounds__(kBlock) k_rhs_equal(const double* __restrict__ z, int N, double* __restrict__ b) {
  pdl_entry();
  const int n1 = N + 1;
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= n1 * n1) return;
  const int j = col / n1, i = col - j * n1;
  const int k0 = kRhsPlanes * (int)blockIdx.y, k1 = min(N, k0 + kRhsPlanes - 1);
  const long long pn = (long long)n1 * n1, pc = (long long)N * N;
  double* o = b + pn * k0 + col;
  const bool in = i > 0 && j > 0 && i < N && j < N;
  const double* c = z + (in ? (i - 1) + (long long)N * (j - 1) : 0);
  const double h = 1.0 / N, w = 0.125 * (h * h * h);
  double lo0 = 0.0, lo1 = 0.0;  // y sums of the cell columns i - 1 and i in the plane below
  if (in && k0 > 0) {
    const double* p = c + pc * (k0 - 1);
    lo0 = p[0] + p[N];
    lo1 = p[1] + p[N + 1];
  }
  c += pc * k0;
  for (int k = k0; k <= k1; ++k, o += pn, c += pc) {
    double v = 0.0;
    if (in && k < N) {
      const double up0 = c[0] + c[N], up1 = c[1] + c[N + 1];
      if (k > 0) v = w * ((lo0 + up0) + (lo1 + up1));
      lo0 = up0;
      lo1 = up1;
    }
    *o = v;
  }
}

// The by-axis form from r = Nc / N = 8 on.  Below, the node rows, which need no scratch, are as
// fast or faster: at r = 2 145 against 156 us of FP64 issue for a 256^3 control on 128^3, at
// r = 4 a state and adjoint solve of one 64^3 sample under a 256^3 control 1912 against 1934 us
// (mixed), 3919 against 3947 (FP64), of 8^3 to 32^3 the same within 0.5%.
constexpr int kRhsAxisR = 8;

// The form of r = 2 and 4: one block per node row (j, k); threads along cx contract the
// (2r)^2 control rows (cy, cz) of the row's support with w(y) w(z) into a column sum per
// cx, then each node i of the row contracts its 2r columns with w(x).
__global__ void __launch_bounds__(kBlock) k_rhs_rows(const double* __restrict__ z, int Nc, int N,
                                                     double* __restrict__ b) {
  pdl_entry();
  extern __shared__ double sm[];  // w[2r], col[Nc]
  const int n1 = N + 1, r = Nc / N, w2 = 2 * r;
  const int j = blockIdx.x, k = blockIdx.y;
  double* brow = b + (long long)n1 * (j + (long long)n1 * k);
  if (j == 0 || j == N || k == 0 || k == N) {
    for (int i = threadIdx.x; i < n1; i += blockDim.x) brow[i] = 0.0;
    return;
  }
  double* w = sm;
  double* col = sm + w2;
  const double inv_r = 1.0 / r;
  for (int m = threadIdx.x; m < w2; m += blockDim.x) w[m] = 1.0 - fabs((m + 0.5) * inv_r - 1.0);
  __syncthreads();
  const long long y0 = (long long)r * (j - 1), z0 = (long long)r * (k - 1);
  for (int cx = threadIdx.x; cx < Nc; cx += blockDim.x) {
    double acc = 0.0;
    for (int mz = 0; mz < w2; ++mz) {
      const double* zp = z + cx + (long long)Nc * (y0 + (long long)Nc * (z0 + mz));
      double accz = 0.0;
      for (int my = 0; my < w2; ++my) accz = fma(w[my], zp[(long long)Nc * my], accz);
      acc = fma(w[mz], accz, acc);
    }
    col[cx] = acc;
  }
  __syncthreads();
  const double hc = 1.0 / Nc;
  const double hc3 = hc * hc * hc;
  for (int i = threadIdx.x; i < n1; i += blockDim.x) {
    double v = 0.0;
    if (i > 0 && i < N) {
      const double* cp = col + r * (i - 1);
      for (int m = 0; m < w2; ++m) v = fma(w[m], cp[m], v);
      v *= hc3;
    }
    brow[i] = v;
  }
}

size_t rhs_slab_bytes(int Nc, int N) {  // u of all control planes
  return Nc >= kRhsAxisR * N ? (size_t)Nc * N * 2 * (N + 1) * sizeof(double) : 0;
}

// scratch: memory the launch may overwrite, at least 16 N (N + 1) bytes (a control plane of u)
void launch_rhs_state(const double* z, int Nc, int N, double* b, void* scratch, size_t scratch_bytes,
                      cudaStream_t st) {
  const double bytes = (double)cells_of(Nc) * 8 + (double)nodes_of(N) * 8;
  if (N > Nc) {
    launch("rhs", bytes, k_rhs_state, dim3(node_blocks(N)), kBlock, 0, st, z, Nc, N, b);
  } else if (N == Nc) {
    launch("rhs", bytes, k_rhs_equal,
           dim3((unsigned)(((N + 1) * (N + 1) + kBlock - 1) / kBlock), (unsigned)((N + kRhsPlanes) / kRhsPlanes)), kBlock,
           0, st, z, N, b);
  } else if (Nc >= kRhsAxisR * N) {
    // slabs of control planes, as many and as equal as the scratch asks for
    const size_t plane = (size_t)N * 2 * (N + 1) * sizeof(double);
    const int fit = (int)std::min<size_t>(Nc, std::max<size_t>(1, scratch_bytes / plane));
    const int slabs = (Nc + fit - 1) / fit, planes = (Nc + slabs - 1) / slabs;
    double* u = (double*)scratch;
    for (int z0 = 0; z0 < Nc; z0 += planes) {
      const int n = std::min(planes, Nc - z0);
      const double ub = (double)n * plane;
      launch("rhs", (double)n * Nc * Nc * 8 + ub, k_rhs_xy, dim3((unsigned)N, (unsigned)n), kBlock,
             (size_t)(Nc / N + 2 * Nc) * sizeof(double), st, z, Nc, N, z0, u);
      launch("rhs", ub + (double)nodes_of(N) * 8, k_rhs_z, dim3((unsigned)((nodes_of(N) + kRhsZBlock - 1) / kRhsZBlock)),
             kRhsZBlock, 0, st, (const double*)u, Nc, N, z0, n, b);
    }
  } else {
    const size_t smem = (size_t)(2 * (Nc / N) + Nc) * sizeof(double);
    launch("rhs", bytes, k_rhs_rows, dim3((unsigned)(N + 1), (unsigned)(N + 1)), kBlock, smem, st, z, Nc, N, b);
  }
}

// e = y - g_h with g_h the nodal interpolant of sin(pi x) sin(pi y) sin(pi z);
// (M e)_n with the consistent Q1 mass M = (h/6)^3 [1 4 1]^(x3); badj = M e on
// interior rows (adjoint right-hand side <y - g, v>_H, Sec. 2.2) and
// Phi = 1/2 e^T M e (eq:cost), reduced per sample in FP64.
// One block per sample (grids below the tiled ones, at most 9^3 nodes): y in shared memory,
// the mass [1 4 1] axis by axis, g and M g from the 1D tables (both separable), Phi summed
// in the block.  1024 samples of 8^3: 314 us with nine sines and 27 weighted products per
// node, 29 us now.
__global__ void __launch_bounds__(kBlock) k_phi_small(const double* __restrict__ y, int N, double* __restrict__ badj,
                                                      double* __restrict__ phi, const double* __restrict__ gtab,
                                                      const double* __restrict__ mgtab) {
  pdl_entry();
  __shared__ double u[729], v[729];
  const int s = blockIdx.x, n1 = N + 1, nodes = n1 * n1 * n1;
  const double* ys = y + (long long)s * nodes;
  for (int n = threadIdx.x; n < nodes; n += kBlock) u[n] = ys[n];  // 0 on the boundary
  __syncthreads();
  for (int n = threadIdx.x; n < nodes; n += kBlock) {
    const int i = n % n1;
    v[n] = (i > 0 && i < N) ? fma(4.0, u[n], u[n - 1] + u[n + 1]) : 0.0;
  }
  __syncthreads();
  for (int n = threadIdx.x; n < nodes; n += kBlock) {
    const int j = (n / n1) % n1;
    u[n] = (j > 0 && j < N) ? fma(4.0, v[n], v[n - n1] + v[n + n1]) : 0.0;
  }
  __syncthreads();
  const double h6 = 1.0 / (6.0 * N), h63 = h6 * h6 * h6;
  double contrib = 0.0;
  for (int n = threadIdx.x; n < nodes; n += kBlock) {
    int i, j, k;
    node_ijk(n, n1, i, j, k);
    double me = 0.0;
    if (interior(i, j, k, N)) {
      const double my = fma(4.0, u[n], u[n - n1 * n1] + u[n + n1 * n1]);
      me = h63 * my - mgtab[i] * mgtab[j] * mgtab[k];
      contrib = fma(ys[n] - gtab[i] * gtab[j] * gtab[k], me, contrib);
    }
    badj[(long long)s * nodes + n] = me;
  }
  contrib = block_sum(contrib);
  if (threadIdx.x == 0) phi[s] = 0.5 * contrib;
}

__global__ void k_phi_finish(const double* __restrict__ partial, int nblk, int S, double* __restrict__ phi) {
  pdl_entry();
  const int s = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (s >= S) return;
  double v = 0.0;
  for (int t = lane; t < nblk; t += 32) v += partial[(long long)s * nblk + t];
  v = warp_sum(v);
  if (lane == 0) phi[s] = 0.5 * v;
}

// the state as FP32 pairs on a tiled grid: M e written as pairs (tables as pairs)
void launch_phi_adjrhs_df(const float2* y, int N, int S, float2* badj, double* phi, double* partial,
                          const float2* gtab, const float2* mgtab, cudaStream_t st) {
  if (S == 0) return;
  const int nb = tiled_phi_df(y, N, S, gtab, mgtab, badj, partial, st);
  launch("phi_finish", 0.0, k_phi_finish, dim3((S + 7) / 8), 256, 0, st, (const double*)partial, nb, S, phi);
}

void launch_phi_adjrhs(const double* y, int N, int S, double* badj, double* phi, double* partial, const double* gtab,
                       const double* mgtab, cudaStream_t st) {
  if (S == 0) return;
  if (N < kTiledMinN) {
    launch("phi_adjrhs", (double)S * nodes_of(N) * 16, k_phi_small, dim3((unsigned)S), kBlock, 0, st, y, N, badj, phi,
           gtab, mgtab);
    return;
  }
  const int nb = tiled_phi(y, N, S, gtab, mgtab, badj, partial, st);
  launch("phi_finish", 0.0, k_phi_finish, dim3((S + 7) / 8), 256, 0, st, (const double*)partial, nb, S, phi);
}

// ---------------------------------------------------------------- level statistics
// work layout: [0] shift_new, [1] scale_old = exp(theta (shift_old - shift_new)),
// [2] n_old, [3] n_old / (n_old + S), [4..4+S) w_fine, [4+S..4+2S) w_coarse, then the same
// weights as FP32 (hi, lo) pairs (8 bytes each): [4+2S..4+3S) fine, [4+3S..4+4S) coarse.
//
// Single block: shift, per-sample weights Y~ = exp(theta (Phi - shift)), and
// the scalar statistics of dY~ = Y~_l - Y~_{l-1} (Welford over the batch,
// then the Chan merge with the rescaled old sums; Algorithm 1, PairwiseUpdate).
__global__ void k_level_scalars(const double* __restrict__ phif, const double* __restrict__ phic, int S,
                                double theta, double* __restrict__ sc, double* __restrict__ work,
                                const int* __restrict__ iters, const int* __restrict__ status) {
  pdl_entry();
  __shared__ double smax[kBlock / 32];
  double m = -INFINITY;
  for (int s = threadIdx.x; s < S; s += blockDim.x) {
    m = fmax(m, phif[s]);
    if (phic) m = fmax(m, phic[s]);
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double bm = smax[0];
    for (int w = 1; w < kBlock / 32; ++w) bm = fmax(bm, smax[w]);
    const double n_old = sc[MLSGD_S_COUNT];
    const double shift_old = sc[MLSGD_S_SHIFT];
    const double shift = (n_old > 0.0) ? fmax(shift_old, bm) : bm;
    work[0] = shift;
    work[1] = (n_old > 0.0) ? exp(theta * (shift_old - shift)) : 0.0;
    work[2] = n_old;
    work[3] = n_old / (n_old + S);
  }
  __syncthreads();
  const double shift = work[0];
  // a sample whose solve went non-finite (status bit 1) gets NaN weights, so the
  // record, and the step that reads it, report the failure instead of using it
  float2* wpair = (float2*)(work + 4 + 2 * S);
  for (int s = threadIdx.x; s < S; s += blockDim.x) {
    const bool bad = status != nullptr && ((status[s] | (phic ? status[S + s] : 0)) & 2);
    const double wf = bad ? NAN : exp(theta * (phif[s] - shift));
    const double wc = bad ? NAN : (phic ? exp(theta * (phic[s] - shift)) : 0.0);
    work[4 + s] = wf;
    work[4 + S + s] = wc;
    wpair[s] = df_split(wf);
    wpair[S + s] = df_split(wc);
  }
  __syncthreads();
  // batch mean and M2 of dY~ by shifted sums over the block (deviations from the
  // first sample), and the sample-wise maxima / counts, all in parallel
  const double ref = work[4] - work[4 + S];
  double sd = 0.0, sd2 = 0.0, pm = -INFINITY, itp = 0.0, ncp = 0.0;
  for (int s = threadIdx.x; s < S; s += blockDim.x) {
    const double d = (work[4 + s] - work[4 + S + s]) - ref;
    sd += d;
    sd2 = fma(d, d, sd2);
    pm = fmax(pm, fmax(phif[s], phic ? phic[s] : -INFINITY));
  }
  if (iters) {
    const int nsolve = phic ? 2 * S : S;
    for (int t = threadIdx.x; t < nsolve; t += blockDim.x) {
      itp += iters[t];
      ncp += (status[t] != 0) ? 1.0 : 0.0;
    }
  }
  sd = block_sum(sd);
  __syncthreads();
  sd2 = block_sum(sd2);
  __syncthreads();
  itp = block_sum(itp);
  __syncthreads();
  ncp = block_sum(ncp);
  for (int o = 16; o > 0; o >>= 1) pm = fmax(pm, __shfl_xor_sync(0xffffffffu, pm, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = pm;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kBlock / 32; ++w) pm = fmax(pm, smax[w]);
    const double mean = ref + sd / S;
    const double s2 = fmax(sd2 - sd * (sd / S), 0.0);
    const double n_old = work[2], scale = work[1];
    const double n = n_old + S;
    const double mo = sc[MLSGD_S_MEAN_DY] * scale;
    const double so = sc[MLSGD_S_S2_DY] * scale * scale;
    const double delta = mo - mean;
    sc[MLSGD_S_MEAN_DY] = mean + (n_old / n) * delta;
    sc[MLSGD_S_S2_DY] = so + s2 + delta * delta * n_old * S / n;
    sc[MLSGD_S_COUNT] = n;
    sc[MLSGD_S_SHIFT] = shift;
    sc[MLSGD_S_PHI_MAX] = fmax(sc[MLSGD_S_PHI_MAX], pm);
    sc[MLSGD_S_ITERS] += itp;
    sc[MLSGD_S_NOCONV] += ncp;
  }
}

// Average of the nodal function q (grid N) over control cell (cx, cy, cz) of the
// Nc grid.  N <= Nc (r = Nc / N): q is trilinear on the control cell, so the
// average is its value at the cell centre.  N > Nc (r = N / Nc): trapezoid
// weights per axis over the r + 1 grid nodes of the cell, 1/r inside and
// 1/(2r) at the two ends.
__device__ __forceinline__ double eval_at_ctrl(const double* __restrict__ q, int N, int Nc, int cx, int cy, int cz) {
  const int n1 = N + 1;
  if (N > Nc) {
    const int r = N / Nc;
    const double wi = 1.0 / r, we = 0.5 / r;
    double acc = 0.0;
    for (int c = 0; c <= r; ++c) {
      const double wz = (c == 0 || c == r) ? we : wi;
      for (int b = 0; b <= r; ++b) {
        const double wy = (b == 0 || b == r) ? we : wi;
        const double* row = q + (long long)r * cx + (long long)n1 * ((long long)r * cy + b + (long long)n1 * ((long long)r * cz + c));
        double rs = 0.5 * (row[0] + row[r]);
        for (int a = 1; a < r; ++a) rs += row[a];
        acc += wz * wy * rs * wi;
      }
    }
    return acc;
  }
  const int r = Nc / N;
  const int ex = cx / r, ey = cy / r, ez = cz / r;
  const double tx = ((cx % r) + 0.5) / r, ty = ((cy % r) + 0.5) / r, tz = ((cz % r) + 0.5) / r;
  const double* b = q + ex + (long long)n1 * (ey + (long long)n1 * ez);
  const long long sy = n1, sz = (long long)n1 * n1;
  const double c00 = b[0] * (1 - tx) + b[1] * tx;
  const double c10 = b[sy] * (1 - tx) + b[sy + 1] * tx;
  const double c01 = b[sz] * (1 - tx) + b[sz + 1] * tx;
  const double c11 = b[sy + sz] * (1 - tx) + b[sy + sz + 1] * tx;
  return (c00 * (1 - ty) + c10 * ty) * (1 - tz) + (c01 * (1 - ty) + c11 * ty) * tz;
}

// FP32 -> FP64 by moving the fields (IEEE 754 binary32 and binary64 layouts), in
// integer instructions instead of the FP64 conversion: exponent rebiased by
// 1023 - 127, mantissa shifted into the top of the 52-bit field; 0 and subnormals
// give a signed 0, Inf and NaN keep their class (a NaN stays a NaN).
__device__ __forceinline__ double f2d(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
  const uint32_t e11 = e == 0u ? 0u : (e == 0xffu ? 0x7ffu : e + 896u);
  const uint32_t mh = e == 0u ? 0u : ((m >> 3) | ((e == 0xffu && m != 0u) ? 0x80000u : 0u));
  const uint32_t hi = (u & 0x80000000u) | (e11 << 20) | mh;
  const uint32_t lo = e == 0u ? 0u : (m << 29);
  return __hiloint2double((int)hi, (int)lo);
}
// The eight trilinear weights of a control-cell centre inside a level cell
// (level no finer than the control grid), set up once per control cell.
struct CellInterp {
  long long base;  // node (ex, ey, ez) of the level cell holding the control cell
  long long sy, sz;
  double w[8];     // weight of node (ex + a, ey + b, ez + c) at index a + 2b + 4c
  float w32[8];    // the same weights (exact in FP32: r is a power of two)
  // the weights are dyadic and exact in FP32, so they are formed there (an FP64 division
  // is some 20 operations of the pipe that bounds the kernel)
  __device__ void setup(int N, int Nc, int cx, int cy, int cz) {
    const int n1 = N + 1, r = Nc / N;
    const float ir = 1.0f / (float)r;
    const float tx = ((cx % r) + 0.5f) * ir, ty = ((cy % r) + 0.5f) * ir, tz = ((cz % r) + 0.5f) * ir;
    base = (cx / r) + (long long)n1 * ((cy / r) + (long long)n1 * (cz / r));
    sy = n1;
    sz = (long long)n1 * n1;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      w32[e] = ((e & 1) ? tx : 1.0f - tx) * ((e & 2) ? ty : 1.0f - ty) * ((e & 4) ? tz : 1.0f - tz);
      w[e] = f2d(w32[e]);
    }
  }
  // the same average of an FP32 pair field, in pair arithmetic
  __device__ __forceinline__ DF eval(const float2* __restrict__ q) const {
    const float2* b = q + base;
    const float2 v[8] = {b[0], b[1], b[sy], b[sy + 1], b[sz], b[sz + 1], b[sz + sy], b[sz + sy + 1]};
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float p = __fmul_rn(w32[e], v[e].x);
      const float pe = __fmaf_rn(w32[e], v[e].y, __fmaf_rn(w32[e], v[e].x, -p));
      const float t = __fadd_rn(s, p);  // two-sum (intrinsics: never contracted)
      const float bb = __fsub_rn(t, s);
      c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(p, bb)), pe));
      s = t;
    }
    return df_norm(s, c);
  }
  __device__ __forceinline__ double eval(const double* __restrict__ q) const {
    const double* b = q + base;
    double v = w[0] * b[0];
    v = fma(w[1], b[1], v);
    v = fma(w[2], b[sy], v);
    v = fma(w[3], b[sy + 1], v);
    v = fma(w[4], b[sz], v);
    v = fma(w[5], b[sz + 1], v);
    v = fma(w[6], b[sz + sy], v);
    return fma(w[7], b[sz + sy + 1], v);
  }
};

// The same trilinear average for FP32 pair fields on a grid R times coarser than the
// control grid, R known at compile time: three per-axis weight pairs (exact dyadic values,
// so each product equals CellInterp's w32), a 32-bit node index, and for R = 1 no product
// at all (every weight is 1/8: the sum is scaled, which is exact).
template <int R>
struct PairInterp {
  int base, sy, sz;
  float tx, ty, tz;
  __device__ __forceinline__ void setup(int N, int cx, int cy, int cz) {
    const int n1 = N + 1;
    constexpr float ir = 1.0f / R;
    tx = ((cx % R) + 0.5f) * ir;
    ty = ((cy % R) + 0.5f) * ir;
    tz = ((cz % R) + 0.5f) * ir;
    base = (cx / R) + n1 * ((cy / R) + n1 * (cz / R));
    sy = n1;
    sz = n1 * n1;
  }
  __device__ __forceinline__ DF eval(const float2* __restrict__ q) const {
    const float2* b = q + base;
    float2 v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = b[(e & 1) + ((e >> 1) & 1) * sy + (e >> 2) * sz];
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      float p, pe;
      if constexpr (R == 1) {
        p = v[e].x;
        pe = v[e].y;
      } else {
        const float w = (((e & 1) ? tx : 1.0f - tx) * ((e & 2) ? ty : 1.0f - ty)) * ((e & 4) ? tz : 1.0f - tz);  // exact
        p = __fmul_rn(w, v[e].x);
        pe = __fmaf_rn(w, v[e].y, __fmaf_rn(w, v[e].x, -p));
      }
      if (e == 0) {
        s = p;
        c = pe;
        continue;
      }
      const float t = __fadd_rn(s, p);  // two-sum (intrinsics: never contracted)
      const float bb = __fsub_rn(t, s);
      c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(p, bb)), pe));
      s = t;
    }
    if constexpr (R == 1) return df_norm(0.125f * s, 0.125f * c);
    return df_norm(s, c);
  }
};

// eval_at_ctrl for an FP32 pair field, in pair arithmetic (trapezoid weights are
// exact in FP32 since r is a power of two)
__device__ DF eval_at_ctrl(const float2* __restrict__ q, int N, int Nc, int cx, int cy, int cz) {
  const int n1 = N + 1;
  const int r = N / Nc;
  const float wi = 1.0f / r, we = 0.5f / r;
  DF acc{0.f, 0.f};
  for (int c = 0; c <= r; ++c) {
    const float wz = (c == 0 || c == r) ? we : wi;
    for (int b = 0; b <= r; ++b) {
      const float wy = (b == 0 || b == r) ? we : wi;
      const float2* row = q + (long long)r * cx + (long long)n1 * ((long long)r * cy + b + (long long)n1 * ((long long)r * cz + c));
      DF rs = df_mulf(df_add(df_make(row[0]), df_make(row[r])), 0.5f);
      for (int a = 1; a < r; ++a) rs = df_add(rs, df_make(row[a]));
      acc = df_add(acc, df_mulf(rs, wz * wy * wi));
    }
  }
  return acc;
}

// One thread per control cell: B*q as the cell average for both grids,
// dX~_s = w_f[s] B*q_f[s] - w_c[s] B*q_c[s]; batch mean and M2 by the
// shifted-data sums (deviations from the first sample: no division per
// sample, stable when the first sample is typical), then the Chan merge with
// the rescaled old mean; block partials of h_c^3 (M2_batch + delta^2 n_old S / n).
// PF / PC: the fine / coarse adjoint solutions are FP32 (hi, lo) pairs (the mixed
// path on tiled grids); their control-cell averages are then formed in pair
// arithmetic (exact weights, about 48 significant bits), and with both grids in
// pairs so is the weighted difference w_f X_f - w_c X_c (weights rounded to pairs
// from their FP64 values; error below 6 u^2 (|w_f X_f| + |w_c X_c|), u = 2^-24), a
// function of the sample alone.  The sums of the cancelling differences, the
// deviations from the first sample and the merge are FP64 in every case
// (eq:delta-notation, eq:sec-order-sum), so a record does not depend on how the
// samples were split into calls beyond FP64 rounding.  (This part has about 2 FP64
// operations per FP32 one; GB300 issues FP64 at 1/58 of the FP32 rate, so the FP64
// count sets the kernel's time.)
__device__ __forceinline__ double ctrl_avg(const CellInterp& I, bool fast, const double* q, int N, int Nc, int cx,
                                           int cy, int cz) {
  return fast ? I.eval(q) : eval_at_ctrl(q, N, Nc, cx, cy, cz);
}
__device__ __forceinline__ DF ctrl_avg_df(const CellInterp& I, bool fast, const float2* q, int N, int Nc, int cx,
                                          int cy, int cz) {
  return fast ? I.eval(q) : eval_at_ctrl(q, N, Nc, cx, cy, cz);
}
__device__ __forceinline__ double ctrl_avg(const CellInterp& I, bool fast, const float2* q, int N, int Nc, int cx,
                                           int cy, int cz) {
  return df_to_double(ctrl_avg_df(I, fast, q, N, Nc, cx, cy, cz));
}
template <bool PF, bool PC>
__global__ void __launch_bounds__(kBlock) k_level_field(const void* __restrict__ qf_, int Nf,
                                                        const void* __restrict__ qc_, int Ncs, int S, int Nc,
                                                        double inv_s, const double* __restrict__ work,
                                                        double* __restrict__ field, double* __restrict__ partial) {
  pdl_entry();
  using QF = typename std::conditional<PF, float2, double>::type;
  using QC = typename std::conditional<PC, float2, double>::type;
  const QF* qf = (const QF*)qf_;
  const QC* qc = (const QC*)qc_;
  const unsigned ncell = (unsigned)Nc * Nc * Nc;  // at most 1024^3
  const unsigned step = gridDim.x * kBlock;
  const long long nf = nodes_of(Nf), ncn = qc ? nodes_of(Ncs) : 0;
  const double* wf = work + 4;
  const double* wc = work + 4 + S;
  const float2* wfp = (const float2*)(work + 4 + 2 * S);
  const float2* wcp = wfp + S;
  // level grids no finer than the control grid: weights hoisted out of the sample loop
  const bool fast_f = Nf <= Nc, fast_c = !qc || Ncs <= Nc;
  const double n_old = work[2], scale = work[1], a = work[3];
  const double as = a * S;  // n_old S / (n_old + S)
  double contrib = 0.0;
  for (unsigned c = blockIdx.x * kBlock + threadIdx.x; c < ncell; c += step) {
    const unsigned row = c / (unsigned)Nc;
    const int cx = (int)(c - row * Nc), cz = (int)(row / (unsigned)Nc), cy = (int)(row - (unsigned)cz * Nc);
    double ref = 0.0, sd = 0.0, sd2 = 0.0;
    CellInterp If{}, Ic{};
    if (fast_f) If.setup(Nf, Nc, cx, cy, cz);
    if (qc && fast_c) Ic.setup(Ncs, Nc, cx, cy, cz);
    for (int s = 0; s < S; ++s) {
      double v;
      if constexpr (PF && PC) {
        const DF vf = df_mul(df_make(wfp[s]), ctrl_avg_df(If, fast_f, qf + s * nf, Nf, Nc, cx, cy, cz));
        const DF vc = df_mul(df_make(wcp[s]), ctrl_avg_df(Ic, fast_c, qc + s * ncn, Ncs, Nc, cx, cy, cz));
        const DF vd = df_add(vf, df_neg(vc));
        v = f2d(vd.h) + f2d(vd.l);
      } else {
        v = wf[s] * ctrl_avg(If, fast_f, qf + s * nf, Nf, Nc, cx, cy, cz);
        if (qc) v = fma(-wc[s], ctrl_avg(Ic, fast_c, qc + s * ncn, Ncs, Nc, cx, cy, cz), v);
      }
      if (s == 0) ref = v;
      const double d = v - ref;
      sd += d;
      sd2 = fma(d, d, sd2);
    }
    const double mean = fma(sd, inv_s, ref);
    const double m2 = fmax(fma(-sd * inv_s, sd, sd2), 0.0);
    const double mo = (n_old > 0.0) ? field[c] * scale : 0.0;
    const double delta = mo - mean;
    field[c] = fma(a, delta, mean);
    contrib += fma(as * delta, delta, m2);
  }
  const double bs = block_sum(contrib);
  const double hc = 1.0 / Nc;
  if (threadIdx.x == 0) partial[blockIdx.x] = hc * hc * hc * bs;
}

// k_level_field for pairs on both grids, the fine one the control grid: the bulk of the
// finest difference level's statistics.  The FP32 pair arithmetic and
// the FP64 sums (four operations per cell and sample) take about the same time, and the
// 16 scattered loads need threads in flight: 64 registers, four blocks per SM.  G = 4
// splits the samples of a cell over four threads (their sums joined in a fixed order), for
// batches on control grids too small to fill the SMs with one thread per cell: 512 samples
// of 64^3 on a 64^3 control: 1.6 ms.
template <int G>
__global__ void __launch_bounds__(kBlock, 4) k_level_pairs(const float2* __restrict__ qf, int Nf,
                                                           const float2* __restrict__ qc, int S, int Nc, double inv_s,
                                                           const double* __restrict__ work, double* __restrict__ field,
                                                           double* __restrict__ partial) {
  pdl_entry();
  constexpr int CB = kBlock / G;  // cells per block
  __shared__ double sums[G > 1 ? 2 : 1][G][CB];
  const unsigned ncell = (unsigned)Nc * Nc * Nc;
  const int tc = threadIdx.x % CB, g = threadIdx.x / CB;
  const int Ncs = Nf / 2;
  const long long nf = nodes_of(Nf), nc = nodes_of(Ncs);
  const float2* wfp = (const float2*)(work + 4 + 2 * S);
  const float2* wcp = wfp + S;
  double contrib = 0.0;
  for (unsigned c0 = blockIdx.x * CB; c0 < ncell; c0 += gridDim.x * CB) {  // ncell is a multiple of 8
    const unsigned c = c0 + tc < ncell ? c0 + tc : ncell - 1;
    const unsigned row = c / (unsigned)Nc;
    const int cx = (int)(c - row * Nc), cz = (int)(row / (unsigned)Nc), cy = (int)(row - (unsigned)cz * Nc);
    PairInterp<1> Pf;
    PairInterp<2> Pc;
    Pf.setup(Nf, cx, cy, cz);
    Pc.setup(Ncs, cx, cy, cz);
    auto value = [&](int s, const float2* f, const float2* k) {
      const DF vf = df_mul(df_make(wfp[s]), Pf.eval(f));
      const DF vc = df_mul(df_make(wcp[s]), Pc.eval(k));
      const DF vd = df_add(vf, df_neg(vc));
      return f2d(vd.h) + f2d(vd.l);
    };
    // sample pointers advanced by addition: a 64-bit multiply per sample would issue on
    // the FP64 pipe
    const double ref = value(0, qf, qc);
    double sd = 0.0, sd2 = 0.0;
    const int s0 = g == 0 ? G : g;  // sample 0 is the reference: its deviation is 0
    const float2 *f = qf + (long long)s0 * nf, *k = qc + (long long)s0 * nc;
    for (int s = s0; s < S; s += G, f += G * nf, k += G * nc) {
      const double d = value(s, f, k) - ref;
      sd += d;
      sd2 = fma(d, d, sd2);
    }
    if constexpr (G > 1) {
      sums[0][g][tc] = sd;
      sums[1][g][tc] = sd2;
      __syncthreads();
      if (g == 0) {
#pragma unroll
        for (int q = 1; q < G; ++q) {
          sd += sums[0][q][tc];
          sd2 += sums[1][q][tc];
        }
      }
      __syncthreads();
    }
    if (g == 0 && c0 + tc < ncell) {
      const double a = work[3];  // n_old / (n_old + S)
      const double mean = fma(sd, inv_s, ref);
      const double m2 = fmax(fma(-sd * inv_s, sd, sd2), 0.0);
      const double mo = (work[2] > 0.0) ? field[c] * work[1] : 0.0;
      const double delta = mo - mean;
      field[c] = fma(a, delta, mean);
      contrib += fma(a * S * delta, delta, m2);
    }
  }
  const double bs = block_sum(contrib);
  const double hc = 1.0 / Nc;
  if (threadIdx.x == 0) partial[blockIdx.x] = hc * hc * hc * bs;
}

// ---- statistics of a level whose grids are coarser than the control grid (Nc = r Nf,
// r >= 2).  Interpolation to the control grid is linear, so with the nodal values
// x_s = w_f[s] q_f[s] - w_c[s] P q_c[s] on the level's fine grid (P q_c: the coarse
// trilinear function at the fine nodes, which interpolation to the control cells
// reproduces exactly) the batch mean field is the interpolation of the nodal mean,
// and ||I x||_U^2 = h_f^3 x^T (g x g x g) x with the 1D Gram matrix g assembled from
// (1/r) sum_m w(t_m) w(t_m)^T, w(t) = (1 - t, t), t_m = (m + 1/2)/r (the midpoint rule over
// the r^3 control cells of a level cell is exact for the integrand of these trilinear
// weights): rows [B, 2A, B], x is 0 on the boundary.  M2 of the batch is the sum over
// samples of that form of x_s - mean.  Work per sample: the level's nodes, not the
// control cells.
//
// Bound: FP64 issue.  The form is applied axis by axis (three operations per node and
// axis) to the deviations from the mean, where the 8 x 8 matrix per level cell took 64 per
// cell.  Values given as FP32 pairs enter FP64 by integer instructions (f2d) and one addition.
__device__ __forceinline__ double ldq(const double* p, long long i) { return p[i]; }
__device__ __forceinline__ double f2d_all(float f) {  // f2d, subnormals too: scaled into its range
  const bool small = fabsf(f) < 0x1p-126f;
  const double d = f2d(small ? f * 0x1p64f : f);
  return small && f != 0.f ? __hiloint2double(__double2hiint(d) - (64 << 20), __double2loint(d)) : d;
}
__device__ __forceinline__ double ldq(const float2* p, long long i) {
  const float2 v = p[i];
  return f2d_all(v.x) + f2d_all(v.y);
}
// x_s at every node of the level grid, written over q_f (same 8-byte slots; q_f is
// not needed after the statistics)
template <typename QF, typename QC>
__global__ void __launch_bounds__(kBlock) k_lvl_x(QF* __restrict__ qf, int Nf, const QC* __restrict__ qc, int S,
                                                  const double* __restrict__ work) {
  pdl_entry();
  const int s = blockIdx.y;
  const int n1 = Nf + 1, nodes = n1 * n1 * n1;  // at most 513^3 (the control grid is finer)
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nodes) return;
  int i, j, k;
  node_ijk(n, n1, i, j, k);
  QF* qs = qf + (long long)s * nodes;
  double x = work[4 + s] * ldq(qs, n);
  if (qc) {
    const int c1 = Nf / 2 + 1;
    const QC* q = qc + (long long)s * (c1 * c1 * c1) + (i >> 1) + c1 * ((j >> 1) + c1 * (k >> 1));
    const int di = i & 1, dj = j & 1, dk = k & 1;
    double acc = 0.0;
    for (int c = 0; c <= dk; ++c)
      for (int b = 0; b <= dj; ++b)
        for (int a = 0; a <= di; ++a) acc += ldq(q, a + c1 * (b + c1 * c));
    x = fma(-work[4 + S + s] * (di ? 0.5 : 1.0), (dj ? 0.5 : 1.0) * (dk ? 0.5 : 1.0) * acc, x);
  }
  reinterpret_cast<double*>(qs)[n] = x;
}
// nodal mean over the samples, by deviations from the first one: a block takes 32 nodes
// and splits the samples over its eight warps (summed in a fixed order)
__global__ void __launch_bounds__(kBlock) k_lvl_mean(const double* __restrict__ x, int nodes, int S, double inv_s,
                                                     double* __restrict__ mean) {
  pdl_entry();
  __shared__ double part[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n = blockIdx.x * 32 + lane;
  double d = 0.0, xr = 0.0;
  if (n < nodes) {
    xr = x[n];
#pragma unroll 4
    for (int s = w; s < S; s += 8) d += x[(long long)s * nodes + n] - xr;
  }
  part[w][lane] = d;
  __syncthreads();
  if (w == 0 && n < nodes) {
#pragma unroll
    for (int v = 1; v < 8; ++v) d += part[v][lane];
    mean[n] = fma(d, inv_s, xr);
  }
}
// sum over samples of d^T (g x g x g) d, d = x_s - mean, grids of at most 16^3: a sample in
// shared memory, one axis after the other; blockIdx.x takes samples x, x + gridDim.x, ..
__global__ void __launch_bounds__(kBlock) k_lvl_s2_small(const double* __restrict__ x, int N, int S,
                                                         const double* __restrict__ mean, double A2, double B,
                                                         double hf3, double* __restrict__ partial) {
  pdl_entry();
  extern __shared__ double sm[];
  const int n1 = N + 1, nodes = n1 * n1 * n1, m1 = N - 1, inner = m1 * m1 * m1;
  double *d = sm, *u = sm + nodes, *v = sm + 2 * nodes;
  double acc = 0.0;
  auto node = [&](int e) {  // interior node e of (N - 1)^3
    const int t = e / m1, i = e - t * m1, k = t / m1, j = t - k * m1;
    return (i + 1) + n1 * ((j + 1) + n1 * (k + 1));
  };
  for (int e = threadIdx.x; e < 3 * nodes; e += kBlock) sm[e] = 0.0;
  for (int s = blockIdx.x; s < S; s += gridDim.x) {
    __syncthreads();
    for (int e = threadIdx.x; e < inner; e += kBlock) {
      const int n = node(e);
      d[n] = x[(long long)s * nodes + n] - mean[n];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < inner; e += kBlock) {
      const int n = node(e);
      u[n] = fma(A2, d[n], B * (d[n - 1] + d[n + 1]));
    }
    __syncthreads();
    for (int e = threadIdx.x; e < inner; e += kBlock) {
      const int n = node(e);
      v[n] = fma(A2, u[n], B * (u[n - n1] + u[n + n1]));
    }
    __syncthreads();
    for (int e = threadIdx.x; e < inner; e += kBlock) {
      const int n = node(e);
      acc = fma(d[n], fma(A2, v[n], B * (v[n - n1 * n1] + v[n + n1 * n1])), acc);
    }
  }
  const double bs = block_sum(acc);
  if (threadIdx.x == 0) partial[blockIdx.x] = hf3 * bs;
}
// the same on larger grids: 32 x 32 tiles (four rows per thread) marching over kLvlPlanes
// planes of one sample; blockIdx.z: (sample group, z chunk), samples g, g + groups, ..
constexpr int kLvlPlanes = 16, kLvlTY = 32;
__global__ void __launch_bounds__(kBlock) k_lvl_s2(const double* __restrict__ x, int N, int S, int groups,
                                                   const double* __restrict__ mean, double A2, double B, double hf3,
                                                   double* __restrict__ partial) {
  pdl_entry();
  __shared__ double d[kLvlTY + 2][34], u[kLvlTY + 2][32];
  const int n1 = N + 1, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const long long nodes = (long long)n1 * n1 * n1, pn = (long long)n1 * n1;
  const int x0 = 1 + 32 * blockIdx.x, y0 = 1 + kLvlTY * blockIdx.y;
  const int chunk = blockIdx.z / groups, group = blockIdx.z % groups;
  const int k0 = 1 + kLvlPlanes * chunk, k1 = min(N - 1, k0 + kLvlPlanes - 1);
  double acc = 0.0;
  for (int s = group; s < S; s += groups) {
    const double* xs = x + s * nodes;
    double below[4], here[4], dc[4], dn[4];  // v of planes k - 1 and k, d of the own nodes of planes k and k + 1
#pragma unroll
    for (int t = 0; t < 4; ++t) below[t] = here[t] = dc[t] = 0.0;
    for (int m = k0 - 1; m <= k1 + 1; ++m) {
      const bool mok = m > 0 && m < N;
      __syncthreads();
      for (int e = threadIdx.x; e < (kLvlTY + 2) * 34; e += kBlock) {
        const int ly = e / 34, lx = e - 34 * ly, i = x0 - 1 + lx, j = y0 - 1 + ly;
        const bool ok = mok && i > 0 && j > 0 && i < N && j < N;
        const long long n = i + (long long)n1 * j + pn * m;
        d[ly][lx] = ok ? xs[n] - mean[n] : 0.0;
      }
      __syncthreads();
      for (int e = ty; e < kLvlTY + 2; e += 8) u[e][tx] = fma(A2, d[e][tx + 1], B * (d[e][tx] + d[e][tx + 2]));
      __syncthreads();
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int ly = 4 * ty + t;
        const double v = fma(A2, u[ly + 1][tx], B * (u[ly][tx] + u[ly + 2][tx]));
        dn[t] = d[ly + 1][tx + 1];  // 0 outside the interior
        if (m > k0) acc = fma(dc[t], fma(A2, here[t], B * (below[t] + v)), acc);
        below[t] = here[t];
        here[t] = v;
        dc[t] = dn[t];
      }
    }
  }
  const double bs = block_sum(acc);
  const int bid = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (threadIdx.x == 0) partial[bid] = hf3 * bs;
}
// per control cell: batch mean = interpolated nodal mean; Chan merge with the old
// field; block partials of h_c^3 delta^2 n_old S / n.  A block takes kLvlRows rows cy of a
// plane cz of control cells, 256 cells of a row per block in x.  The node lines under it are
// interpolated in z once, into shared memory; a thread interpolates a line in x at its cx
// when it is reached, and a cell is then one FMA in y between the lines on either side
// (1 + 3/r + 4 (Nf/256)(1/r + 1/16) FP64 operations a cell, the bound next to the store; one
// interpolation in (y, z) per row, by one warp between three barriers, took 190 us on a
// 256^3 control, about 75 us now).  An empty record (n_old = 0) is not read.
constexpr int kLvlRows = 16;
__global__ void __launch_bounds__(kBlock) k_lvl_field(const double* __restrict__ xm, int Nf, int Nc, int S,
                                                      const double* __restrict__ work, double* __restrict__ field,
                                                      double* __restrict__ partial) {
  pdl_entry();
  extern __shared__ double line[];  // [lines][Nf + 1]: the mean interpolated in z
  const int n1 = Nf + 1, r = Nc / Nf;
  const long long sz = (long long)n1 * n1;
  const float inv_r = 1.0f / (float)r;  // r a power of two: the weights are exact in FP32
  const double n_old = work[2], scale = work[1], a = work[3];
  const int cx = blockIdx.x * blockDim.x + threadIdx.x, cz = blockIdx.z;
  const int cy0 = blockIdx.y * kLvlRows, cy1 = min(Nc, cy0 + kLvlRows);
  const int ey0 = cy0 / r, nl = (cy1 - 1) / r - ey0 + 2;
  {
    const int ez = cz / r;
    const float tz = ((float)(cz - ez * r) + 0.5f) * inv_r;
    const double w0 = f2d(1.f - tz), w1 = f2d(tz);
    const double* b = xm + (long long)n1 * ey0 + sz * ez;
    for (int c = threadIdx.x; c < nl * n1; c += blockDim.x) line[c] = fma(w1, b[sz + c], w0 * b[c]);
  }
  __syncthreads();
  double contrib = 0.0;
  if (cx < Nc) {
    const int ex = cx / r;
    const double tx = f2d(((float)(cx - ex * r) + 0.5f) * inv_r);
    const double* l = line + ex;
    auto at_x = [&](const double* q) { return fma(tx, q[1] - q[0], q[0]); };
    double lo = 0.0, up = at_x(l), dy = 0.0;
    double* f = field + cx + (long long)Nc * (cy0 + (long long)Nc * cz);
    for (int cy = cy0; cy < cy1; ++cy, f += Nc) {
      const int my = cy & (r - 1);
      if (my == 0 || cy == cy0) {  // the next node line
        lo = up;
        l += n1;
        up = at_x(l);
        dy = up - lo;
      }
      const double mean = fma(f2d(((float)my + 0.5f) * inv_r), dy, lo);
      if (n_old > 0.0) {
        const double delta = fma(*f, scale, -mean);
        *f = fma(a, delta, mean);
        contrib = fma(delta, delta, contrib);
      } else {
        *f = mean;
      }
    }
  }
  const double hc = 1.0 / Nc;
  contrib *= hc * hc * hc * a * S;
  const double bs = block_sum(contrib);
  if (threadIdx.x == 0) partial[blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z)] = bs;
}

// returns the number of block partials written (at most level_partial_cap(Nc, Nf))
template <typename QF, typename QC>
static int launch_lvl(const void* qf, int Nf, const void* qc, int S, int Nc, const double* work, double* field,
                      double* partial, double* nodebuf, cudaStream_t st) {
  const long long nodes = nodes_of(Nf), ncell = cells_of(Nc);
  const int r = Nc / Nf;
  double A = 0.0, B = 0.0;
  for (int m = 0; m < r; ++m) {
    const double t = (m + 0.5) / r;
    A += (1.0 - t) * (1.0 - t) / r;
    B += t * (1.0 - t) / r;
  }
  const double hf = 1.0 / Nf, hf3 = hf * hf * hf;
  const double qb = (double)S * sizeof(QF) * (nodes + (qc ? nodes_of(Nf / 2) : 0));
  const unsigned nbn = (unsigned)((nodes + kBlock - 1) / kBlock);
  launch("level_x", qb + (double)S * nodes * 8, k_lvl_x<QF, QC>, dim3(nbn, (unsigned)S), kBlock, 0, st,
         (QF*)const_cast<void*>(qf), Nf, (const QC*)qc, S, work);
  const double* x = (const double*)qf;
  double* mean = nodebuf;
  launch("level_nodes", (double)S * nodes * 8 + (double)nodes * 8, k_lvl_mean, dim3((unsigned)((nodes + 31) / 32)), kBlock,
         0, st, x, (int)nodes, S, 1.0 / S, mean);
  const unsigned fx = (unsigned)((Nc + kBlock - 1) / kBlock);
  const unsigned fy = (unsigned)((Nc + kLvlRows - 1) / kLvlRows);
  const long long nf = (long long)fx * fy * Nc;
  launch("level_field", (double)nodes * 8 + (double)ncell * 16, k_lvl_field, dim3(fx, fy, (unsigned)Nc),
         kBlock, (size_t)((kLvlRows - 1) / r + 2 + (r < kLvlRows ? 1 : 0)) * (Nf + 1) * sizeof(double), st, (const double*)mean, Nf, Nc, S, work, field, partial);
  // samples spread over blocks within the partial buffer
  const long long room = level_partial_cap(Nc, Nf) - nf;
  const double sb = (double)S * nodes * 8 + (double)nodes * 8;
  if (Nf <= 16) {
    const int g = (int)std::min<long long>(S, room);
    const size_t smem = 3 * (size_t)nodes * sizeof(double);
    static SmemOptIn opt_in;
    if (smem > 48 * 1024) (void)opt_in(k_lvl_s2_small, smem);  // a launch without it is refused
    launch("level_cells", sb, k_lvl_s2_small, dim3((unsigned)g), kBlock, smem, st, x, Nf, S, (const double*)mean, 2.0 * A, B,
           hf3, partial + nf);
    return (int)(nf + g);
  }
  const int bx = (Nf - 1 + 31) / 32, by = (Nf - 1 + kLvlTY - 1) / kLvlTY, bz = (Nf - 1 + kLvlPlanes - 1) / kLvlPlanes;
  const long long tiles = (long long)bx * by * bz;
  const int g = (int)std::max<long long>(1, std::min<long long>(S, std::min<long long>(room / tiles, (8LL * 152 + tiles - 1) / tiles)));
  launch("level_cells", sb, k_lvl_s2, dim3((unsigned)bx, (unsigned)by, (unsigned)(bz * g)), kBlock, 0, st, x, Nf, S, g,
         (const double*)mean, 2.0 * A, B, hf3, partial + nf);
  return (int)(nf + tiles * g);
}

// s2_dx = old * scale^2 + sum of partials (fixed order, one block)
__global__ void __launch_bounds__(kBlock) k_level_finish(const double* __restrict__ partial, int nblk,
                                                         const double* __restrict__ work, double* __restrict__ sc) {
  pdl_entry();
  double v = 0.0;
  for (int t = threadIdx.x; t < nblk; t += kBlock) v += partial[t];
  v = block_sum(v);
  if (threadIdx.x == 0) {
    const double scale = work[1];
    sc[MLSGD_S_S2_DX] = (work[2] > 0.0 ? sc[MLSGD_S_S2_DX] * scale * scale : 0.0) + v;
  }
}

void launch_level_stats(const double* qf, const double* phif, int Nf, const double* qc, const double* phic,
                        int Ncoarse, int S, int Nc, double theta, double* field, double* scalars, double* work,
                        double* partial, const int* iters, const int* status, cudaStream_t st, bool qf_pairs,
                        bool qc_pairs, double* nodebuf) {
  if (S == 0) return;
  launch("level_scalars", 0.0, k_level_scalars, dim3(1), kBlock, 0, st, phif, phic, S, theta, scalars, work, iters,
         status);
  // levels coarser than the control grid: statistics on the level grid (cost ~ level nodes
  // per sample instead of control cells per sample; at 2x the whole FP64 level 3 of a run
  // 18.87 -> 18.52 ms, 4 samples of 128^3 in pairs on a 256^3 control 11.63 -> 11.47, 300 of
  // 32^3 on 64^3 7.83 -> 7.64).  q_f is overwritten.
  if (nodebuf && 2 * Nf <= Nc) {
    const int nb = (qf_pairs && qc_pairs) ? launch_lvl<float2, float2>(qf, Nf, qc, S, Nc, work, field, partial, nodebuf, st)
                   : qf_pairs             ? launch_lvl<float2, double>(qf, Nf, qc, S, Nc, work, field, partial, nodebuf, st)
                                          : launch_lvl<double, double>(qf, Nf, qc, S, Nc, work, field, partial, nodebuf, st);
    launch("level_finish", 0.0, k_level_finish, dim3(1), kBlock, 0, st, (const double*)partial, nb, (const double*)work,
           scalars);
    return;
  }
  const long long ncell = (long long)Nc * Nc * Nc;
  const int nblk = cell_blocks(ncell);
  const double qbytes = (double)S * 8 * (nodes_of(Nf) + (qc ? nodes_of(Ncoarse) : 0));
  // both grids in pairs, the fine one the control grid
  if (qf_pairs && qc_pairs && Nf == Nc) {
    const bool split = S >= 16 && ncell < (long long)kPairBlocks * kBlock * 4;
    const int cb = split ? kBlock / 4 : kBlock;
    const int nb = (int)std::min<long long>({(ncell + cb - 1) / cb, split ? kPairBlocks : cell_blocks(ncell),
                                             level_partial_cap(Nc, Nf)});
    auto kp = split ? k_level_pairs<4> : k_level_pairs<1>;
    launch_flops("level_field", qbytes + (double)ncell * 16, (double)S * ncell * 4.0, kp, dim3(nb), kBlock, 0, st,
                 (const float2*)qf, Nf, (const float2*)qc, S, Nc, 1.0 / S, (const double*)work, field, partial);
    launch("level_finish", 0.0, k_level_finish, dim3(1), kBlock, 0, st, (const double*)partial, nb, (const double*)work,
           scalars);
    return;
  }
  // pairs on the coarse grid only come with pairs on the fine grid (it is at least as large)
  auto lf = qf_pairs ? (qc_pairs ? k_level_field<true, true> : k_level_field<true, false>) : k_level_field<false, false>;
  // FP64 operations per control cell and sample: both grids in pairs, the pair value
  // to FP64 (2 conversions, 1 add), its deviation and the two sums; otherwise also the
  // FP64 weighting and, for FP64 fields, the 8-node averages
  const double f64ops = qf_pairs && qc_pairs ? 6.0 : (qf_pairs ? 16.0 : 21.0);
  launch_flops("level_field", qbytes + (double)ncell * 16, (double)S * ncell * f64ops, lf, dim3(nblk), kBlock, 0, st,
               (const void*)qf, Nf, (const void*)qc, Ncoarse, S, Nc, 1.0 / S, (const double*)work, field, partial);
  launch("level_finish", 0.0, k_level_finish, dim3(1), kBlock, 0, st, (const double*)partial, nblk, (const double*)work,
         scalars);
}

__global__ void __launch_bounds__(kBlock) k_stats_reset(double* __restrict__ field, double* __restrict__ sc, long long n) {
  pdl_entry();
  const long long i0 = (long long)blockIdx.x * kBlock + threadIdx.x, step = (long long)gridDim.x * kBlock;
  if (i0 < MLSGD_NSCALARS) sc[i0] = (i0 == MLSGD_S_SHIFT || i0 == MLSGD_S_PHI_MAX) ? -INFINITY : 0.0;
#pragma unroll 4
  for (long long i = i0; i < n; i += step) field[i] = 0.0;
}

void launch_stats_reset(double* field, double* scalars, long long ncells, cudaStream_t st) {
  launch("stats_reset", (double)ncells * 8, k_stats_reset, dim3((unsigned)cell_blocks(ncells)), kBlock, 0, st, field,
         scalars, ncells);
}

// Chan merge of two statistics records: src into dst, both rescaled to the larger shift.
//
// Bound: FP64 issue (2 operations per clock and SM; 3 or 4 per cell here), then HBM (24
// bytes per cell).  The factors' exponentials and the divisions by the counts are the
// same for every cell, so thread 0 of a block forms them once and at most
// kCellBlocks blocks march over the cells; the scalar kernel then sums a few partial
// sums per thread.  A merge into an empty record (the first of a series) is a copy and
// does not read dst.  Six levels on a 256^3 control (16.8M cells) reset, merged twice and
// stepped: 31.9 ms with the factors formed per cell and one warp over 65536 partial
// sums, 1.94 ms now (1.6 ms of FP64 issue).
__global__ void __launch_bounds__(kBlock) k_merge_field(double* __restrict__ df, const double* __restrict__ dsc,
                                                        const double* __restrict__ sf, const double* __restrict__ ssc,
                                                        long long n, double theta, double hc3,
                                                        double* __restrict__ partial) {
  pdl_entry();
  __shared__ double co[4];  // fa, fb, na / nt, h_c^3 na nb / nt
  __shared__ int form;      // 0: both empty, 1: dst empty, 2: src holds the larger shift (fb = 1), 3: dst does
  if (threadIdx.x == 0) {
    const double na = dsc[MLSGD_S_COUNT], nb = ssc[MLSGD_S_COUNT], nt = na + nb;
    const double shift = fmax(dsc[MLSGD_S_SHIFT], ssc[MLSGD_S_SHIFT]);
    const double fa = na > 0.0 ? exp(theta * (dsc[MLSGD_S_SHIFT] - shift)) : 0.0;
    const double fb = nb > 0.0 ? exp(theta * (ssc[MLSGD_S_SHIFT] - shift)) : 0.0;
    const bool some = nt > 0.0;
    form = !some ? 0 : (fb == 1.0 ? (na == 0.0 ? 1 : 2) : 3);
    co[0] = fa;
    co[1] = fb;
    co[2] = some ? na / nt : 0.0;
    co[3] = some ? hc3 * na * nb / nt : 0.0;
  }
  __syncthreads();
  const double fa = co[0], fb = co[1], w = co[2];
  const long long step = (long long)gridDim.x * kBlock;
  const long long i0 = (long long)blockIdx.x * kBlock + threadIdx.x;
  double acc = 0.0;
  if (form == 1) {
#pragma unroll 4
    for (long long i = i0; i < n; i += step) {
      const double b = sf[i];
      df[i] = fma(w, b, b);  // w = 0: b (NaN for an infinite b, as w (a - b) gives)
    }
  } else if (form == 2) {
#pragma unroll 4
    for (long long i = i0; i < n; i += step) {
      const double b = sf[i], d = fma(df[i], fa, -b);
      df[i] = fma(w, d, b);
      acc = fma(d, d, acc);
    }
  } else if (form == 3) {
#pragma unroll 4
    for (long long i = i0; i < n; i += step) {
      const double b = sf[i] * fb, d = fma(df[i], fa, -b);
      df[i] = fma(w, d, b);
      acc = fma(d, d, acc);
    }
  }
  const double bs = block_sum(acc);
  if (threadIdx.x == 0) partial[blockIdx.x] = co[3] * bs;
}

__global__ void __launch_bounds__(kBlock) k_merge_scalars(const double* __restrict__ partial, int nblk,
                                                          double* __restrict__ dsc, const double* __restrict__ ssc,
                                                          double theta) {
  pdl_entry();
  double v = 0.0;
  for (int t = threadIdx.x; t < nblk; t += kBlock) v += partial[t];
  v = block_sum(v);
  if (threadIdx.x != 0) return;
  const double na = dsc[MLSGD_S_COUNT], nb = ssc[MLSGD_S_COUNT];
  const double nt = na + nb;
  if (nt <= 0.0) return;
  const double shift = fmax(dsc[MLSGD_S_SHIFT], ssc[MLSGD_S_SHIFT]);
  const double fa = na > 0.0 ? exp(theta * (dsc[MLSGD_S_SHIFT] - shift)) : 0.0;
  const double fb = nb > 0.0 ? exp(theta * (ssc[MLSGD_S_SHIFT] - shift)) : 0.0;
  const double ya = dsc[MLSGD_S_MEAN_DY] * fa, yb = ssc[MLSGD_S_MEAN_DY] * fb;
  const double d = ya - yb;
  dsc[MLSGD_S_MEAN_DY] = yb + (na / nt) * d;
  dsc[MLSGD_S_S2_DY] = dsc[MLSGD_S_S2_DY] * fa * fa + ssc[MLSGD_S_S2_DY] * fb * fb + d * d * na * nb / nt;
  dsc[MLSGD_S_S2_DX] = dsc[MLSGD_S_S2_DX] * fa * fa + ssc[MLSGD_S_S2_DX] * fb * fb + v;
  dsc[MLSGD_S_COUNT] = nt;
  dsc[MLSGD_S_SHIFT] = shift;
  dsc[MLSGD_S_PHI_MAX] = fmax(dsc[MLSGD_S_PHI_MAX], ssc[MLSGD_S_PHI_MAX]);
  dsc[MLSGD_S_ITERS] += ssc[MLSGD_S_ITERS];
  dsc[MLSGD_S_NOCONV] += ssc[MLSGD_S_NOCONV];
}

void launch_stats_merge(double* dfield, double* dsc, const double* sfield, const double* ssc, long long ncells,
                        double hc3, double theta, double* partial, cudaStream_t st) {
  const int nblk = cell_blocks(ncells);
  launch("merge", (double)ncells * 24, k_merge_field, dim3(nblk), kBlock, 0, st, dfield, (const double*)dsc, sfield,
         ssc, ncells, theta, hc3, partial);
  launch("merge_scalars", 0.0, k_merge_scalars, dim3(1), kBlock, 0, st, (const double*)partial, nblk, dsc, ssc, theta);
}

// ---------------------------------------------------------------- combine and step
// EX = sum_l f_l mean_l (f_l = exp(theta (c_l - c*))), grad = EX / denom + alpha z,
// z <- z - tau grad when `update`.  partial rows: 0 = ||grad||^2, 1 = ||EX||^2,
// 2 = ||grad - gprev||^2, 3 = ||gprev||^2 (0 without gprev), 4 = ||z||^2 (before the
// step), 5+l = ||mean_l||^2
// (unscaled, counted without h_c^3).
// Bound: FP64 issue (2 L + 6 operations per cell of L levels, 2 per clock and SM), then
// HBM (L + 3 words per cell).  At most kCellBlocks blocks march over the cells,
// so the L + 5 block reductions are paid once per block and not once per 256 cells; the
// level count is a template parameter, which keeps the L running sums in registers; the
// division by the denominator is one reciprocal per thread and three operations per cell
// (some twenty for a division; the quotient rounded once more, one operation per cell: six
// levels on a 256^3 control reset, merged twice and stepped 1.88 ms, 1.94 with these three).
struct FieldList { const double* f[16]; };

// a / b correctly rounded, with y = 1/b correctly rounded: the quotient's residual is exact in
// an FMA and corrects it (Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", 1990).  By a division where a or b is so large or small that a step
// could leave the normal range (`plain`: b is).
__device__ __forceinline__ double quotient(double a, double b, double y, bool plain) {
  constexpr unsigned lo = (1023u - 700u) << 20, hi = (1023u + 700u) << 20;  // 2^-700 <= |a| < 2^700
  const unsigned h = (unsigned)__double2hiint(a) & 0x7fffffffu;
  if (plain || h - lo >= hi - lo) return a / b;
  const double q = a * y;
  return fma(fma(-q, b, a), y, q);
}

template <int L>
__global__ void __launch_bounds__(kBlock) k_combine_step(FieldList fl, const double* __restrict__ factors, long long n,
                                                         double denom, double alpha, double tau, int update,
                                                         double* __restrict__ z, double* __restrict__ grad,
                                                         const double* __restrict__ gprev, double* __restrict__ partial,
                                                         int nblk) {
  pdl_entry();
  double fac[L], ml[L];
#pragma unroll
  for (int l = 0; l < L; ++l) {
    fac[l] = factors[l];
    ml[l] = 0.0;
  }
  const double inv = 1.0 / denom;
  const bool plain = !(denom > 0x1p-200 && denom < 0x1p200);
  double row[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  const long long step = (long long)gridDim.x * kBlock;
#pragma unroll 2
  for (long long i = (long long)blockIdx.x * kBlock + threadIdx.x; i < n; i += step) {
    double m[L];
#pragma unroll
    for (int l = 0; l < L; ++l) m[l] = fl.f[l][i];
    const double zi = z[i];
    double ex = fac[0] * m[0];
    ml[0] = fma(m[0], m[0], ml[0]);
#pragma unroll
    for (int l = 1; l < L; ++l) {
      ex = fma(fac[l], m[l], ex);
      ml[l] = fma(m[l], m[l], ml[l]);
    }
    const double g = fma(alpha, zi, quotient(ex, denom, inv, plain));
    row[0] = fma(g, g, row[0]);
    row[1] = fma(ex, ex, row[1]);
    row[4] = fma(zi, zi, row[4]);
    if (gprev) {
      const double gp = gprev[i], d = g - gp;
      row[2] = fma(d, d, row[2]);
      row[3] = fma(gp, gp, row[3]);
    }
    if (grad) grad[i] = g;
    if (update) z[i] = fma(-tau, g, zi);
  }
#pragma unroll
  for (int r = 0; r < 5 + L; ++r) {
    const double v = block_sum(r < 5 ? row[r < 5 ? r : 0] : ml[r < 5 ? 0 : r - 5]);
    if (threadIdx.x == 0) partial[(long long)r * nblk + blockIdx.x] = v;
    __syncthreads();
  }
}

// z <- z - tau g, and gout <- g (the gradient kept for the next step size)
__global__ void k_step_apply(long long n, double tau, const double* __restrict__ g, double* __restrict__ z,
                             double* __restrict__ gout) {
  pdl_entry();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double gi = g[i];
  z[i] -= tau * gi;
  gout[i] = gi;
}

// out[r] = sum of row r of partial (one block per row)
__global__ void __launch_bounds__(kBlock) k_rows_finish(const double* __restrict__ partial, int nblk,
                                                        double* __restrict__ out) {
  pdl_entry();
  double v = 0.0;
  for (int t = threadIdx.x; t < nblk; t += kBlock) v += partial[(long long)blockIdx.x * nblk + t];
  v = block_sum(v);
  if (threadIdx.x == 0) out[blockIdx.x] = v;
}

int combine_blocks(long long ncells) { return cell_blocks(ncells); }

void launch_combine_step(const double* const* fields, const double* factors, int L, long long ncells, double denom,
                         double alpha, double tau, bool update, double* z, double* grad, const double* gprev,
                         double* partial, int nblk, cudaStream_t st) {
  FieldList fl;
  for (int l = 0; l < L && l < 16; ++l) fl.f[l] = fields[l];
  const double bytes = (double)ncells * 8 * (L + 1 + (update ? 1 : 0) + (grad ? 1 : 0) + (gprev ? 1 : 0));
  using Kern = decltype(&k_combine_step<1>);
  static const Kern kern[16] = {k_combine_step<1>,  k_combine_step<2>,  k_combine_step<3>,  k_combine_step<4>,
                                k_combine_step<5>,  k_combine_step<6>,  k_combine_step<7>,  k_combine_step<8>,
                                k_combine_step<9>,  k_combine_step<10>, k_combine_step<11>, k_combine_step<12>,
                                k_combine_step<13>, k_combine_step<14>, k_combine_step<15>, k_combine_step<16>};
  launch("combine", bytes, kern[L - 1], dim3(nblk), kBlock, 0, st, fl, factors, ncells, denom, alpha, tau,
         update ? 1 : 0, z, grad, gprev, partial, nblk);
  const int rows = L + 5;
  launch("combine_finish", 0.0, k_rows_finish, dim3(rows), kBlock, 0, st, (const double*)partial, nblk,
         partial + (long long)rows * nblk);
}

void launch_step_apply(long long ncells, double tau, const double* g, double* z, double* gout, cudaStream_t st) {
  const int nblk = (int)((ncells + kBlock - 1) / kBlock);
  launch("step_apply", (double)ncells * 32, k_step_apply, dim3(nblk), kBlock, 0, st, ncells, tau, g, z, gout);
}

}  // namespace mlsgd
