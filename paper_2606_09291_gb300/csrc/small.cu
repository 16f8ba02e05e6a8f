// small.cu - a whole mixed-precision solve on an 8^3 or 16^3 grid in one launch, one
// block per sample (rows a4, a6).
//
// On these grids a pass over a sample is a few thousand nodes: run pass by pass, a solve
// is some 200 dependent launches (22 per inner PCG iteration with the V-cycle level by
// level), each a few microseconds of launch latency, partial sums in global memory and
// tail, whatever the batch.  Everything a sample needs fits the shared memory of one
// block (8^3: 27 KB; 16^3: 108 KB), so here a block keeps its sample's coefficient
// levels, operand and residuals on the SM and runs the refinement loop to the end:
// coarse coefficients, FP32 inner PCG with its V(1,1)-cycle, FP64-accurate residual,
// stop test.  What bounds it (ncu, 1024 samples of 8^3 and 64 of 16^3): latency, of shared
// memory and of about 14 block barriers per inner iteration (8 and 5 of 21 cycles per
// instruction of a warp on 8^3, 3 and 4 of 15 on 16^3); issue is 45 and 53% busy.  FP64 in one
// warp (64 clocks an operation) is kept out of the inner iterations; the FP64 refinement
// residuals of 8^3 take 45% of that pipe.
// Measured (three refinement steps of six iterations, state or adjoint): 1024 samples of
// 8^3 180 us a solve (310 with a thread per node instead of per interior node; at about 300
// samples, where both are one wave, 117 against 115) against 2.2 ms in passes, 256 of 16^3
// 320 us against 3.1 ms, 64 of 16^3 200 us against 1.6 ms.
//
// Arithmetic: that of the pass-by-pass solver on the same grid (solver.cu for 8^3: FP64
// refinement residual and solution; tiled.cu for 16^3: solution and b as FP32 pairs, partial
// sums per thread over 8 planes and the rows of a thread), except that the 4^3 and 2^3 levels
// are one matrix (coarse4_build) and that the sums of the FP32 partial sums of r.z and p.q, and
// their quotients alpha and beta, are formed in FP32 pairs (46 bits) while those hold them, in
// FP64 beyond (alpha64); alpha and beta are FP32 numbers either way.  30 drawn calls on 8^3 and
// 16^3 against 64 bits: 1.001 times the pass-by-pass solver's error, by rtol in both.
#include "internal.cuh"
#include "kernels.h"
#include "launch.h"
#include "levels.cuh"
#include "onchip.cuh"
#include "refine.cuh"

namespace mlsgd {

namespace {

struct SmallArgs {
  const float* a32;           // operator coefficient [S][N^3]
  const __nv_bfloat16* abf;   // V-cycle coefficient [S][N^3]
  const double* b;            // right-hand side (FP64), or null with bp
  const float2* bp;           // right-hand side as FP32 (hi, lo) pairs (16^3 only)
  long long bstride;          // nodes between samples of b / bp (0: one vector for all)
  double* x64;                // solution in FP64 [S][nodes], or null with xp
  float2* xp;                 // 16^3: solution as FP32 pairs [S][nodes] (always written)
  SolveScalars* sc;
  double tol2;
  float omega;
  int fixed;                  // > 0: that many refinement steps
  int cap;                    // refinement steps after which a solve gives up
  int inner, inner_next;      // inner iterations of the first and the later steps
};

// mean of the eight children (the coarse coefficient), FP32 sums in the order of k_coarsen_coef
__device__ __forceinline__ float coarsen_cell(const float* af, int c, int Nc) {
  const int I = c % Nc, J = (c / Nc) % Nc, K = c / (Nc * Nc), Nf = 2 * Nc;
  const float* f = af + 2 * I + Nf * (2 * J + Nf * 2 * K);
  float acc = 0.f;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) acc += f[p + Nf * (q + Nf * r)];
  return 0.125f * acc;
}

// ---------------------------------------------------------------- 8^3
// a thread per interior node (343): 11 warps and four blocks per SM, where one per node (729)
// left half the lanes of every step idle in 24 warps and two blocks
constexpr int kT8 = 352, kW8 = kT8 / 32;

__device__ __forceinline__ double sum_groups(double v) {  // lane l holds warp l's sum (l < 24, else 0)
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const double p0 = __shfl_sync(0xffffffffu, v, 0), p1 = __shfl_sync(0xffffffffu, v, 8),
               p2 = __shfl_sync(0xffffffffu, v, 16);  // lanes 8g: the block sum of group g
  return (p0 + p2) + p1;
}

// floats of the levels from 8^3 down: x8, t8, t4, the 4^3 matrix and its vectors, a4, a2;
// on 16^3 also r8 and a8
constexpr int kLv8 = 2 * 729 + 125 + 27 * 27 + 54 + 64 + 8, kLv16 = kLv8 + 729 + 512;

// a / b of two pairs (about 46 bits) rounded to FP32; 0 unless ok
__device__ __forceinline__ float df_quotient(DF a, DF b, bool ok) {
  if (!ok) return 0.f;
  const float q = __fdiv_rn(a.h, b.h);
  const float p = __fmul_rn(q, b.h), e = __fmaf_rn(q, b.h, -p);
  const float rem = __fsub_rn(__fsub_rn(__fsub_rn(a.h, p), e), __fmaf_rn(q, b.l, -a.l));
  const float c = __fdiv_rn(rem, b.h);
  return fabsf(c) < INFINITY ? __fadd_rn(q, c) : q;
}

// alpha = rz / pq and beta = rz / rz_old from pairs; NaN where a sum is beyond FP32 (its pair is NaN)
__device__ __forceinline__ float pair_alpha(DF rz, DF pq) {
  return df_quotient(rz, pq, !(pq.h <= 0.f) && rz.h != 0.f);
}
__device__ __forceinline__ float pair_beta(DF rz, DF old) { return df_quotient(rz, old, old.h != 0.f); }
// Then they are formed again from the partial sums, M.redf[0] of r.z and M.redf[1] of p.q, by
// FP64 sums and quotients, those of the pass-by-pass solver (SM_ALPHA, SM_BETA in solver.cu):
// a right-hand side whose products leave the FP32 range ends as it does there.  Small sums
// need no such care: from 2^-100 down the pairs' error tends to 2^-149, still under the
// rounding of the FP32 partial sums themselves.  Out of line and with no state but M.rz (the
// last FP64 r.z), since the inner iterations have no register to spare: a level gradient of 1024
// samples of 8^3 took 729 us without this and 735 with it, 64 samples of 16^3 the same (FP64
// forms of the inner or the whole solve beside the pairs': 0.7 to 3% more on 8^3, 6% on 16^3).
// Every thread calls them with the same values.
template <typename SM>
__device__ __noinline__ float alpha64(SM& M) {
  const double rz = M.sum64(0), pq = M.sum64(1);
  M.rz = rz;
  return (float)((pq > 0.0 && rz != 0.0) ? rz / pq : 0.0);
}
template <typename SM>
__device__ __noinline__ float beta64(SM& M, DF old) {
  const double o = isnan(old.h) ? M.rz : df_to_double(old);
  return (float)(o != 0.0 ? M.sum64(0) / o : 0.0);
}

struct Smem8 {
  double xd[729];       // solution for the refinement residual
  double redd[kW8], rz;
  float a32[512], abf[512];
  float op[729];        // operand of A p
  float r8[729];        // residual of the V-cycle
  float lv[kLv8];
  float redf[2][kW8];
  int go;
  __device__ double sum64(int which) const {
    double v = 0.0;
    for (int w = 0; w < kW8; ++w) v += (double)redf[which][w];
    return v;
  }
};

__global__ void __launch_bounds__(kT8, 4) k_small8(SmallArgs A) {
  pdl_entry();
  __shared__ Smem8 M;
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float omega = A.omega;
  for (int c = tid; c < 512; c += kT8) {
    M.a32[c] = A.a32[(long long)s * 512 + c];
    M.abf[c] = __bfloat162float(A.abf[(long long)s * 512 + c]);
  }
  const bool in = tid < 343;  // the thread's interior node
  const int i = 1 + tid % 7, j = 1 + (tid / 7) % 7, k = 1 + tid / 49, n = in ? i + 9 * (j + 9 * k) : 0;
  const double bv = in ? A.b[s * A.bstride + n] : 0.0;  // b is 0 on the boundary
  for (int e = tid; e < 729; e += kT8) {
    M.op[e] = M.r8[e] = 0.f;
    M.xd[e] = 0.0;
  }
  for (int e = tid; e < kLv8; e += kT8) M.lv[e] = 0.f;
  CoarseLevels L;
  L.r8 = M.r8; L.a8 = M.abf;
  L.x8 = M.lv; L.t8 = L.x8 + 729;
  L.t4 = L.t8 + 729; L.g4 = L.t4 + 125; L.s4 = L.g4 + 729;
  float* a4 = L.s4 + 54;
  float* a2 = a4 + 64;
  L.x4 = nullptr; L.a4 = a4; L.a2 = a2;
  __syncthreads();
  if (tid < 64) a4[tid] = coarsen_cell(M.abf, tid, 4);
  const float w8 = in ? omega / diag_of<8>(M.abf, i, j, k) : 0.f;
  __syncthreads();
  if (tid < 8) a2[tid] = coarsen_cell(a4, tid, 2);
  __syncthreads();
  coarse4_build<kT8>(L, omega);
  Outer o{0.0, 0.0, 0.0, 0, 0, 0};
  // block sum of a double, result in warp 0
  auto sum64 = [&](double v) {
    v = warp_sum(v);
    if (lane == 0) M.redd[warp] = v;
    __syncthreads();
    double g = 0.0;
    if (warp == 0) {
      g = lane < kW8 ? M.redd[lane] : 0.0;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
    }
    return g;
  };
  // block sum of a float as a pair, in every thread (FP64 additions and a division in one
  // warp were a quarter of an iteration)
  auto sum32 = [&](float v, int which) {  // 0: r.z, 1: p.q
    v = warp_sum(v);
    if (lane == 0) M.redf[which][warp] = v;
    __syncthreads();
    DF g{lane < kW8 ? M.redf[which][lane] : 0.f, 0.f};
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
      g = df_add(g, DF{__shfl_xor_sync(0xffffffffu, g.h, o), __shfl_xor_sync(0xffffffffu, g.l, o)});
    return DF{__shfl_sync(0xffffffffu, g.h, 0), __shfl_sync(0xffffffffu, g.l, 0)};
  };
  DF rz{0.f, 0.f};  // r . z
  {
    const double v = sum64(bv * bv);
    if (tid == 0) {
      o.bb = o.rr = v;
      bool go = v > 0.0;
      if (!(v < INFINITY)) { go = false; o.status = 2; }
      M.go = go;
    }
  }
  __syncthreads();
  double x = 0.0;
  bool go = M.go != 0;
  for (int step = 0; go; ++step) {
    double r64 = bv;
    if (step > 0) {  // r = b - A x in FP64
      if (in) M.xd[n] = x;
      __syncthreads();
      r64 = 0.0;
      if (in) {
        Cells8<double, float> C;
        C.sum = 0.0;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              const double v = (double)M.a32[(i - 1 + p) + 8 * ((j - 1 + q) + 8 * (k - 1 + r))];
              C.c[p][q][r] = v;
              C.sum += v;
            }
        r64 = bv - (1.0 / (12.0 * 8)) * q1_row(C, (const double*)M.xd, i, j, k, 9);
      }
      const double v = sum64(r64 * r64);
      if (tid == 0) M.go = outer_go(o, v, A.tol2, A.cap);
      __syncthreads();
      go = M.go != 0;
      if (!go) break;
    }
    if (A.fixed > 0 && step == A.fixed) break;
    const int inner = step == 0 ? A.inner : A.inner_next;
    float r = (float)r64, d = 0.f, p = 0.f;
    for (int it = 0;; ++it) {
      if (in) M.r8[n] = r;
      __syncthreads();
      const float z = vcycle8<kT8, true>(L, n, i, j, k, in, w8, omega);
      const DF rzn = sum32(r * z, 0);
      float be = it > 0 ? pair_beta(rzn, rz) : 0.f;
      if (isnan(be)) be = beta64(M, rz);
      p = it > 0 ? z + be * p : z;
      rz = rzn;
      if (in) M.op[n] = p;
      __syncthreads();
      float q = 0.f;
      if (in) {
        Cells8<float, float> C;
        cells8(C, M.a32, i, j, k, 8);
        q = float(1.0 / (12.0 * 8)) * q1_row(C, (const float*)M.op, i, j, k, 9);
      }
      const DF pq = sum32(p * q, 1);
      float al = pair_alpha(rz, pq);
      if (isnan(al)) al = alpha64(M);
      d += al * p;
      if (it == inner - 1) break;
      r = r - al * q;
    }
    x += (double)d;
    if (tid == 0) { o.iters += 1; o.pad += inner; }
  }
  o.rz = df_to_double(rz);
  __syncthreads();
  if (in) M.xd[n] = x;  // the boundary is 0
  __syncthreads();
  for (int e = tid; e < 729; e += kT8) A.x64[(long long)s * 729 + e] = M.xd[e];
  if (tid == 0) store_scalars(A.sc + s, o);
}

// ---------------------------------------------------------------- 16^3
// 1024 threads: thread (xq, yq, g) owns the nodes x = xq + 1, y = yq + 1 of the planes
// 4g + 1 .. 4g + 4 (xq, yq < 15; plane 16 is the boundary), whose r, p, z, q, correction
// and omega D^-1 stay in its registers.  Shared memory holds what neighbours read: the
// operand, the residual to restrict, and the vectors whose dot product the threads of the
// tile passes would sum.
constexpr int kT16 = 1024;
constexpr int kN16 = 17 * 17 * 17;

struct Smem16 {
  float b0[kN16];  // operand of a stencil; with b1: the solution pairs of a refinement residual
  float b1[kN16];  // t, then r (dot)
  float b2[kN16];  // z, q or the refinement residual (dot)
  float a32[4096], abf[4096];
  float lv[kLv16];
  double redd[24], rz;
  float redf[2][8];
  int go;
  __device__ double sum64(int which) const {  // the block sums of the two segments, as `dot` forms them
    const float* w = redf[which];
    return (double)((w[0] + w[2]) + (w[1] + w[3])) + (double)((w[4] + w[6]) + (w[5] + w[7]));
  }
};
static_assert(sizeof(Smem16) <= 227 * 1024, "shared memory");

// operator row over h/12 of tiled.cu's passes: three partial sums, operand window and
// cells read from shared memory
__device__ __forceinline__ float q1_tile(const float* x, const float* a, int n, int c) {
  float C[2][2][2];  // [r][p][q]
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q) C[r][p][q] = a[c + p + 16 * q + 256 * r];
  auto X = [&](int pl, int u, int v) { return x[n + (u - 1) + 17 * (v - 1) + 289 * (pl - 1)]; };
  float pxy[2][2], pxz[2][2], pyz[2][2];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      pxy[v][u] = C[0][u][v] + C[1][u][v];
      pxz[v][u] = C[v][u][0] + C[v][u][1];
      pyz[v][u] = C[v][0][u] + C[v][1][u];
    }
  const float sum8 = (pxy[0][0] + pxy[0][1]) + (pxy[1][0] + pxy[1][1]);
  float accp[3];
  accp[1] = 4.f * sum8 * X(1, 1, 1);
#pragma unroll
  for (int v = 0; v < 2; ++v)
#pragma unroll
    for (int u = 0; u < 2; ++u) accp[1] -= pxy[v][u] * X(1, 2 * u, 2 * v);
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int pl = 2 * r;
    float a2 = 0.f;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      a2 -= pxz[r][u] * X(pl, 2 * u, 1);
      a2 -= pyz[r][u] * X(pl, 1, 2 * u);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) a2 -= C[r][p][q] * X(pl, 2 * p, 2 * q);
    accp[pl] = a2;
  }
  return accp[1] + (accp[0] + accp[2]);
}

__global__ void __launch_bounds__(kT16, 1) k_small16(SmallArgs A) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smraw[];
  Smem16& M = *reinterpret_cast<Smem16*>(smraw);
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int xq = tid & 15, yq = (tid >> 4) & 15, g = tid >> 8;
  const float omega = A.omega, scale = float(1.0 / (12.0 * 16));
  const bool col = xq < 15 && yq < 15;
  const int nu = col ? (g == 3 ? 3 : 4) : 0;               // own nodes
  const int n0 = (xq + 1) + 17 * (yq + 1) + 289 * (4 * g + 1);  // first own node
  const int c0 = xq + 16 * yq + 256 * (4 * g);                  // its lowest cell
  for (int c = tid; c < 4096; c += kT16) {
    M.a32[c] = A.a32[(long long)s * 4096 + c];
    M.abf[c] = __bfloat162float(A.abf[(long long)s * 4096 + c]);
  }
  for (int e = tid; e < kN16; e += kT16) M.b0[e] = M.b1[e] = 0.f;
  for (int e = tid; e < kLv16; e += kT16) M.lv[e] = 0.f;
  CoarseLevels L;
  L.r8 = M.lv; L.x8 = L.r8 + 729; L.t8 = L.x8 + 729;
  float* a8 = L.t8 + 729;
  L.t4 = a8 + 512; L.g4 = L.t4 + 125; L.s4 = L.g4 + 729;
  float* a4 = L.s4 + 54;
  float* a2 = a4 + 64;
  L.x4 = nullptr; L.a8 = a8; L.a4 = a4; L.a2 = a2;
  // the right-hand side's pair at node n of this sample
  auto b_pair = [&](int n) {
    return A.bp ? A.bp[s * A.bstride + n] : df_split(A.b[s * A.bstride + n]);
  };
  // boundary nodes of the outputs
  for (int e = tid; e < kN16; e += kT16) {
    int i, j, k;
    node_ijk(e, 17, i, j, k);
    const bool in = interior(i, j, k, 16);
    M.b2[e] = 0.f;
    if (!in) {
      A.xp[(long long)s * kN16 + e] = make_float2(0.f, 0.f);
      if (A.x64) A.x64[(long long)s * kN16 + e] = 0.0;
    }
  }
  __syncthreads();
  float r[4], p[4], z[4], d[4], dv[4], q[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    r[u] = p[u] = z[u] = d[u] = dv[u] = q[u] = 0.f;
    if (u < nu) {
      r[u] = b_pair(n0 + 289 * u).x;
      M.b2[n0 + 289 * u] = r[u];
      auto sum4 = [&](int c) { return (M.abf[c] + M.abf[c + 1]) + (M.abf[c + 16] + M.abf[c + 17]); };
      const float below = sum4(c0 + 256 * u), above = sum4(c0 + 256 * (u + 1));
      dv[u] = omega * __fdividef(1.0f, float(1.0 / 48.0) * (below + above));
    }
  }
  for (int c = tid; c < 512; c += kT16) a8[c] = coarsen_cell(M.abf, c, 8);
  __syncthreads();
  if (tid < 64) a4[tid] = coarsen_cell(a8, tid, 4);
  // node of the 8^3 level
  int i8 = 0, j8 = 0, k8 = 0;
  if (tid < 729) node_ijk(tid, 9, i8, j8, k8);
  const bool in8 = tid < 729 && interior(i8, j8, k8, 8);
  const float w8 = in8 ? omega / diag_of<8>(L.a8, i8, j8, k8) : 0.f;
  __syncthreads();
  if (tid < 8) a2[tid] = coarsen_cell(a4, tid, 2);
  __syncthreads();
  coarse4_build<kT16>(L, omega);
  Outer o{0.0, 0.0, 0.0, 0, 0, 0};
  // ||b||^2 as the solver's init pass sums it: three blocks of 256 threads, eight nodes a
  // thread at stride 256 (FP32 over the pair heads; FP64 for an FP64 right-hand side of its own)
  {
    const bool own64 = !A.bp && A.bstride != 0;
    double v = 0.0;
    if (tid < 768) {
      const int m0 = (tid >> 8) * 2048 + (tid & 255);
      float f = 0.f;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int n = m0 + 256 * t;
        if (n >= kN16) continue;
        if (own64) {
          int ii, jj, kk;
          node_ijk(n, 17, ii, jj, kk);
          if (interior(ii, jj, kk, 16)) {
            const double bv = A.b[s * A.bstride + n];
            v = fma(bv, bv, v);
          }
        } else {
          f = __fmaf_rn(M.b2[n], M.b2[n], f);
        }
      }
      if (!own64) v = (double)f;
      v = warp_sum(v);
      if (lane == 0) M.redd[warp] = v;
    }
    __syncthreads();
    if (warp == 0) {
      v = sum_groups(lane < 24 ? M.redd[lane] : 0.0);
      if (lane == 0) {
        o.bb = o.rr = v;
        bool go = v > 0.0;
        if (!(v < INFINITY)) { go = false; o.status = 2; }
        M.go = go;
      }
    }
  }
  __syncthreads();
  // dot product of two shared vectors in the order of the tile passes: thread (tx, ty) of
  // segment sg sums rows 4 ty + 1 .. 4 ty + 4 over the segment's eight planes, then the
  // block sum of the segment, then the two segments (a pair, in every thread)
  auto dot = [&](const float* u, const float* v, int which) {  // 0: r.z, 1: p.q
    if (warp < 8) {
      const int sg = warp >> 2, ty = warp & 3;
      float red = 0.f;
      if (lane < 15) {
        const int base = lane + 1 + 17 * (4 * ty + 1) + 289 * (8 * sg + 1);
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (8 * sg + k < 15 && 4 * ty + t < 15) {
              const int n = base + 17 * t + 289 * k;
              red = __fmaf_rn(u[n], v[n], red);
            }
      }
      red = warp_sum(red);
      if (lane == 0) M.redf[which][warp] = red;
    }
    __syncthreads();
    float w = lane < 8 ? M.redf[which][lane] : 0.f;
    w += __shfl_xor_sync(0xffffffffu, w, 2);
    w += __shfl_xor_sync(0xffffffffu, w, 1);
    const float p0 = __shfl_sync(0xffffffffu, w, 0), p1 = __shfl_sync(0xffffffffu, w, 4);
    return df_add(DF{p0, 0.f}, DF{p1, 0.f});
  };
  DF rz{0.f, 0.f};  // r . z
  bool go = M.go != 0;
  const float2 zero2 = make_float2(0.f, 0.f);
  if (!go) {  // no step is taken: x = 0
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < nu) A.xp[(long long)s * kN16 + n0 + 289 * u] = zero2;
  }
  for (int step = 0; go; ++step) {
    if (step > 0) {  // r = b - A x from the pairs, error-free products and sums in FP32
      float2* xs = reinterpret_cast<float2*>(M.b0);  // b0 and b1
      __syncthreads();                               // the last step's reads of b0, b1
      for (int e = tid; e < kN16; e += kT16) xs[e] = A.xp[(long long)s * kN16 + e];
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) {
          const int n = n0 + 289 * u, c = c0 + 256 * u;
          auto X = [&](int pl, int a, int b) { return xs[n + (a - 1) + 17 * (b - 1) + 289 * (pl - 1)]; };
          auto C = [&](int rr, int pp, int qq) { return M.a32[c + pp + 16 * qq + 256 * rr]; };
          r[u] = refine_residual(C, X, b_pair(n), 16);
          M.b2[n] = r[u];
        }
      __syncthreads();
      double v = 0.0;
      if (warp < 16) {  // rows 2 ty + 1, 2 ty + 2 of segment sg
        const int sg = warp >> 3, ty = warp & 7;
        float red = 0.f;
        if (lane < 15) {
          const int base = lane + 1 + 17 * (2 * ty + 1) + 289 * (8 * sg + 1);
#pragma unroll
          for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int t = 0; t < 2; ++t)
              if (8 * sg + k < 15 && 2 * ty + t < 15) {
                const float rv = M.b2[base + 17 * t + 289 * k];
                red = __fmaf_rn(rv, rv, red);
              }
        }
        v = warp_sum((double)red);
        if (lane == 0) M.redd[warp] = v;
      }
      __syncthreads();
      if (warp == 0) {
        v = lane < 16 ? M.redd[lane] : 0.0;
#pragma unroll
        for (int w = 4; w > 0; w >>= 1) v += __shfl_xor_sync(0xffffffffu, v, w);
        v = __shfl_sync(0xffffffffu, v, 0) + __shfl_sync(0xffffffffu, v, 8);
        if (lane == 0) M.go = outer_go(o, v, A.tol2, A.cap);
      }
      for (int e = tid; e < 2 * kN16; e += kT16) M.b0[e] = 0.f;  // boundary nodes of b0 and b1
      __syncthreads();
      go = M.go != 0;
      if (!go) break;
    }
    if (A.fixed > 0 && step == A.fixed) break;
    const int inner = step == 0 ? A.inner : A.inner_next;
    float al = 0.f;
    for (int it = 0;; ++it) {
      // V-cycle on r: pre-smoothing, residual, 8^3 and below, prolongation, post-smoothing
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) M.b0[n0 + 289 * u] = r[u] * dv[u];
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) M.b1[n0 + 289 * u] = __fmaf_rn(-scale, q1_tile(M.b0, M.abf, n0 + 289 * u, c0 + 256 * u), r[u]);
      __syncthreads();
      if (in8) {
        const float* f = M.b1 + 2 * i8 + 17 * (2 * j8) + 289 * (2 * k8);
        float v = 0.f;
#pragma unroll
        for (int w = -1; w <= 1; ++w)
#pragma unroll
          for (int b = -1; b <= 1; ++b)
#pragma unroll
            for (int a = -1; a <= 1; ++a) {
              const float wt = float((a == 0 ? 1.0 : 0.5) * (b == 0 ? 1.0 : 0.5) * (w == 0 ? 1.0 : 0.5));
              v += wt * f[a + 17 * b + 289 * w];
            }
        L.r8[tid] = v;
      }
      __syncthreads();
      (void)vcycle8<kT16, true>(L, tid, i8, j8, k8, in8, w8, omega);
      __syncthreads();
      const int px = (xq + 1) & 1, py = (yq + 1) & 1;
      const float* e8 = L.t8 + ((xq + 1) >> 1) + 9 * ((yq + 1) >> 1);
      auto plane = [&](int c) {  // coarse plane c interpolated in x and y
        const float* e = e8 + 81 * c;
        const float e00 = e[0];
        if (!px && !py) return e00;
        if (!py) return (e00 + e[1]) * 0.5f;
        if (!px) return (e00 + e[9]) * 0.5f;
        return ((e00 + e[1]) * 0.5f + (e[9] + e[10]) * 0.5f) * 0.5f;
      };
      float x2[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) {
          const int k = 4 * g + 1 + u;
          const float y = (k & 1) ? (plane(k >> 1) + plane((k >> 1) + 1)) * 0.5f : plane(k >> 1);
          x2[u] = __fadd_rn(__fmul_rn(r[u], dv[u]), y);  // rounded product first, as the tile pass
          M.b0[n0 + 289 * u] = x2[u];
        }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) {
          const float res = __fmaf_rn(-scale, q1_tile(M.b0, M.abf, n0 + 289 * u, c0 + 256 * u), r[u]);
          z[u] = __fmaf_rn(res, dv[u], x2[u]);
          M.b1[n0 + 289 * u] = r[u];
          M.b2[n0 + 289 * u] = z[u];
        }
      __syncthreads();
      const DF rzn = dot(M.b1, M.b2, 0);
      // p = z + beta p, q = A p
      float be = it == 0 ? 0.f : pair_beta(rzn, rz);
      if (isnan(be)) be = beta64(M, rz);
      rz = rzn;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) {
          p[u] = it == 0 ? z[u] : __fmaf_rn(be, p[u], z[u]);
          M.b0[n0 + 289 * u] = p[u];
        }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < nu) {
          q[u] = scale * q1_tile(M.b0, M.a32, n0 + 289 * u, c0 + 256 * u);
          M.b2[n0 + 289 * u] = q[u];
        }
      __syncthreads();
      const DF pq = dot(M.b0, M.b2, 1);
      al = pair_alpha(rz, pq);
      if (isnan(al)) al = alpha64(M);
      if (it == inner - 1) break;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        d[u] = it == 0 ? al * p[u] : __fmaf_rn(al, p[u], d[u]);
        r[u] = __fmaf_rn(-al, q[u], r[u]);
      }
    }
    // x (+)= d + alpha p in pair arithmetic
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < nu) {
        const float inc = inner > 1 ? __fmaf_rn(al, p[u], d[u]) : al * p[u];
        float2* xo = A.xp + (long long)s * kN16 + n0 + 289 * u;
        *xo = step == 0 ? make_float2(inc, 0.f) : pair_add(*xo, inc);
      }
    if (tid == 0) { o.iters += 1; o.pad += inner; }
  }
  if (A.x64) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < nu) {
        const long long e = (long long)s * kN16 + n0 + 289 * u;
        const float2 v = A.xp[e];
        A.x64[e] = (double)v.x + (double)v.y;
      }
  }
  o.rz = df_to_double(rz);
  if (tid == 0) store_scalars(A.sc + s, o);
}

}  // namespace

bool small_supported(int N) { return N == 8 || N == 16; }

cudaError_t small_mixed(SolverBufs& B, const float* a32, const __nv_bfloat16* abf, const double* b, long long bstride,
                        double* x_out, double* r64, const PcgParams& prm, int inner_iters, int inner_next,
                        int fixed_steps, const float2* b_pair, bool pair_out, cudaStream_t st) {
  const int N = B.N, S = B.S;
  if (N == 8 && (b_pair || pair_out)) return cudaErrorInvalidValue;
  SmallArgs A{};
  A.a32 = a32; A.abf = abf; A.b = b; A.bp = b_pair; A.bstride = bstride;
  A.x64 = pair_out ? nullptr : x_out;
  A.xp = pair_out ? (float2*)x_out : (float2*)r64;
  A.sc = B.sc;
  A.tol2 = prm.rtol * prm.rtol;
  A.omega = (float)prm.omega;
  A.fixed = fixed_steps > 0 ? fixed_steps : 0;
  A.cap = fixed_steps > 0 ? fixed_steps : prm.max_iter;
  A.inner = inner_iters;
  A.inner_next = inner_next > 0 ? inner_next : inner_iters;
  const double nodes = (double)nodes_of(N), cells = (double)cells_of(N);
  const double bytes = (bstride ? S : 1) * nodes * 8 + S * (nodes * 8 + cells * 6);
  if (N == 8) {
    launch("small_f32", bytes, k_small8, dim3((unsigned)S), dim3(kT8), 0, st, A);
  } else {
    static SmemOptIn opt_in;
    const cudaError_t e = opt_in(k_small16, sizeof(Smem16));
    if (e != cudaSuccess) return e;
    launch("small_f32", bytes, k_small16, dim3((unsigned)S), dim3(kT16), sizeof(Smem16), st, A);
  }
  return cudaGetLastError();
}

}  // namespace mlsgd
