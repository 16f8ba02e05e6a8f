// refine.cuh - error-free FP32 arithmetic of the refinement residual on FP32 (hi, lo)
// pairs (the z-marching residual pass and the one-block solve).
#pragma once
#include "internal.cuh"

namespace mlsgd {

// two_sum: s + e == a + b exactly (Knuth); products use the FMA to split
// c * x into p + pe exactly.  A coefficient is an unevaluated pair (h, l).
struct F2 { float h, l; };
__device__ __forceinline__ F2 two_sum(float a, float b) {  // intrinsics: never contracted
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return F2{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
// (S, comp) += sgn * (c.h + c.l) * (x.x + x.y), sgn = +1 or -1
template <bool NEG>
__device__ __forceinline__ void df_term(float& S, float& comp, F2 c, float2 x) {
  const float p = __fmul_rn(c.h, x.x);
  const float pe = __fmaf_rn(c.h, x.x, -p);
  const float low = __fmaf_rn(c.h, x.y, __fmaf_rn(c.l, x.x, pe));
  const float q = NEG ? -p : p;
  const F2 t = two_sum(S, q);
  S = t.h;
  comp = __fadd_rn(comp, __fadd_rn(t.l, NEG ? -low : low));
}

// (S, comp) += sgn (c.h + c.l) x for an FP32 operand x: the product c.h x is split
// exactly by the FMA, c.l x enters the compensation
template <bool NEG>
__device__ __forceinline__ void res_term(float& S, float& comp, F2 c, float x) {
  const float p = __fmul_rn(c.h, x);
  const float low = __fmaf_rn(c.l, x, __fmaf_rn(c.h, x, -p));
  const F2 t = two_sum(S, NEG ? -p : p);
  S = t.h;
  comp = __fadd_rn(comp, __fadd_rn(t.l, NEG ? -low : low));
}
// the same for a single FP32 coefficient c (a cell of the body diagonals)
template <bool NEG>
__device__ __forceinline__ void res_term1(float& S, float& comp, float c, float x) {
  const float p = __fmul_rn(c, x);
  const float low = __fmaf_rn(c, x, -p);
  const F2 t = two_sum(S, NEG ? -p : p);
  S = t.h;
  comp = __fadd_rn(comp, __fadd_rn(t.l, NEG ? -low : low));
}

// (b - A x) at one interior node of an N^3 grid, rounded to FP32: exact pair sums of the
// cells C(r, p, q) (plane, x, y offset), exact products with the operand pairs
// X(plane, x, y), compensated sums, the scale h/12 and the subtraction from b in the same
// arithmetic.  No FP64 instruction.
template <typename FC, typename FX>
__device__ __forceinline__ float refine_residual(FC&& cell, FX&& X, float2 bv, int N) {
  float C[2][2][2];
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q) C[r][p][q] = cell(r, p, q);
  F2 pxy[2][2], pxz[2][2], pyz[2][2];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      pxy[v][u] = two_sum(C[0][u][v], C[1][u][v]);
      pxz[v][u] = two_sum(C[v][u][0], C[v][u][1]);
      pyz[v][u] = two_sum(C[v][0][u], C[v][1][u]);
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
  df_term<false>(S, comp, F2{4.f * S8, 4.f * E8}, X(1, 1, 1));
#pragma unroll
  for (int v = 0; v < 2; ++v)
#pragma unroll
    for (int u = 0; u < 2; ++u) df_term<true>(S, comp, pxy[v][u], X(1, 2 * u, 2 * v));
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int pl = 2 * r;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      df_term<true>(S, comp, pxz[r][u], X(pl, 2 * u, 1));
      df_term<true>(S, comp, pyz[r][u], X(pl, 1, 2 * u));
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) df_term<true>(S, comp, F2{C[r][p][q], 0.f}, X(pl, 2 * p, 2 * q));
  }
  const double scd = 1.0 / (12.0 * N);
  const float sch = (float)scd, scl = (float)(scd - (double)sch);  // h/12 as an FP32 pair
  const F2 axs = two_sum(S, comp);
  const float p = __fmul_rn(axs.h, sch);
  const float pe = __fmaf_rn(axs.h, scl, __fmaf_rn(axs.l, sch, __fmaf_rn(axs.h, sch, -p)));
  const F2 d = two_sum(bv.x, -p);
  return d.h + (d.l + (bv.y - pe));
}

// x (+)= inc for a pair x: two-sum of the head and inc, renormalised (about 48 bits)
__device__ __forceinline__ float2 pair_add(float2 xv, float inc) {
  const float sh = xv.x + inc;
  const float bb = sh - xv.x;
  const float se = (xv.x - (sh - bb)) + (inc - bb);
  const float lo = xv.y + se;
  const float h = sh + lo;
  return make_float2(h, lo - (h - sh));
}

}  // namespace mlsgd
