// tile32.cu - fused FP32 passes of the mixed solver on grids the whole-row slab passes do
// not cover (128^3 and up; any grid with the tile passes selected): APPLY, APPLYX, PRE,
// PREU, POST (rows a4, a6; see tiled.cu for what each computes).
//
// A block of 256 threads owns a tile of 32 x 32 interior nodes (x0 = 1 + 32 bx,
// y0 = 1 + 32 by; lane = column, warp ty = rows 4 ty .. 4 ty + 3) and marches along z over
// a chunk of planes.  What bounds a pass is instruction issue, so the work per node is
// kept small:
//   * node plane m of a staged vector (34 rows with the halo) is copied in 16-byte pieces
//     (cp.async) two planes ahead into a ring of three slots; a row is widened to 16-byte
//     boundaries: node (x0 - 1 + c, y0 - 1 + r) sits at 40 r + delta_r + c with
//     delta_r = (s + m + y0 - 1 + r) mod 4, since N + 1, its square and its cube are 1 mod 4;
//     an mbarrier per slot counts the copies in;
//   * a thread derives the operand at its own four nodes and one of the 132 halo nodes
//     (boundary nodes are 0 by position, whatever the vectors hold there), and keeps the
//     own raw values in registers for the plane's epilogue;
//   * the operator is summed per operand plane: the 3 x 6 window of plane k + 1, read
//     once, gives the upper part of node plane k, the centre of plane k + 1 and the lower
//     part of plane k + 2, which are carried in registers, with the upper cell plane.
// So a plane takes one block barrier, 4.5 window loads per node instead of 13.5 and about
// a third of the instructions of a pass that loads three windows per plane and stages
// 4-byte elements.  The parts (centre, lower, upper) are summed in the order of that pass,
// and the partial sums of the dot products per (tile, segment of kSegPlanes planes) too.
// One 256^3 sample: POST 143 us with three windows a plane, 121 us now; APPLYX 147 -> 120;
// PREU 136 -> 98; one 128^3: POST 30 -> 25, PRE 22 -> 18.
//
// The z chunk is chosen so that the blocks make few, full waves of three blocks per SM.
// Every wait on an mbarrier is bounded (about a second of SM clock); one that runs out
// sets *err, and the thread skips its remaining waits but still reaches every block
// barrier, so the kernel ends and the host reads the flag.
#include <cstdio>

#include "internal.cuh"
#include "kernels.h"
#include "launch.h"

namespace mlsgd {

namespace {

enum Mode { T_APPLY = 0, T_PRE = 1, T_POST = 2, T_PREU = 4, T_APPLYX = 5 };
constexpr int kSegPlanes = 8;  // partial-sum segment (the same as tiled.cu's kZSeg)
constexpr int kSlots = 3, kAhead = 2;
constexpr int kRows = 34, kPitch = 40;          // staged node rows, floats per row
constexpr int kRaw = kRows * kPitch;             // floats per slot
constexpr int kOpPitch = 36, kOp = kRows * kOpPitch;
constexpr int kCellRows = 33;
constexpr int kCRows = 18, kCPitch = 24, kCRaw = kCRows * kCPitch;  // staged coarse plane
constexpr int kHalo = 2 * 34 + 2 * 32;

template <typename TA> constexpr int kCellPitch = sizeof(TA) == 2 ? 40 : 36;
template <typename TA> constexpr int kCellChunks = sizeof(TA) == 2 ? 5 : 9;  // 16-byte pieces of a cell row

template <typename TA, int MODE>
struct Smem {
  static constexpr int NV = MODE == T_PREU ? 3 : 2;  // APPLY: z, p_old; PRE, POST: r, dinv; PREU: r, q, dinv
  static constexpr bool kPost = MODE == T_POST;
  float raw[NV][kSlots][kRaw];
  float op[2][kOp];
  TA cells[kSlots][kCellRows * kCellPitch<TA>];
  float craw[kPost ? kSlots : 1][kPost ? kCRaw : 4];
  float eps[kPost ? 2 : 1][kPost ? kOp : 4];
  float4 ownr[MODE == T_APPLY ? 1 : 256];  // the epilogue's raw values of a thread's nodes: p_old or r
  float4 owndv[kPost ? 256 : 1];           // and omega D^-1
  unsigned long long bar[kSlots];
};

struct Args {
  const float* in0;   // APPLY: z   PRE, POST, PREU: r
  const float* in1;   // APPLY: p (old)   PREU: q
  const float* dinv;  // omega D^-1
  const float* ec;    // POST: coarse correction
  const void* a;      // cells
  float* out0;        // APPLY: q   PRE, PREU: t   POST: z
  float* out1;        // APPLY: p (new)   PREU: r (new)
  float* x;           // APPLYX: x += alpha_prev p_old
  double* partial;
  const SolveScalars* sc;
  const int* act;
  int* err;
  int N, nzc, zc, nseg, first, xfirst;
};

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(su32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {  // bounded
  if (bar_try(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (bar_try(bar, parity)) return true;
    if (clock64() - t0 > (2LL << 30)) return false;
  }
}
__device__ __forceinline__ float cell_f(float c) { return c; }
__device__ __forceinline__ float cell_f(__nv_bfloat16 c) { return __bfloat162float(c); }

template <typename TA, int MODE>
__global__ void __launch_bounds__(256, 3) k_tile32(Args A) {
  pdl_entry();
  using SM = Smem<TA, MODE>;
  constexpr bool kX = MODE == T_APPLYX, kApply = MODE == T_APPLY || kX, kPost = MODE == T_POST;
  constexpr bool kPre = MODE == T_PRE || MODE == T_PREU;
  constexpr int NV = SM::NV, CPI = kCellPitch<TA>, CCH = kCellChunks<TA>;
  extern __shared__ __align__(16) unsigned char smraw[];
  SM& M = *reinterpret_cast<SM*>(smraw);
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const int N = A.N, n1 = N + 1;
  const int chunk = blockIdx.z % A.nzc;
  const int s = A.act != nullptr ? A.act[blockIdx.z / A.nzc] : (int)(blockIdx.z / A.nzc);
  if (A.sc != nullptr && !A.sc[s].active) return;
  if (*(volatile int*)A.err != 0) return;  // an earlier wait ran out: the results are void anyway
  const int x0 = 1 + 32 * blockIdx.x, y0 = 1 + 32 * blockIdx.y;
  const int kbeg = 1 + chunk * A.zc, kend = min(N - 1, kbeg + A.zc - 1), first = kbeg - 1;
  const long long pn = (long long)n1 * n1, nodes = pn * n1, pc = (long long)N * N;
  const float scale = float(1.0 / (12.0 * N));
  float beta = 0.f, alpha = 0.f;
  if (kApply && !A.first) beta = (float)A.sc[s].beta;
  if (kX || MODE == T_PREU) alpha = (float)A.sc[s].alpha;
  const int nv = (kApply && A.first) ? 1 : NV;  // the first APPLY reads no old p
  const float* vin[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) vin[v] = v == 0 ? A.in0 : (v == 1 && (kApply || MODE == T_PREU) ? A.in1 : A.dinv);
  const TA* cells = (const TA*)A.a + s * pc * N;

  // ---- staging.  Offsets are 32-bit, from the sample's base rounded down to 16 bytes, and
  // advance by a plane per issue; a thread copies pieces e = tid and 511 - tid of the
  // 34 x 10 pieces of a node plane (row e / 10), and pieces tid, tid + 256 of the cell plane;
  // rows are whole numbers of pieces, so piece e goes to position e
  static_assert(kPitch == 4 * 10 && kCPitch == 4 * 6 && CPI == CCH * (16 / (int)sizeof(TA)), "whole pieces per row");
  const long long sbase = (long long)s * nodes;
  const unsigned sadj = (unsigned)(sbase & 3);
#pragma unroll
  for (int v = 0; v < NV; ++v) vin[v] += sbase & ~3LL;
  unsigned noff[2], coff[2];  // of plane `next`
  bool nok[2], cok[2];
  constexpr int kCellPieces = kCellRows * CCH, kPer = 16 / sizeof(TA);
  constexpr int kCellRounds = (kCellPieces + 255) / 256;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int e = j == 0 ? tid : 511 - tid, r = e / 10, p = 4 * (e - 10 * r);
    nok[j] = e < kRows * 10 && y0 - 1 + r <= N;  // rows outside the grid are skipped
    noff[j] = sadj + (unsigned)(first * n1 + y0 - 1 + r) * (unsigned)n1 + (unsigned)(x0 - 1 + p);
    const int ce = tid + 256 * j, cr = ce / CCH, cc = kPer * (ce - CCH * cr);
    cok[j] = ce < kCellPieces && y0 - 1 + cr < N && x0 - 1 + cc < N;
    coff[j] = (unsigned)(first * N + y0 - 1 + cr) * (unsigned)N + (unsigned)(x0 - 1 + cc);
  }
  // POST: the coarse planes' pieces (18 rows of 6) by the last threads, from the sample's
  // coarse base rounded down
  const unsigned pe = (unsigned)(N / 2 + 1) * (unsigned)(N / 2 + 1);
  const long long ebase = (long long)s * pe * (N / 2 + 1);
  const float* ec = kPost ? A.ec + (ebase & ~3LL) : nullptr;
  int cslot = (first >> 1) % kSlots;
  unsigned eoff = 0;
  bool eok = false;
  if constexpr (kPost) {
    const int e = 255 - tid, r = e / 6, p = 4 * (e - 6 * r), cy0 = (y0 - 1) >> 1;
    eok = e < kCRows * 6 && cy0 + r <= N / 2;
    eoff = (unsigned)(ebase & 3) + (unsigned)((first >> 1) * (N / 2 + 1) + cy0 + r) * (unsigned)(N / 2 + 1) +
           (unsigned)(((x0 - 1) >> 1) + p);
  }
  const uint32_t bar0 = su32(M.bar);
  // plane m (the planes are issued in order) into ring slot `slot`
  auto issue = [&](int m, int slot) {
    if (m > 0 && m < N) {  // the planes 0 and N are 0
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (!nok[j]) continue;
        const unsigned src = noff[j] & ~3u;
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (v < nv) copy16(M.raw[v][slot] + 4 * (j == 0 ? tid : 511 - tid), vin[v] + src);
      }
    }
    if (m < N) {  // cell rows y0 - 1 .. y0 + 31, 16-byte aligned
#pragma unroll
      for (int j = 0; j < kCellRounds; ++j)
        if (cok[j]) copy16(M.cells[slot] + kPer * (tid + 256 * j), cells + coff[j]);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      noff[j] += (unsigned)pn;
      coff[j] += (unsigned)pc;
    }
    if constexpr (kPost) {  // coarse plane m / 2 + 1 with every even fine plane, m / 2 with the first
      auto coarse = [&](int cp) {
        if (eok && cp > 0 && cp < N / 2) copy16(M.craw[0] + cslot * kCRaw + 4 * (255 - tid), ec + (eoff & ~3u));  // boundary planes are 0
        eoff += pe;
        cslot = cslot == kSlots - 1 ? 0 : cslot + 1;
      };
      if (m == first) coarse(m >> 1);
      if (!(m & 1)) coarse((m >> 1) + 1);  // first is even
    }
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(bar0 + 8 * slot) : "memory");
  };
  bool dead = false;
  auto wait_slot = [&](int slot, int parity) {
    if (!dead && !bar_wait(bar0 + 8 * slot, (uint32_t)parity)) {
      dead = true;
      atomicOr(A.err, 1);
    }
  };

  // ---- this thread's nodes and its halo node
  const int gi = x0 + tx, gj0 = y0 + 4 * ty;
  unsigned okb = 0;  // bit t: node (gi, gj0 + t) is interior in (x, y)
#pragma unroll
  for (int t = 0; t < 4; ++t)
    if (gi < N && gj0 + t < N) okb |= 1u << t;
  int hr = 0, hc = 0;  // staged row and column of the halo node
  {
    const int h = tid;
    if (h < 34) { hr = 0; hc = h; }
    else if (h < 68) { hr = 33; hc = h - 34; }
    else if (h < 100) { hr = h - 68 + 1; hc = 0; }
    else { hr = h - 100 + 1; hc = 33; }
  }
  const bool halo = tid < kHalo;
  const int hraw = hr * kPitch + hc, hop = hr * kOpPitch + hc;
  const bool hok = halo && x0 - 1 + hc > 0 && x0 - 1 + hc < N && y0 - 1 + hr > 0 && y0 - 1 + hr < N;

  // POST: coarse plane c interpolated in x and y at the staged nodes: item (a, b) of 17 x 17
  // (those past 256 go to the last threads) writes nodes (2a + p, 2b + q); boundary
  // values are 0 by position (bits of imask), whatever is staged there
  int iraw[2], irow[2];
  unsigned imask = 0;
  int islot = (first >> 1) % kSlots;  // slot of the coarse plane interpolated next
  if constexpr (kPost) {
    const int nc1 = N / 2 + 1, cy0 = (y0 - 1) >> 1, ex0 = (x0 - 1) >> 1;
#pragma unroll
    for (int rd = 0; rd < 2; ++rd) {
      const int it = rd == 0 ? tid : 511 - tid, b = it / 17, a = it - 17 * b;
      irow[rd] = b;
      iraw[rd] = b * kCPitch + a;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int ca = ex0 + a + (e & 1), cb = cy0 + b + (e >> 1);
        if (ca > 0 && ca < nc1 - 1 && cb > 0 && cb < nc1 - 1) imask |= 1u << (4 * rd + e);
      }
    }
  }
  auto interp_xy = [&](int c) {
    if constexpr (kPost) {
      const float* cp = M.craw[0] + islot * kCRaw;
      islot = islot == kSlots - 1 ? 0 : islot + 1;
      const unsigned mk = (c <= 0 || c >= N / 2) ? 0u : imask;
      const int d0 = s + c + ((y0 - 1) >> 1);  // offset of coarse row r: (d0 + r) & 3
      float* ed = M.eps[0] + (c & 1) * kOp;
#pragma unroll
      for (int rd = 0; rd < 2; ++rd) {
        if (rd == 1 && tid < 511 - 17 * 17 + 1) continue;
        const float* q0 = cp + iraw[rd] + ((d0 + irow[rd]) & 3);
        const float* q1 = cp + iraw[rd] + kCPitch + ((d0 + irow[rd] + 1) & 3);
        const unsigned mm = mk >> (4 * rd);
        const float e00 = (mm & 1u) ? q0[0] : 0.f, e10 = (mm & 2u) ? q0[1] : 0.f;
        const float e01 = (mm & 4u) ? q1[0] : 0.f, e11 = (mm & 8u) ? q1[1] : 0.f;
        const float r0 = (e00 + e10) * 0.5f, r1 = (e01 + e11) * 0.5f;
        float* o = ed + 2 * iraw[rd] + (2 * kOpPitch - 2 * kCPitch) * irow[rd];  // node (2a, 2b)
        o[0] = e00;
        o[1] = r0;
        o[kOpPitch] = (e00 + e01) * 0.5f;
        o[kOpPitch + 1] = (r0 + r1) * 0.5f;
      }
    }
  };

  // operand plane m (raw in ring slot `slot`) into operand slot m & 1; the own raw values
  // go to ownr, owndv.  Branch-free: values are formed at every node and selected to 0 off
  // the interior (what the slots hold there does not matter).
  const int rown = (4 * ty + 1) * kPitch + tx + 1, oown = (4 * ty + 1) * kOpPitch + tx + 1;
  auto derive = [&](int m, int slot, bool interp_next) {
    float* xp = M.op[0] + (m & 1) * kOp;
    const bool mint = m > 0 && m < N;
    if (kPost && interp_next && !(m & 1)) interp_xy((m >> 1) + 1);
    const float* e0 = M.eps[0] + (kPost ? ((m >> 1) & 1) * kOp : 0);
    const float* e1 = M.eps[0] + (kPost ? (((m >> 1) + 1) & 1) * kOp : 0);
    const float* rp = M.raw[0][0] + slot * kRaw;
    const int dm = s + m + y0 - 1;
    const bool mixed_planes = kPost && (m & 1);
    auto value = [&](const float* o, int oi, float& r, float& dv) {  // o: raw node, oi: operand index
      const float v0 = o[0];
      if constexpr (kApply) {
        r = o[kSlots * kRaw];
        return A.first ? v0 : __fmaf_rn(beta, r, v0);
      } else {
        dv = o[(NV - 1) * kSlots * kRaw];
        r = MODE == T_PREU ? __fmaf_rn(-alpha, o[kSlots * kRaw], v0) : v0;
        float v = __fmul_rn(r, dv);
        if constexpr (kPost) v = __fadd_rn(v, mixed_planes ? (e0[oi] + e1[oi]) * 0.5f : e0[oi]);
        return v;
      }
    };
    float r[4], dv[4];
    const unsigned mask = mint ? okb : 0u;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      dv[t] = 0.f;
      const float v = value(rp + rown + t * kPitch + ((dm + 1 + t) & 3), oown + t * kOpPitch, r[t], dv[t]);
      xp[oown + t * kOpPitch] = ((mask >> t) & 1u) ? v : 0.f;  // row 4 ty + 1 + t = 1 + t mod 4
    }
    if constexpr (MODE != T_APPLY) M.ownr[tid] = make_float4(r[0], r[1], r[2], r[3]);
    if constexpr (kPost) M.owndv[tid] = make_float4(dv[0], dv[1], dv[2], dv[3]);
    if (halo) {
      float rr, dd;
      const float v = value(rp + hraw + ((dm + hr) & 3), hop, rr, dd);
      xp[hop] = (mint && hok) ? v : 0.f;
    }
  };

  // ---- prologue
  if (tid == 0) {
#pragma unroll
    for (int q = 0; q < kSlots; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 256;\n" ::"r"(bar0 + 8 * q) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  for (int m = first; m <= min(first + kAhead, kend + 1); ++m) issue(m, m - first);
  wait_slot(0, 0);
  if constexpr (kPost) {
    interp_xy(first >> 1);
    interp_xy((first >> 1) + 1);
    __syncthreads();
  }
  derive(first, 0, false);
  __syncthreads();  // operand plane `first` is complete

  using Win = float[3][6];
  using Cel = float[2][5];
  auto load_win = [&](int m, Win& W) {
    const float* xp = M.op[m & 1] + 4 * ty * kOpPitch + tx;
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) W[c][r] = xp[r * kOpPitch + c];
  };
  auto load_cells = [&](int slot, Cel& C) {  // cells (gi - 1 + p, gj0 - 1 + q)
    const TA* cp = M.cells[slot] + 4 * ty * CPI + tx;
#pragma unroll
    for (int r = 0; r < 5; ++r)
#pragma unroll
      for (int p = 0; p < 2; ++p) C[p][r] = cell_f(cp[r * CPI + p]);
  };
  // the part of a node plane from the operand plane below or above it, through cells C
  auto off_part = [&](const Win& W, const Cel& C, float (&o)[4]) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      float a2 = 0.f;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        a2 -= (C[u][t] + C[u][t + 1]) * W[2 * u][t + 1];
        a2 -= (C[0][t + u] + C[1][t + u]) * W[1][t + 2 * u];
      }
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int p = 0; p < 2; ++p) a2 -= C[p][t + q] * W[2 * p][t + 2 * q];
      o[t] = a2;
    }
  };
  auto centre_part = [&](const Win& W, const Cel& Cl, const Cel& Ch, float (&o)[4]) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      float pxy[2][2];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) pxy[v][u] = Cl[u][t + v] + Ch[u][t + v];
      const float sum8 = (pxy[0][0] + pxy[0][1]) + (pxy[1][0] + pxy[1][1]);
      float a1 = 4.f * sum8 * W[1][t + 1];
#pragma unroll
      for (int v = 0; v < 2; ++v)
#pragma unroll
        for (int u = 0; u < 2; ++u) a1 -= pxy[v][u] * W[2 * u][t + 2 * v];
      o[t] = a1;
    }
  };
  // entering iteration k: lower and centre part of plane k, lower part of plane k + 1, the
  // operand of plane k at the own nodes, cell plane k
  float lowA[4], cenA[4], lowB[4], ctr[4];
  Cel Cn;
  {
    Win W;
    Cel Cl;
    load_cells(0, Cl);
    load_win(first, W);
    off_part(W, Cl, lowA);
    wait_slot(1, 0);
    derive(kbeg, 1, true);
    __syncthreads();
    // every warp has derived plane `first` and read its cells: its slot is free
    if (first + kAhead + 1 <= kend + 1) issue(first + kAhead + 1, 0);
    load_cells(1, Cn);
    load_win(kbeg, W);
    centre_part(W, Cl, Cn, cenA);
    off_part(W, Cn, lowB);
#pragma unroll
    for (int t = 0; t < 4; ++t) ctr[t] = W[1][t + 1];
  }
  // the sample's outputs (uniform bases) and 32-bit node offsets
  float* out0 = A.out0 + sbase;
  float* out1 = (kApply || MODE == T_PREU) ? A.out1 + sbase : nullptr;
  float* xg = kX ? A.x + sbase : nullptr;
  float red = 0.f;
  int slot = 2, par = 0;  // ring slot and phase of plane k + 1
  unsigned gk = (unsigned)pn * kbeg + (unsigned)n1 * gj0 + gi;  // node (gi, gj0) of plane k
#pragma unroll 1
  for (int k = kbeg; k <= kend; ++k, gk += (unsigned)pn) {
    float xv[4];
    if constexpr (kX) {  // x of the own nodes, in flight while the plane is derived
#pragma unroll
      for (int t = 0; t < 4; ++t) xv[t] = (((okb >> t) & 1u) && !A.xfirst) ? xg[gk + n1 * t] : 0.f;
    }
    float4 rk = make_float4(0.f, 0.f, 0.f, 0.f), dk = rk;  // own raw values of plane k
    if constexpr (MODE != T_APPLY) rk = M.ownr[tid];
    if constexpr (kPost) dk = M.owndv[tid];
    const float rawA[4] = {rk.x, rk.y, rk.z, rk.w}, dvA[4] = {dk.x, dk.y, dk.z, dk.w};
    wait_slot(slot, par);
    derive(k + 1, slot, true);
    __syncthreads();
    // operand plane k + 1 is complete; the raw slot and the cells of plane k are no longer read
    const int prev = slot == 0 ? kSlots - 1 : slot - 1;  // the slot of plane k, free now
    if (k + kAhead + 1 <= kend + 1) issue(k + kAhead + 1, prev);
    Win W;
    load_win(k + 1, W);
    float up[4];
    off_part(W, Cn, up);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const bool ok = (okb >> t) & 1u;
      const float sum = cenA[t] + (lowA[t] + up[t]);
      const unsigned o = gk + n1 * t;
      if constexpr (kApply) {
        const float ax = scale * sum, pv = ctr[t];
        if (ok) out0[o] = ax;
        if (ok) out1[o] = pv;
        red = ok ? __fmaf_rn(pv, ax, red) : red;
        if (kX && ok) xg[o] = __fmaf_rn(alpha, rawA[t], xv[t]);
      } else if constexpr (kPre) {
        const float tv = __fmaf_rn(-scale, sum, rawA[t]);
        if (ok) out0[o] = tv;
        if (MODE == T_PREU && ok) out1[o] = rawA[t];
      } else {
        const float zv = __fmaf_rn(__fmaf_rn(-scale, sum, rawA[t]), dvA[t], ctr[t]);
        if (ok) out0[o] = zv;
        red = ok ? __fmaf_rn(rawA[t], zv, red) : red;
      }
    }
    if (k < kend) {
      Cel Ch;
      load_cells(slot, Ch);
      centre_part(W, Cn, Ch, cenA);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        lowA[t] = lowB[t];
        ctr[t] = W[1][t + 1];
      }
      off_part(W, Ch, lowB);
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int r = 0; r < 5; ++r) Cn[p][r] = Ch[p][r];
    }
    if (!kPre && (k == kend || (k - 1) % kSegPlanes == kSegPlanes - 1)) {  // block-uniform
      const float b = block_sum(red);
      if (tid == 0) {
        const int per = gridDim.x * gridDim.y * A.nseg;
        A.partial[(long long)s * per + (((k - 1) / kSegPlanes) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = (double)b;
      }
      red = 0.f;
    }
    if (++slot == kSlots) {
      slot = 0;
      par ^= 1;
    }
  }
  // every issued plane has been waited for
}

// planes per chunk (whole segments) so that the blocks' waves, of about three per SM,
// cost least; a chunk derives two planes more than it computes
int chunk_segments(long long tiles, int nseg) {
  int best = nseg;
  double cost = 1e300;
  for (int spc = 1; spc <= nseg; ++spc) {
    const long long blocks = tiles * ((nseg + spc - 1) / spc);
    const double c = (double)((blocks + 3 * 152 - 1) / (3 * 152)) * (kSegPlanes * spc + 3);
    if (c < cost) { cost = c; best = spc; }
  }
  return best;
}

template <typename TA, int MODE>
void run(const char* cls, double bytes, Args args, const Batch& bt, cudaStream_t st) {
  const TiledShape t = tiled_shape(args.N, bt.S, 4);
  int spc = chunk_segments((long long)t.bx * t.by * bt.n, t.nseg);
  if (bt.zchunks > 0) spc = bt.zchunks < t.nseg ? (t.nseg + bt.zchunks - 1) / bt.zchunks : 1;
  args.nzc = (t.nseg + spc - 1) / spc;
  args.zc = spc * kSegPlanes;
  args.nseg = t.nseg;
  args.act = bt.act;
  args.err = bt.err;
  constexpr size_t smem = sizeof(Smem<TA, MODE>);
  static_assert((sizeof(TA) == 4 && MODE == T_POST) || smem + 1024 <= 228 * 1024 / 3, "three blocks per SM");
  static SmemOptIn opt_in;
  (void)opt_in(k_tile32<TA, MODE>, smem, true);  // a launch without it is refused
  launch(cls, bytes, k_tile32<TA, MODE>, dim3(t.bx, t.by, (unsigned)(bt.n * args.nzc)), dim3(256), smem, st, args);
}

double vbytes(int N, int n, double vec, double coef, size_t ta) {
  return (double)n * (vec * (double)nodes_of(N) * 4 + coef * (double)cells_of(N) * ta);
}

}  // namespace

void tile32_apply(const float* z, const float* pold, float* pnew, const float* a, float* q, float* x, double* partial,
                  const SolveScalars* sc, int N, const Batch& bt, bool first, bool x_first, cudaStream_t st) {
  Args A{};
  A.in0 = z; A.in1 = pold; A.a = a; A.out0 = q; A.out1 = pnew; A.x = x; A.partial = partial; A.sc = sc; A.N = N;
  A.first = first ? 1 : 0;
  A.xfirst = x_first ? 1 : 0;
  if (x) run<float, T_APPLYX>("apply_f32", vbytes(N, bt.n, x_first ? 5 : 6, 1, 4), A, bt, st);
  else run<float, T_APPLY>("apply_f32", vbytes(N, bt.n, first ? 3 : 4, 1, 4), A, bt, st);
}
template <typename TA>
void tile32_pre(const float* r, const float* q, const TA* a, const float* dinv, float* t, float* rnew,
                const SolveScalars* sc, int N, const Batch& bt, cudaStream_t st) {
  Args A{};
  A.in0 = r; A.in1 = q; A.a = a; A.dinv = dinv; A.out0 = t; A.out1 = rnew; A.sc = sc; A.N = N;
  if constexpr (sizeof(TA) == 2) {  // the fine level
    if (q) {
      run<TA, T_PREU>("pre_f32", vbytes(N, bt.n, 5, 1, sizeof(TA)), A, bt, st);
      return;
    }
  }
  run<TA, T_PRE>("pre_f32", vbytes(N, bt.n, 3, 1, sizeof(TA)), A, bt, st);
}
template <typename TA>
void tile32_post(const float* r, const TA* a, const float* dinv, const float* ec, float* z, double* partial,
                 const SolveScalars* sc, int N, const Batch& bt, cudaStream_t st) {
  Args A{};
  A.in0 = r; A.a = a; A.dinv = dinv; A.ec = ec; A.out0 = z; A.partial = partial; A.sc = sc; A.N = N;
  run<TA, T_POST>("post_f32", vbytes(N, bt.n, 3, 1, sizeof(TA)) + (double)bt.n * nodes_of(N / 2) * 4, A, bt, st);
}
template void tile32_pre<float>(const float*, const float*, const float*, const float*, float*, float*,
                                const SolveScalars*, int, const Batch&, cudaStream_t);
template void tile32_pre<__nv_bfloat16>(const float*, const float*, const __nv_bfloat16*, const float*, float*, float*,
                                        const SolveScalars*, int, const Batch&, cudaStream_t);
template void tile32_post<float>(const float*, const float*, const float*, const float*, float*, double*,
                                 const SolveScalars*, int, const Batch&, cudaStream_t);
template void tile32_post<__nv_bfloat16>(const float*, const __nv_bfloat16*, const float*, const float*, float*, double*,
                                         const SolveScalars*, int, const Batch&, cudaStream_t);

}  // namespace mlsgd
