// tile64.cu - fused FP64 passes of the solver on 32^3 grids and up: APPLY, PRE, POST
// (rows a4, a6; what each computes: see below).
//
// FP64 issues at 2 operations per clock and SM on this part, 64 times slower than FP32, so
// a pass is bound by its FP64 operations and by nothing else: a warp's instruction holds
// the pipe for 16 clocks, in which the SM issues 64 others.  The operator is therefore
// summed by cells, with everything two nodes can share formed once and passed through
// shared memory.  The corners of a cell split by parity into two tetrahedra; the face
// diagonals of a cell join corners of one parity, the body diagonals opposite corners, so
// for corner v, with T the sum of the four values of its parity and x_a the opposite corner,
//   cell's share of (A x)_v / (h/12) = a (5 x_v - T - x_a).
//   * per cell: T of both parities from the diagonals of its lower and upper face, the
//     upper ones carried to the cell above (4 additions), times a (2), and the sums over
//     the two cells of a column that meet at a node plane (2 additions): Wa for the nodes
//     that are corners (0,0) or (1,1) of the column, Wb for (1,0) and (0,1);
//   * per node: Y = four of those column sums (3 additions) and the eight a x_a (8 FMAs);
//   * with w = omega/D, D = (h/3) sum of the eight cells, the diagonal cancels:
//       PRE   x1 = w r:           t = r - A x1 = (1 - 5/4 omega) r + h/12 Y
//       POST  x2 = w r + P e_c:   z = x2 + w (r - A x2) = (1 - 5/4 omega) x2 + w (r + h/12 Y),
//             partial r.z
//       APPLY p <- z + beta p:    q = A p = h/12 (5 sum8 p - Y), partial p.q
// That is 23 (PRE), 27 (POST) and 28 (APPLY) operations per node against 46, 58 and 47 of
// a node-by-node sum of the 21 points.
//
// A block of 256 threads owns 32 x 16 interior nodes (two rows per thread) and marches
// along z over a chunk of planes, two barriers a plane: operand plane k + 1 is derived
// (34 x 18 nodes, a ring of four planes); the cell layer above plane k is summed (33 x 17
// cells); the nodes of plane k are finished.  The next plane's values are loaded into
// registers a plane ahead, which at this rate hides any latency.  Boundary nodes count as
// 0 whatever the vectors hold there, and only interior nodes are written.
// Partial sums are formed per (tile, segment of kSeg planes) whatever the chunk, so the
// iterates do not depend on the batch or the chunking.
// Measured: FP64 level 3 of an optimisation run (9 samples of 64^3 with 32^3 partners, 24
// iterations) 28.6 ms with the node-by-node passes, 20.2 ms when they were replaced (18.6 with
// what followed elsewhere); state and adjoint of one 128^3 sample at rtol 1e-10 15.2 ms.
#include "internal.cuh"
#include "kernels.h"
#include "launch.h"

namespace mlsgd {

namespace {

enum Mode { M_APPLY = 0, M_PRE = 1, M_POST = 2 };
constexpr int kSeg = 4;                                // planes per partial-sum segment
constexpr int kW = 32, kH = 16, kT = 256;              // tile, threads
constexpr int kPX = kW + 2, kPY = kH + 2, kP = kPX * kPY;  // operand plane with halo
constexpr int kCX = kW + 1, kCY = kH + 1, kC = kCX * kCY;  // cells of a layer
constexpr int kEX = kW / 2 + 1, kEY = kH / 2 + 1, kE = kEX * kEY;  // POST: coarse cells under the operand plane
static_assert(kP > 2 * kT && kP <= 3 * kT && kC > 2 * kT && kC <= 3 * kT && kE <= kT, "three rounds of items");

template <int MODE>
struct Smem {
  double op[4][kP];     // operand planes, plane m in m & 3
  double cell[3][kC];   // cell layers, layer L in L % 3
  double wa[kC], wb[kC];
  double cz[MODE == M_APPLY ? kC : 1];  // sums of the two cells of a column
  double eps[MODE == M_POST ? 2 : 1][MODE == M_POST ? kP : 1];  // coarse planes summed in x and y (unscaled)
  double red[kT];
};

struct Args {
  const double *in0, *in1;  // APPLY: z, p (old)   PRE, POST: r, omega D^-1
  const double* ec;         // POST: coarse correction
  const double* a;          // cells
  double *out0, *out1;      // APPLY: q, p (new)   PRE: t   POST: z
  double* partial;
  const SolveScalars* sc;
  const int* act;
  double om;                // 1 - 5/4 omega
  int N, nzc, zc, nseg, first;
};

// OCC: blocks per SM the registers allow.  Three (80 registers, a few spilled) where the
// launch has more than two blocks per SM, else two without spills.
template <int MODE, int OCC>
__global__ void __launch_bounds__(kT, OCC) k_tile64(Args A) {
  // launched after the kernel before has ended and without letting the next one's blocks in:
  // placed early, blocks share SMs unevenly (FP64 level 3 of a run: 22.7 ms, 20.7 without); the
  // wait holds whatever the launch
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  Smem<MODE>& M = *reinterpret_cast<Smem<MODE>*>(smraw);
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const int N = A.N, n1 = N + 1;
  const int chunk = blockIdx.z % A.nzc;
  const int s = A.act != nullptr ? A.act[blockIdx.z / A.nzc] : (int)(blockIdx.z / A.nzc);
  if (A.sc != nullptr && !A.sc[s].active) return;
  const int x0 = 1 + kW * blockIdx.x, y0 = 1 + kH * blockIdx.y;
  const int kbeg = 1 + chunk * A.zc, kend = min(N - 1, kbeg + A.zc - 1);
  const unsigned pn = (unsigned)(n1 * n1), pc = (unsigned)(N * N);
  const long long nodes = (long long)pn * n1;
  const double scale = 1.0 / (12.0 * N);
  const bool rd1 = MODE != M_APPLY || !A.first;  // the first APPLY reads no old p
  const double beta = (MODE == M_APPLY && !A.first) ? A.sc[s].beta : 0.0;
  const double* v0 = A.in0 + s * nodes;
  const double* v1 = A.in1 + s * nodes;
  const double* cells = A.a + s * (long long)pc * N;

  // ---- items: operand entries tid + 256 j and cells; the partial third rounds go to the
  // first and to the last threads
  auto ent = [&](int j) { return tid + kT * j; };
  auto cel = [&](int j) { return j < 2 ? tid + kT * j : 3 * kT - 1 - tid; };
  const bool ent2 = ent(2) < kP, cel2 = cel(2) < kC;
  unsigned eoff[3], coff[3];  // node and cell offsets in a plane
  unsigned fl = 0;            // bit j: entry is interior; bits 4 + j: cell exists; bits 8 + 2j..: odd column + odd row
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int e = ent(j), c = e % kPX, r = e / kPX, gi = x0 - 1 + c, gj = y0 - 1 + r;
    if (e < kP && gi > 0 && gj > 0 && gi < N && gj < N) fl |= 1u << j;
    fl |= (unsigned)((c & 1) + (r & 1)) << (8 + 2 * j);
    eoff[j] = ((fl >> j) & 1u) ? (unsigned)(gi + n1 * gj) : 0u;
    const int q = cel(j), ci = x0 - 1 + q % kCX, cj = y0 - 1 + q / kCX;
    if (q < kC && ci < N && cj < N) fl |= 16u << j;
    coff[j] = ((fl >> (4 + j)) & 1u) ? (unsigned)(ci + N * cj) : 0u;
  }
  double va[3], vb[3], cc[3];
  auto load_nodes = [&](int m) {  // plane m of the node vectors (0 off the interior)
    const bool mint = m > 0 && m < N;
    const unsigned b = mint ? pn * (unsigned)m : 0u;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const bool ok = mint && ((fl >> j) & 1u);
      va[j] = ok ? v0[b + eoff[j]] : 0.0;
      vb[j] = (ok && rd1) ? v1[b + eoff[j]] : 0.0;
    }
  };
  auto load_cells = [&](int L) {
#pragma unroll
    for (int j = 0; j < 3; ++j) cc[j] = (L < N && ((fl >> (4 + j)) & 1u)) ? cells[pc * (unsigned)L + coff[j]] : 0.0;
  };
  // POST: coarse plane c summed in x and y at the staged nodes: item (a, b) writes the nodes
  // (2a + p, 2b + q) (the tile's origin is even); weights 1, 1/2, 1/4 (and 1/2 between two
  // coarse planes) are applied where the sums are used
  double ev[4] = {0.0, 0.0, 0.0, 0.0};
  const int it = kT - 1 - tid;  // the entries' third round goes to the first threads
  auto load_coarse = [&](int c) {
    if constexpr (MODE == M_POST) {
      const int nc = N / 2, nc1 = nc + 1, ca = ((x0 - 1) >> 1) + it % kEX, cb = ((y0 - 1) >> 1) + it / kEX;
      const double* e = A.ec + s * (long long)nc1 * nc1 * nc1 + (long long)c * nc1 * nc1;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = ca + (q & 1), j = cb + (q >> 1);
        ev[q] = (it < kE && c > 0 && c < nc && i > 0 && i < nc && j > 0 && j < nc) ? e[i + nc1 * j] : 0.0;
      }
    }
  };
  auto interp_xy = [&](int c) {
    if constexpr (MODE == M_POST) {
      if (it < kE) {
        double* o = M.eps[c & 1] + 2 * (it % kEX) + kPX * 2 * (it / kEX);
        const double r0 = ev[0] + ev[1];
        o[0] = ev[0];
        o[1] = r0;
        o[kPX] = ev[0] + ev[2];
        o[kPX + 1] = r0 + (ev[2] + ev[3]);
      }
    }
  };
  // operand plane m from the loaded values; POST: an even plane also sums the coarse plane
  // that the next one needs
  auto derive = [&](int m) {
    double* o = M.op[m & 3];
    const int c0 = m >> 1;
    if (MODE == M_POST && !(m & 1)) {
      interp_xy(c0 + 1);
      load_coarse(c0 + 2);
    }
    const bool mint = m > 0 && m < N;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (j == 2 && !ent2) continue;
      const int e = ent(j);
      double v;
      if constexpr (MODE == M_APPLY) {
        v = A.first ? va[j] : fma(beta, vb[j], va[j]);
      } else if constexpr (MODE == M_PRE) {
        v = va[j] * vb[j];
      } else {
        const int h = (int)((fl >> (8 + 2 * j)) & 3u) + (m & 1);  // weight 2^-h
        const double w = __hiloint2double(0x3FF00000 - (h << 20), 0);
        double ee = M.eps[c0 & 1][e];
        if (m & 1) ee += M.eps[(c0 + 1) & 1][e];
        v = fma(w, ee, va[j] * vb[j]);
        v = (mint && ((fl >> j) & 1u)) ? v : 0.0;
      }
      o[e] = v;
    }
  };

  // ---- this thread's nodes
  const int gi = x0 + tx, gj = y0 + 2 * ty;
  const bool ok0 = gi < N && gj < N, ok1 = gi < N && gj + 1 < N;
  const unsigned g0 = (unsigned)(gi + n1 * gj);
  double* out0 = A.out0 + s * nodes;
  double* out1 = MODE == M_APPLY ? A.out1 + s * nodes : nullptr;
  double red = 0.0;
  double dl1[3], dl2[3], ue[3], uo[3], cp[3];  // per cell item: diagonals of the lower face, U and a of the layer below
#pragma unroll
  for (int j = 0; j < 3; ++j) dl1[j] = dl2[j] = ue[j] = uo[j] = cp[j] = 0.0;

  if constexpr (MODE == M_POST) {  // kbeg - 1 is even
    load_coarse((kbeg - 1) >> 1);
    interp_xy((kbeg - 1) >> 1);
    load_coarse(((kbeg - 1) >> 1) + 1);
    __syncthreads();
  }
  load_nodes(kbeg - 1);
  derive(kbeg - 1);
  load_nodes(kbeg);
  load_cells(kbeg - 1);
  __syncthreads();  // (POST: the sums that plane kbeg reads)
  int c3 = (kbeg - 1) % 3;  // ring slot of layer L
#pragma unroll 1
  for (int L = kbeg - 1; L <= kend; ++L) {
    double cn[3];
    derive(L + 1);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cn[j] = cc[j];
      if (j < 2 || cel2) M.cell[c3][cel(j)] = cc[j];
    }
    if (L < kend) {
      load_nodes(L + 2);
      load_cells(L + 1);
    }
    const unsigned go = g0 + pn * (unsigned)L;
    double r[2] = {0.0, 0.0}, wd[2] = {0.0, 0.0};  // own raw values of plane L
    if (MODE != M_APPLY && L >= kbeg) {
      if (ok0) r[0] = v0[go];
      if (ok1) r[1] = v0[go + n1];
      if (MODE == M_POST) {
        if (ok0) wd[0] = v1[go];
        if (ok1) wd[1] = v1[go + n1];
      }
    }
    __syncthreads();
    // cell layer L (between node planes L and L + 1)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (j == 2 && !cel2) continue;
      const int q = cel(j), b = q + q / kCX;  // operand entry of the cell's corner (0, 0)
      if (L == kbeg - 1) {
        const double* x = M.op[L & 3] + b;
        dl1[j] = x[0] + x[kPX + 1];
        dl2[j] = x[1] + x[kPX];
      }
      const double* x = M.op[(L + 1) & 3] + b;
      const double u1 = x[0] + x[kPX + 1], u2 = x[1] + x[kPX];
      const double e = cn[j] * (dl1[j] + u2), o = cn[j] * (dl2[j] + u1);
      if (L >= kbeg) {
        M.wa[q] = e + uo[j];
        M.wb[q] = o + ue[j];
        if (MODE == M_APPLY) M.cz[q] = cn[j] + cp[j];
      }
      ue[j] = e;
      uo[j] = o;
      dl1[j] = u1;
      dl2[j] = u2;
      if (MODE == M_APPLY) cp[j] = cn[j];
    }
    __syncthreads();
    if (L >= kbeg) {
      const int cl = c3 == 0 ? 2 : c3 - 1;  // slot of the layer below
      const int nb = tx + kPX * 2 * ty, cb = tx + kCX * 2 * ty;  // corner of the 3 x 4 window, of the 2 x 3 cells
      double y[2], s8[2] = {0.0, 0.0};
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const double* wa = M.wa + cb + kCX * t;
        const double* wb = M.wb + cb + kCX * t;
        y[t] = (wa[0] + wa[kCX + 1]) + (wb[1] + wb[kCX]);
      }
      if constexpr (MODE == M_APPLY) {
        double rs[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) rs[q] = M.cz[cb + kCX * q] + M.cz[cb + kCX * q + 1];
        s8[0] = rs[0] + rs[1];
        s8[1] = rs[1] + rs[2];
      }
#pragma unroll
      for (int l = 0; l < 2; ++l) {  // cells below with operand plane L - 1, above with L + 1
        const double* x = M.op[(L - 1 + 2 * l) & 3] + nb;
        const double* c = M.cell[l ? c3 : cl] + cb;
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
          for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int t = 0; t < 2; ++t) y[t] = fma(c[p + kCX * (t + q)], x[2 * p + kPX * (t + 2 * q)], y[t]);
      }
      const double* xc = M.op[L & 3] + nb + kPX + 1;
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const bool ok = t ? ok1 : ok0;
        const unsigned o = go + n1 * t;
        if constexpr (MODE == M_APPLY) {
          const double p = xc[kPX * t], q = scale * fma(5.0, s8[t] * p, -y[t]);
          if (ok) {
            out0[o] = q;
            out1[o] = p;
          }
          red = fma(ok ? p : 0.0, q, red);
        } else if constexpr (MODE == M_PRE) {
          const double v = fma(A.om, r[t], scale * y[t]);
          if (ok) out0[o] = v;
        } else {
          const double z = fma(wd[t], fma(scale, y[t], r[t]), A.om * xc[kPX * t]);
          if (ok) out0[o] = z;
          red = fma(r[t], z, red);  // r = 0 where the node is not the thread's
        }
      }
      if (MODE != M_PRE && (L == kend || (L - 1) % kSeg == kSeg - 1)) {  // block-uniform
        M.red[tid] = red;
        __syncthreads();
        if (tid < 32) {  // one warp's additions instead of five in each
          double v = M.red[tid];
#pragma unroll
          for (int w = 1; w < kT / 32; ++w) v += M.red[tid + 32 * w];
          v = warp_sum(v);
          if (tid == 0)
            A.partial[(long long)s * (gridDim.x * gridDim.y * A.nseg) +
                      (((L - 1) / kSeg) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = v;
        }
        red = 0.0;
      }
    }
    c3 = c3 == 2 ? 0 : c3 + 1;
  }
}

int tiles_x(int N) { return (N - 1 + kW - 1) / kW; }
int tiles_y(int N) { return (N - 1 + kH - 1) / kH; }
int segments(int N) { return (N - 1 + kSeg - 1) / kSeg; }

template <int MODE, int OCC>
void run_occ(const char* cls, double bytes, const Args& A, dim3 grid, cudaStream_t st) {
  constexpr size_t smem = sizeof(Smem<MODE>);
  static_assert(smem + 1024 <= 228 * 1024 / 3, "three blocks per SM");
  static SmemOptIn opt_in;
  (void)opt_in(k_tile64<MODE, OCC>, smem);  // a launch without it is refused
  launch_after(cls, bytes, k_tile64<MODE, OCC>, grid, dim3(kT), smem, st, A);
}
template <int MODE>
void run(const char* cls, double bytes, Args A, const Batch& bt, cudaStream_t st) {
  const int bx = tiles_x(A.N), by = tiles_y(A.N), nseg = segments(A.N);
  // Planes per chunk: an SM's blocks share its FP64 pipe, so the time is the work of the
  // fullest SM; a chunk costs about 0.6 planes more than it has (the cell layer and the
  // operand planes before its first), and one block alone leaves the pipe idle a quarter of
  // the time (9 samples of 64^3: 20.6 ms a solve pair with one block per SM, 17.7 with two).
  auto per_sm = [&](int q) { return ((long long)bx * by * bt.n * ((nseg + q - 1) / q) + 151) / 152; };
  int spc = nseg;
  double best = 1e300;
  for (int q = 1; q <= nseg; ++q) {
    const double cost = (per_sm(q) == 1 ? 1.35 : (double)per_sm(q)) * (kSeg * q + 0.6);
    if (cost < best) { best = cost; spc = q; }
  }
  if (bt.zchunks > 0) spc = bt.zchunks < nseg ? (nseg + bt.zchunks - 1) / bt.zchunks : 1;
  A.nseg = nseg;
  A.nzc = (nseg + spc - 1) / spc;
  A.zc = spc * kSeg;
  A.act = bt.act;
  const dim3 grid(bx, by, (unsigned)(bt.n * A.nzc));
  // three blocks per SM against two, a solve pair: 3 samples of 64^3 7.1 against 8.5 ms, 16 25.9
  // against 26.7, one of 128^3 15.2 against 16.0; with at most two there the spills cost:
  // 9 of 64^3 14.5 against 14.3, 9 of 32^3 3.60 against 3.52
  if (per_sm(spc) > 2) run_occ<MODE, 3>(cls, bytes, A, grid, st);
  else run_occ<MODE, 2>(cls, bytes, A, grid, st);
}

double vbytes(int N, int n, double vec, double coef) {
  return (double)n * 8 * (vec * (double)nodes_of(N) + coef * (double)cells_of(N));
}

}  // namespace

int tile64_blocks_per_sample(int N) { return tiles_x(N) * tiles_y(N) * segments(N); }

void tile64_apply(const double* z, const double* pold, double* pnew, const double* a, double* q, double* partial,
                  const SolveScalars* sc, int N, const Batch& bt, bool first, cudaStream_t st) {
  Args A{};
  A.in0 = z; A.in1 = pold; A.a = a; A.out0 = q; A.out1 = pnew; A.partial = partial; A.sc = sc; A.N = N;
  A.first = first ? 1 : 0;
  run<M_APPLY>("apply_f64", vbytes(N, bt.n, first ? 3 : 4, 1), A, bt, st);
}
void tile64_pre(const double* r, const double* a, const double* wdinv, double* t, const SolveScalars* sc, int N,
                const Batch& bt, double omega, cudaStream_t st) {
  Args A{};
  A.in0 = r; A.in1 = wdinv; A.a = a; A.out0 = t; A.sc = sc; A.N = N; A.om = 1.0 - 1.25 * omega;
  run<M_PRE>("pre_f64", vbytes(N, bt.n, 3, 1), A, bt, st);
}
void tile64_post(const double* r, const double* a, const double* wdinv, const double* ec, double* z, double* partial,
                 const SolveScalars* sc, int N, const Batch& bt, double omega, cudaStream_t st) {
  Args A{};
  A.in0 = r; A.in1 = wdinv; A.ec = ec; A.a = a; A.out0 = z; A.partial = partial; A.sc = sc; A.N = N;
  A.om = 1.0 - 1.25 * omega;
  run<M_POST>("post_f64", vbytes(N, bt.n, 3, 1) + (double)bt.n * 8 * nodes_of(N / 2), A, bt, st);
}

}  // namespace mlsgd
