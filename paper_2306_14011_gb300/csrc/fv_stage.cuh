// Fused residual / SSP-RK3 stage kernel for 2D and 3D uniform Cartesian grids.
//
// One CTA owns a tile of cells.  It
//   1. stages the tile plus a 2-cell halo of every conserved variable into
//      shared memory: one TMA box (x, y[, z], var) completing on an mbarrier,
//      then plain loads for the halo cells that lie outside the domain
//      (periodic wrap or transmissive copy) -- TMA fills those with zeros;
//      without a tensor map (odd nx, tiny grids) every cell is a plain load;
//   2. per axis d, computes every face flux of the tile exactly once: MUSCL
//      face states of Eq. (6) (eps/2 * minmod slope) and the Roe flux; each
//      thread takes a run of consecutive faces along the normal, carrying the
//      stencil differences and the last flux from face to face;
//   3. in the same loop, accumulates per cell, in shared memory, sum_d coef_d
//      (F_{k+1/2} - F_{k-1/2}) -- the flux-difference form of Eq. (5) --
//      starting, in the RK modes, from the stage's base value (U^s,
//      3/4 U^n + 1/4 U^s or 1/3 U^n + 2/3 U^s), so the accumulator ends as the
//      SSP-RK3 stage of Eq. (4) discretised in time;
//   4. in the last axis's loop, writes the residual or the new stage state
//      (coalesced along x).
// Faces on a tile boundary are computed by both neighbouring CTAs (a
// 1/tile_x + 1/tile_y [+ 1/tile_z] overhead); inside a tile each face is
// evaluated once.
#pragma once
#include "../../include/fv.h"
#include "fv_device.cuh"
#include "fv_internal.h"

namespace fvk {

constexpr uint64_t kTmaWaitNs = 2000000000ull;  // 2 s bound on the tile-load wait

struct TileGeom {
  int BX, BY, BZ;   // tile box with halo
  int plane;        // doubles per variable in the box
  int RX, RY;       // row and plane stride of the cell accumulator (RX odd where it costs little: x-lines on all banks)
  int cells;        // accumulator length per variable
  int np;           // face runs of an axis pass, at most
};

// Run length of the face lines of one axis: nline lines of fn faces, so that
// the runs give each of `threads` threads one (or as few as np slots allow).
__host__ __device__ constexpr int run_length(int fn, int nline, int threads, int np) {
  int K = (fn * nline + threads - 1) / threads;
  while (K < fn && ((fn + K - 1) / K) * nline > np) ++K;
  return K;
}

__host__ __device__ constexpr TileGeom tile_geom(int dim, int tx, int ty, int tz, int threads) {
  TileGeom g{};
  g.BX = tx + 4;
  g.BY = ty + 4;
  g.BZ = (dim == 3) ? tz + 4 : 1;
  g.plane = g.BX * g.BY * g.BZ;
  g.RX = tx >= 8 ? tx + 1 : tx;
  g.RY = g.RX * ty;
  g.cells = g.RY * tz;
  // Two slots per run (its first and its latest flux): as many as 48 KB hold
  // beside the tile and the accumulator, and for larger tiles as many as a
  // buffer of the largest face count would take.
  const int cells = tx * ty * tz;
  int fmax = 0;
  for (int d = 0; d < dim; ++d) {
    const int t = d == 0 ? tx : (d == 1 ? ty : tz), f = cells / t * (t + 1);
    fmax = fmax > f ? fmax : f;
  }
  const int cap0 = (fmax + cells - g.cells) / 2, cap1 = (6144 / (dim + 2) - g.plane - g.cells) / 2;
  const int cap = cap0 > cap1 ? cap0 : cap1;
  g.np = 0;
  for (int d = 0; d < dim; ++d) {
    const int t = d == 0 ? tx : (d == 1 ? ty : tz), nline = cells / t;
    const int K = run_length(t + 1, nline, threads, cap);
    const int items = ((t + 1 + K - 1) / K) * nline;
    g.np = g.np > items ? g.np : items;
  }
  return g;
}

// The tile shape and thread count a kernel is compiled for, or (TX = 0) any,
// given at run time.  With a fixed shape every shared-memory offset of the face
// loops is a constant of its instruction.
template <int TX_, int TY_, int TZ_, int THREADS_>
struct Shape {
  static constexpr int TX = TX_, TY = TY_, TZ = TZ_, THREADS = THREADS_;
  static constexpr bool fixed = TX_ > 0;
};
using AnyShape = Shape<0, 0, 0, 0>;

template <int DIM, class SH>
__device__ __forceinline__ TileGeom shape_geom(const int tile[3]) {
  if constexpr (SH::fixed) {
    constexpr TileGeom g = tile_geom(DIM, SH::TX, SH::TY, SH::TZ, SH::THREADS);
    return g;
  } else {
    return tile_geom(DIM, tile[0], tile[1], DIM == 3 ? tile[2] : 1, (int)blockDim.x);
  }
}
template <class SH>
__device__ __forceinline__ int block_threads() {
  return SH::fixed ? SH::THREADS : (int)blockDim.x;
}

// Interior index that ghost coordinate c of an axis with n cells reads.
__device__ __forceinline__ int ghost_source(int c, int n, int bclo, int bchi) {
  if (c < 0) return bclo == 0 ? ((c % n) + n) % n : 0;
  if (c >= n) return bchi == 0 ? c % n : n - 1;
  return c;
}

// Load halo cells of the tile box (the 4 layers along each axis next to the
// valid tile, over the valid extent of the other axes).  only_outside: skip
// cells inside the domain (already staged by TMA).
template <int DIM>
__device__ __forceinline__ void load_halo(double *tile, const StageArgs &a, const int o[3], const int ext[3],
                                          const TileGeom &G, bool only_outside) {
  constexpr int NV = DIM + 2;
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    if (only_outside && o[d] >= 2 && o[d] + ext[d] + 2 <= a.n[d]) continue;
    const int a1 = (d == 0) ? 1 : 0, a2 = (d == 2) ? 1 : 2;  // the other two axes
    const int e1 = ext[a1], e2 = (DIM == 3) ? ext[a2] : 1;
    const int cnt = 4 * e1 * e2;
    for (int h = threadIdx.x; h < cnt; h += blockDim.x) {
      const int layer = h & 3;
      const int r = h >> 2;
      int l[3];
      l[d] = (layer < 2) ? layer : ext[d] + layer;
      l[a1] = r % e1 + 2;
      l[a2] = (DIM == 3) ? r / e1 + 2 : 0;
      int gc[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) gc[q] = o[q] - 2 + l[q];
      if (DIM == 2) gc[2] = 0;
      const bool outside = gc[d] < 0 || gc[d] >= a.n[d];
      if (only_outside && !outside) continue;
      gc[d] = ghost_source(gc[d], a.n[d], a.bc[d][0], a.bc[d][1]);
      const long long src = ((long long)gc[2] * a.n[1] + gc[1]) * a.n[0] + gc[0];
      const int dst = (l[2] * G.BY + l[1]) * G.BX + l[0];
#pragma unroll
      for (int v = 0; v < NV; ++v) tile[v * G.plane + dst] = a.Us[v * N + src];
    }
  }
}

// The limited slope of Eq. (6) between two differences of a stencil.  Both
// limiters are symmetric (Psi(r) = r Psi(1/r)), so the two kappa-weighted
// limited slopes coincide and the states are q -+ eps/2 * slope.
template <int LIM>
__device__ __forceinline__ double limited_slope(double a, double b) {
  return LIM == FV_LIM_VANLEER ? vanleer(a, b) : minmod(a, b);
}

// MUSCL face states of Eq. (6) across the face between q1 and q2 on the stencil
// q0..q3, walking along the normal: consecutive faces share the slope of the
// cell between them, which gives the right state of the one and the left state
// of the other.  On entry left is the face's left state (without a limiter:
// dm = q1 - q0) and d0 = q2 - q1; on return both are those of the next face.
// Without a limiter the kappa weights cL = eps(1-kappa)/4, cR = eps(1+kappa)/4
// apply.
template <int LIM>
__device__ __forceinline__ void muscl_step(const double *q, int s, double &left, double &d0, double h, double cL,
                                           double cR, double &QL, double &QR) {
  const double q2 = q[2 * s], dp = q[3 * s] - q2;
  if (LIM == FV_LIM_NONE) {
    QL = fma(cL, left, fma(cR, d0, q[s]));
    QR = fma(-cR, d0, fma(-cL, dp, q2));
    left = d0;
  } else {
    const double slope = limited_slope<LIM>(d0, dp);
    QL = left;
    QR = fma(-h, slope, q2);
    left = fma(h, slope, q2);
  }
  d0 = dp;
}
// The state of that walk before the face with stencil q[0], q[s], q[2s], q[3s].
template <int LIM>
__device__ __forceinline__ void muscl_start(const double *q, int s, double &left, double &d0, double h) {
  const double q1 = q[s], dm = q1 - q[0];
  d0 = q[2 * s] - q1;
  left = LIM == FV_LIM_NONE ? dm : fma(h, limited_slope<LIM>(dm, d0), q1);
}

template <int LIM>
__device__ __forceinline__ void muscl_states(double q0, double q1, double q2, double q3, double h, double cL,
                                             double cR, double &QL, double &QR) {
  const double q[4] = {q0, q1, q2, q3};
  double left, d0;
  muscl_start<LIM>(q, 1, left, d0, h);
  muscl_step<LIM>(q, 1, left, d0, h, cL, cR, QL, QR);
}

// Conserved state (rho, m, E) of primitive variables (rho, u, p), in place:
// m = rho u, E = p / (gamma - 1) + rho |u|^2 / 2.
template <int DIM>
__device__ __forceinline__ void to_conserved(double (&w)[DIM + 2], double inv_g1) {
  double q2 = w[1] * w[1];
#pragma unroll
  for (int d = 1; d < DIM; ++d) q2 = fma(w[1 + d], w[1 + d], q2);
  const double e = fma(scale_pow2<-1>(w[0]), q2, w[DIM + 1] * inv_g1);
#pragma unroll
  for (int d = 0; d < DIM; ++d) w[1 + d] = w[0] * w[1 + d];
  w[DIM + 1] = e;
}

// Every cell of the staged box from conserved to primitive variables, in
// place: u = m / rho, p = (gamma - 1)(E - m.u / 2).  Corner cells the stencils
// never read may hold zeros; whatever they turn into is never used.
template <int DIM>
__device__ __forceinline__ void box_to_primitive(double *tile, const TileGeom &G, double g1) {
  for (int c = threadIdx.x; c < G.plane; c += blockDim.x) {
    const double rho = tile[c];
    const double r = rcp_fp64(rho);
    double k = 0.0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const double m = tile[(1 + d) * G.plane + c];
      const double u = m * r;
      k = (d == 0) ? m * u : fma(m, u, k);
      tile[(1 + d) * G.plane + c] = u;
    }
    tile[(DIM + 1) * G.plane + c] = g1 * fma(-0.5, k, tile[(DIM + 1) * G.plane + c]);
  }
}

// The part of a stage update that does not depend on the fluxes: Us (stage
// 1), 3/4 Un + 1/4 Us (stage 2), 1/3 Un + 2/3 Us (stage 3); 0 for the residual.
template <int MODE>
__device__ __forceinline__ double stage_base(double us, double un) {
  if (MODE == MODE_RESIDUAL) return 0.0;
  if (MODE == MODE_STAGE1) return us;
  if (MODE == MODE_STAGE2) return fma(0.75, un, quarter(us));
  return fma(1.0 / 3.0, un, (2.0 / 3.0) * us);
}

// The value a cell's accumulation starts from: the stage base, plus the
// source term of Eq. (5) when one is set (src = -|Omega| for the residual,
// w dt for an RK stage, since dU/dt = -R/|Omega| has +S).
template <int MODE>
__device__ __forceinline__ double start_value(const StageArgs &a, double us, double un, long long idx, double src) {
  double b = stage_base<MODE>(us, un);
  if (a.S) b = (MODE == MODE_RESIDUAL) ? src * a.S[idx] : fma(src, a.S[idx], b);
  return b;
}

// The tile's cells in turn, x fastest, one per thread: coordinates by
// addition (one division per loop instead of one per cell).
template <int DIM, class SH>
struct CellLoop {
  int c, n, i, j, k, di, dj, dk, e0, e1;
  __device__ __forceinline__ CellLoop(const int ext[3])
      : c(threadIdx.x), n(ext[0] * ext[1] * (DIM == 3 ? ext[2] : 1)), e0(ext[0]), e1(ext[1]) {
    const int r = c / e0, s = block_threads<SH>(), q = s / e0;
    i = c - r * e0;
    di = s - q * e0;
    if (DIM == 3) {
      k = r / e1;
      j = r - k * e1;
      dk = q / e1;
      dj = q - dk * e1;
    } else {
      k = dk = 0;
      j = r;
      dj = q;
    }
  }
  __device__ __forceinline__ bool more() const { return c < n; }
  __device__ __forceinline__ void next() {
    c += block_threads<SH>();
    i += di;
    j += dj;
    if (i >= e0) {
      i -= e0;
      ++j;
    }
    if (DIM == 3) {
      k += dk;
      if (j >= e1) {
        j -= e1;
        ++k;
      }
    }
  }
};

// Every face flux of the tile along axis D, each evaluated once, and their
// differences into the tile's cells.  Faces form lines along D (fn faces
// each); a work item is a run of up to K consecutive faces of one line, so
// each face after the first takes one new stencil value and one new difference
// per variable, and the cell between two faces of a run gets its flux
// difference from the run's own thread, between the two fluxes: the FP64 work
// of the differences and of Eq. (6) runs beside the integer work of the flux,
// and no face buffer is written and read back.  A run's latest flux waits in
// `last` (its own slot), its first one in `first`, from which the thread of the
// run before completes its last cell after a barrier.  Items are numbered
// with the line fastest: neighbouring threads, neighbouring lines.
//
// The accumulator R holds, per cell, sum_d coef_d (F_{k+1/2} - F_{k-1/2}) on
// top of the start value (for the first axis: already there when `ready`, else
// formed from the tile and, in stages 2 and 3, from U^n in R).  The last axis
// writes its cells to a.out (x across the threads: coalesced).
// With a face buffer and separate difference passes, slopes evaluated twice
// and run-time offsets, a 2D cell-stage took 3266 thread instructions and KH
// 2048^2 2.23 ms per step; now 2530 and 1.83 (48x13 tiles, 96 threads).
//
// In 2D the axis D is a run-time value, so that the kernel holds one copy of
// this (long) code: with a copy per axis the warps wait for instructions (0.77
// cycles per issue against 0.08; KH 2048^2, 48x13 tiles: 1.95 ms per step
// against 1.83).  In 3D each axis has its own copy: the run-time offsets of
// five variables would spill (TGV 192^3: 6.85 ms against 6.99).  Variables are
// taken normal-first (rho, m_D, tangential momenta in axis order, E) by their
// place in memory.
template <int DIM, int LIM, int MODE, class SH>
__device__ __forceinline__ void face_pass(const int D, const double *__restrict__ tile, double *__restrict__ first,
                                          double *__restrict__ last, double *__restrict__ R, const StageArgs &a,
                                          const int o[3], const int ext[3], const TileGeom &G, double coef, bool ready,
                                          double (&nrm)[DIM + 2]) {
  constexpr int NV = DIM + 2;
  constexpr int NT = DIM - 1;
  const bool along_z = DIM == 3 && D == 2, last_axis = D == DIM - 1;
  auto pick = [=](int x, int y, int z) { return D == 0 ? x : (along_z ? z : y); };
  // the variable in each normal-first place
  int perm[NV];
  perm[0] = 0;
  perm[1] = 1 + D;
  perm[2] = D == 0 ? 2 : 1;
  if (DIM == 3) perm[3] = D == 2 ? 2 : 3;
  perm[NV - 1] = NV - 1;
  const int e2 = (DIM == 3) ? ext[2] : 1;
  const int fn = pick(ext[0], ext[1], e2) + 1;
  const int la = (D == 0) ? ext[1] : ext[0];  // line index = ca + la * cb over the two other axes
  const int nline = pick(ext[1] * e2, ext[0] * e2, ext[0] * ext[1]);
  const int threads = block_threads<SH>();
  const int K = run_length(fn, nline, threads, G.np);
  const int nrun = (fn + K - 1) / K;
  const int sstride = pick(1, G.BX, G.BX * G.BY);  // along the normal, in the tile
  const int rstride = pick(1, G.RX, G.RY);         // ... in the accumulator
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];
  const long long gstride = (D == 0) ? 1 : (along_z ? (long long)a.n[0] * a.n[1] : a.n[0]);
  const double h = a.half_eps;

  // one cell: flux difference dF[v], accumulator index r, tile pointer pc of its
  // centre, global index g
  auto cell = [&](const double (&dF)[NV], int r, const double *pc, long long g) {
    if (MODE == MODE_FLUXDIFF) {  // this axis's differences alone
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        if (D == 0)
          R[perm[v] * G.cells + r] = dF[v];  // written out after the pass (x runs do not coalesce)
        else
          a.fd[((long long)D * NV + perm[v]) * N + g] = dF[v];
      }
    } else if (D == 0 && !ready) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double *Rv = R + perm[v] * G.cells + r;
        *Rv = (MODE == MODE_RESIDUAL)
                  ? coef * dF[v]
                  : fma(coef, dF[v], stage_base<MODE>(pc[perm[v] * G.plane],
                                                      (MODE == MODE_STAGE2 || MODE == MODE_STAGE3) ? *Rv : 0.0));
      }
    } else {
      double x[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) x[v] = fma(coef, dF[v], R[perm[v] * G.cells + r]);
      if (last_axis) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          a.out[perm[v] * N + g] = x[v];
          if (MODE == MODE_RESIDUAL && a.norm_part) nrm[v] = fma(x[v], x[v], nrm[v]);
        }
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) R[perm[v] * G.cells + r] = x[v];
      }
    }
  };
  // places of the cell below face m of a line
  auto at = [&](int line, int m, const double *&pc, int &r, long long &g) {
    const int cb = (DIM == 3) ? line / la : 0, ca = line - cb * la;
    const int i = D == 0 ? m - 1 : ca, j = D == 1 ? m - 1 : (D == 0 ? ca : cb), k = DIM == 2 ? 0 : (D == 2 ? m - 1 : cb);
    pc = tile + (((DIM == 3) ? k + 2 : 0) * G.BY + j + 2) * G.BX + i + 2;
    r = k * G.RY + j * G.RX + i;
    g = ((long long)(o[2] + k) * a.n[1] + (o[1] + j)) * a.n[0] + (o[0] + i);
  };

  for (int item = threadIdx.x; item < nrun * nline; item += threads) {
    const int run = item / nline, line = item - run * nline;
    const int m0 = run * K, m1 = min(m0 + K, fn);
    const double *p;
    int r;
    long long g;
    at(line, m0, p, r, g);
    p -= sstride;  // p[0], p[s], p[2s], p[3s]: the stencil of face m
    double left[NV], d0[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) muscl_start<LIM>(p + perm[v] * G.plane, sstride, left[v], d0[v], h);
#pragma unroll 1
    for (int m = m0; m < m1; ++m) {
      double QL[NV], QR[NV], F[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v)
        muscl_step<LIM>(p + perm[v] * G.plane, sstride, left[v], d0[v], h, a.cL, a.cR, QL[v], QR[v]);
      if (a.recon == FV_RECON_PRIMITIVE) {  // (rho, u, p) face states -> (rho, m, E)
        to_conserved<DIM>(QL, a.inv_g1);
        to_conserved<DIM>(QR, a.inv_g1);
      }
      roe_F<NT>(QL, QR, a.g1, a.efix, a.inv2efix, a.rc, F);
      if (m == m0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) first[v * G.np + item] = F[v];
      } else {
        double dF[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) dF[v] = F[v] - last[v * G.np + item];
        cell(dF, r, p + sstride, g);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) last[v * G.np + item] = F[v];
      p += sstride;
      r += rstride;
      g += gstride;
    }
  }
  __syncthreads();
  // the cell between a run and the next one of its line
  for (int item = threadIdx.x; item < (nrun - 1) * nline; item += threads) {
    const int run = item / nline, line = item - run * nline;
    const double *pc;
    int r;
    long long g;
    at(line, (run + 1) * K, pc, r, g);
    double dF[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) dF[v] = first[v * G.np + item + nline] - last[v * G.np + item];
    cell(dF, r, pc, g);
  }
  if (!last_axis) __syncthreads();
}

// The tile's cells of the accumulator R into the SoA array dst (the
// flux-difference mode's x differences).
template <int DIM, class SH>
__device__ __forceinline__ void store_cells(const double *R, double *dst, const StageArgs &a, const int o[3],
                                            const int ext[3], const TileGeom &G) {
  constexpr int NV = DIM + 2;
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];
  for (CellLoop<DIM, SH> q(ext); q.more(); q.next()) {
    const long long gi = ((long long)(o[2] + q.k) * a.n[1] + (o[1] + q.j)) * a.n[0] + (o[0] + q.i);
    const int r = q.k * G.RY + q.j * G.RX + q.i;
#pragma unroll
    for (int v = 0; v < NV; ++v) dst[v * N + gi] = R[v * G.cells + r];
  }
}

// Stages 2 and 3: U^n of the tile's cells into the accumulator R, with
// asynchronous copies issued before the tile load completes, so both loads are
// in flight together.
template <int DIM, int MODE, class SH>
__device__ __forceinline__ void prefetch_un(double *R, const StageArgs &a, const int o[3], const int ext[3],
                                            const TileGeom &G) {
  if (MODE != MODE_STAGE2 && MODE != MODE_STAGE3) return;
  constexpr int NV = DIM + 2;
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];
  for (CellLoop<DIM, SH> q(ext); q.more(); q.next()) {
    const long long gi = ((long long)(o[2] + q.k) * a.n[1] + (o[1] + q.j)) * a.n[0] + (o[0] + q.i);
    const int r = q.k * G.RY + q.j * G.RX + q.i;
#pragma unroll
    for (int v = 0; v < NV; ++v) cp_async8(smem_u32(R + v * G.cells + r), a.Un + v * N + gi);
  }
}

// The start value of every cell of the tile into R (this thread's own U^n
// copies have completed): with a source, or where the tile is about to hold
// primitive variables, so that the reads of S stay coalesced.
template <int DIM, int MODE, class SH>
__device__ __forceinline__ void start_cells(const double *tile, double *R, const StageArgs &a, const int o[3],
                                            const int ext[3], const TileGeom &G, double src) {
  constexpr int NV = DIM + 2;
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];
  for (CellLoop<DIM, SH> q(ext); q.more(); q.next()) {
    const long long gi = ((long long)(o[2] + q.k) * a.n[1] + (o[1] + q.j)) * a.n[0] + (o[0] + q.i);
    const int r = q.k * G.RY + q.j * G.RX + q.i;
    const int lc = (((DIM == 3) ? q.k + 2 : 0) * G.BY + (q.j + 2)) * G.BX + (q.i + 2);
#pragma unroll
    for (int v = 0; v < NV; ++v)
      R[v * G.cells + r] =
          start_value<MODE>(a, tile[v * G.plane + lc],
                            (MODE == MODE_STAGE2 || MODE == MODE_STAGE3) ? R[v * G.cells + r] : 0.0, v * N + gi, src);
  }
}

// The bits of the step's largest wave-speed sum (in thread 0): one word, or
// the largest of the time-step kernel's per-CTA maxima (up to 128, one warp's
// four loads; non-negative doubles order like their bits).
__device__ __forceinline__ unsigned long long step_smax(const StageArgs &a) {
  if (!a.smax || threadIdx.x >= 32) return 0ull;
  if (a.nsmax <= 1) return *a.smax;
  unsigned long long m = 0ull;
  for (int q = threadIdx.x; q < a.nsmax; q += 32) m = a.smax[q] > m ? a.smax[q] : m;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, m, off);
    m = x > m ? x : m;
  }
  return m;
}

// All the work of one tile: stage the tile (TMA with mbarrier `bar` at parity
// `phase`, or plain loads), compute the face fluxes axis by axis, accumulate
// the residual (or the new stage state) and write it.  `tile` is the CTA's dynamic shared
// memory (128-byte aligned); s_coef (5 doubles) and red are static shared
// scratch.
// Returns false (uniformly across the CTA) if the tile load timed out.
template <int DIM, int MODE, int LIM = FV_LIM_MINMOD, class SH = AnyShape>
__device__ __forceinline__ bool tile_work(const CUtensorMap *tmap, const StageArgs &a, int bx, int by, int bz,
                                          double *tile, uint64_t *mbar, uint32_t phase, double *s_coef,
                                          double (*red)[32]) {
  constexpr int NV = DIM + 2;
  const TileGeom G = shape_geom<DIM, SH>(a.tile);
  const int tile_n[3] = {SH::fixed ? SH::TX : a.tile[0], SH::fixed ? SH::TY : a.tile[1],
                         DIM == 3 ? (SH::fixed ? SH::TZ : a.tile[2]) : 1};
  double *R = tile + NV * G.plane;
  double *first = R + NV * G.cells, *last = first + NV * G.np;
  const int o[3] = {bx * tile_n[0], by * tile_n[1], (DIM == 3) ? bz * tile_n[2] : 0};
  int ext[3];
  ext[0] = min(tile_n[0], a.n[0] - o[0]);
  ext[1] = min(tile_n[1], a.n[1] - o[1]);
  ext[2] = (DIM == 3) ? min(tile_n[2], a.n[2] - o[2]) : 1;
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];

  // ---- 1. stage the tile and its halo (and, stages 2-3, U^n into R)
  if (a.use_tma) {
    const uint32_t bar = smem_u32(mbar);
    if (threadIdx.x == 0) {
      mbar_expect_tx(bar, (uint32_t)(NV * G.plane * sizeof(double)));
      if (DIM == 2)
        tma_load_3d(smem_u32(tile), tmap, o[0] - 2, o[1] - 2, 0, bar);
      else
        tma_load_4d(smem_u32(tile), tmap, o[0] - 2, o[1] - 2, o[2] - 2, 0, bar);
    }
    prefetch_un<DIM, MODE, SH>(R, a, o, ext, G);
    const bool ok = mbar_wait_bounded(bar, phase, kTmaWaitNs);
    if (__syncthreads_or(!ok)) {
      if (MODE == MODE_STAGE2 || MODE == MODE_STAGE3) cp_async_wait_all();
      if (threadIdx.x == 0) {
        atomicOr(a.flags, FLAG_TIMEOUT);
        mbar_wait_bounded(bar, phase, kTmaWaitNs);  // let a late copy land before the CTA moves on
      }
      return false;
    }
    load_halo<DIM>(tile, a, o, ext, G, true);
  } else {
    prefetch_un<DIM, MODE, SH>(R, a, o, ext, G);
    for (CellLoop<DIM, SH> q(ext); q.more(); q.next()) {
      const long long src = ((long long)(o[2] + q.k) * a.n[1] + (o[1] + q.j)) * a.n[0] + (o[0] + q.i);
      const int dst = (((DIM == 3) ? q.k + 2 : 0) * G.BY + (q.j + 2)) * G.BX + (q.i + 2);
#pragma unroll
      for (int v = 0; v < NV; ++v) tile[v * G.plane + dst] = a.Us[v * N + src];
    }
    load_halo<DIM>(tile, a, o, ext, G, false);
  }

  // ---- 2./3. face fluxes and their differences per axis.  The step and the
  // per-axis scales are formed once per CTA (an FP64 division per thread
  // would cost ~2% of the kernel's FP64 work).
  const unsigned long long smax = (MODE != MODE_RESIDUAL && MODE != MODE_FLUXDIFF) ? step_smax(a) : 0ull;
  if (threadIdx.x == 0) {
    double dt = 0.0, w = 0.0;
    if (MODE != MODE_RESIDUAL) {
      dt = a.smax ? a.cfl / __longlong_as_double((long long)smax) : a.dt_fixed;
      w = (MODE == MODE_STAGE1) ? 1.0 : ((MODE == MODE_STAGE2) ? 0.25 : 2.0 / 3.0);
    }
    s_coef[0] = dt;
#pragma unroll
    for (int d = 0; d < 3; ++d) s_coef[1 + d] = (MODE == MODE_RESIDUAL) ? a.ds[d] : -w * dt * a.inv_h[d];
    s_coef[4] = (MODE == MODE_RESIDUAL) ? -a.vol : w * dt;
  }
  if (MODE == MODE_STAGE2 || MODE == MODE_STAGE3) cp_async_wait_all();  // this thread's U^n copies
  __syncthreads();
  bool ready = false;  // R holds the start values
  if (MODE != MODE_FLUXDIFF && (a.S || (MODE != MODE_RESIDUAL && a.recon == FV_RECON_PRIMITIVE))) {
    start_cells<DIM, MODE, SH>(tile, R, a, o, ext, G, s_coef[4]);
    ready = true;
    __syncthreads();
  }
  if (a.recon == FV_RECON_PRIMITIVE) {  // Eq. (6) on (rho, u, p)
    box_to_primitive<DIM>(tile, G, a.g1);
    __syncthreads();
  }
  const double dt = s_coef[0];
  double nrm[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) nrm[v] = 0.0;
  auto pass = [&](const int D) {
    face_pass<DIM, LIM, MODE, SH>(D, tile, first, last, R, a, o, ext, G, s_coef[1 + D], ready, nrm);
    if (MODE == MODE_FLUXDIFF && D == 0) store_cells<DIM, SH>(R, a.fd, a, o, ext, G);
  };
  if constexpr (DIM == 2) {
#pragma unroll 1
    for (int D = 0; D < 2; ++D) pass(D);
  } else {
    pass(0);
    pass(1);
    pass(2);
  }
  if (MODE == MODE_FLUXDIFF) return true;

  if (MODE == MODE_STAGE3 && a.t_acc && bx == 0 && by == 0 && bz == 0 && threadIdx.x == 0) *a.t_acc += dt;

  if (MODE == MODE_RESIDUAL && a.norm_part) {
    // CTA partial sums of R_v^2 (fixed reduction order: lanes, then warps)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      double sum = nrm[v];  // normal-first along the last axis
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, off);
      if (lane == 0) red[v == 0 || v == NV - 1 ? v : (v == 1 ? DIM : v - 1)][warp] = sum;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
      double sum = 0.0;
      const int nw = (blockDim.x + 31) >> 5;
      for (int q = 0; q < nw; ++q) sum += red[threadIdx.x][q];
      const long long tix = ((long long)bz * a.ntile[1] + by) * a.ntile[0] + bx;
      a.norm_part[tix * NV + threadIdx.x] = sum;
    }
  }
  return true;
}

// Dynamic shared memory of the stage kernels: tile box, cell accumulator, the
// runs' first and latest fluxes, then one mbarrier.
template <int DIM, class SH = AnyShape>
__device__ __forceinline__ uint64_t *stage_mbar(double *tile, const StageArgs &a) {
  constexpr int NV = DIM + 2;
  const TileGeom G = shape_geom<DIM, SH>(a.tile);
  return reinterpret_cast<uint64_t *>(tile + NV * (G.plane + G.cells + 2 * G.np));
}

__device__ __forceinline__ double *aligned_smem(unsigned char *raw) {
  return reinterpret_cast<double *>((reinterpret_cast<uintptr_t>(raw) + 127) & ~uintptr_t(127));
}

// One CTA per tile of the grid.  Register budget: MINB resident CTAs of MAXT
// threads per SM.  The kernels for any tile shape come in three sizes: 2D CTAs
// of up to kStage2dMaxThreads threads (168 registers per thread for the face
// runs and their integer-pipe flux) and of up to 256 (128 registers); 3D box
// CTAs of up to kStage3dMaxThreads threads (168 registers: the five-variable
// runs would spill at 128).  FV_STAGE_MIN_BLOCKS sets their MINB.
#ifndef FV_STAGE_MIN_BLOCKS
#define FV_STAGE_MIN_BLOCKS 2
#endif
template <int DIM, int MODE, int LIM, int MAXT, int MINB, class SH>
__global__ void __launch_bounds__(MAXT, MINB) stage_kernel(const __grid_constant__ CUtensorMap tmap, const StageArgs a) {
  constexpr int NV = DIM + 2;
  extern __shared__ unsigned char smem_raw[];
  __shared__ double s_coef[5];
  __shared__ double red[NV][32];
  double *tile = aligned_smem(smem_raw);
  uint64_t *mbar = stage_mbar<DIM, SH>(tile, a);
  if (a.use_tma) {
    if (threadIdx.x == 0) {
      prefetch_tensormap(&tmap);
      mbar_init(smem_u32(mbar), 1);
      fence_mbar_init();
    }
    __syncthreads();
  }
  long long b = a.tile_begin + blockIdx.x;
  const int bx = (int)(b % a.ntile[0]);
  b /= a.ntile[0];
  const int by = (int)(b % a.ntile[1]);
  const int bz = (int)(b / a.ntile[1]);
  tile_work<DIM, MODE, LIM, SH>(&tmap, a, bx, by, bz, tile, mbar, 0u, s_coef, red);
}

template <int DIM, int LIM, int MAXT, int MINB, class SH>
struct StageKernels {
  typedef void (*Fn)(const CUtensorMap, const StageArgs);
  static Fn of(int mode) {
    switch (mode) {
      case MODE_RESIDUAL: return stage_kernel<DIM, MODE_RESIDUAL, LIM, MAXT, MINB, SH>;
      case MODE_STAGE1: return stage_kernel<DIM, MODE_STAGE1, LIM, MAXT, MINB, SH>;
      case MODE_STAGE2: return stage_kernel<DIM, MODE_STAGE2, LIM, MAXT, MINB, SH>;
      case MODE_STAGE3: return stage_kernel<DIM, MODE_STAGE3, LIM, MAXT, MINB, SH>;
      default: return stage_kernel<DIM, MODE_FLUXDIFF, LIM, MAXT, MINB, SH>;
    }
  }
  static cudaError_t launch(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st) {
    const size_t smem = stage_smem_bytes(DIM, a.tile, threads);
    const long long nblk =
        a.tile_count > 0 ? a.tile_count : (long long)a.ntile[0] * a.ntile[1] * a.ntile[2] - a.tile_begin;
    of(mode)<<<dim3((unsigned)nblk), dim3(threads), smem, st>>>(*tmap, a);
    return cudaGetLastError();
  }
  // Allow each kernel the largest dynamic shared memory the device offers
  // (opt-in limit minus the kernel's static shared memory), so contexts with
  // different tile shapes never lower each other's limit.
  static cudaError_t set_attributes(size_t smem_optin) {
    cudaError_t e = cudaSuccess;
    for (int mode = MODE_RESIDUAL; mode <= MODE_FLUXDIFF && e == cudaSuccess; ++mode) {
      const void *k = (const void *)of(mode);
      cudaFuncAttributes fa;
      e = cudaFuncGetAttributes(&fa, k);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(smem_optin - fa.sharedSizeBytes));
    }
    return e;
  }
};

template <int DIM, int MAXT>
cudaError_t launch_stage_dim(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st) {
  constexpr int MINB = FV_STAGE_MIN_BLOCKS;
  if (a.limiter == FV_LIM_VANLEER)
    return StageKernels<DIM, FV_LIM_VANLEER, MAXT, MINB, AnyShape>::launch(mode, tmap, a, threads, st);
  if (a.limiter == FV_LIM_NONE)
    return StageKernels<DIM, FV_LIM_NONE, MAXT, MINB, AnyShape>::launch(mode, tmap, a, threads, st);
  return StageKernels<DIM, FV_LIM_MINMOD, MAXT, MINB, AnyShape>::launch(mode, tmap, a, threads, st);
}

template <int DIM, int MAXT>
cudaError_t set_stage_attributes_dim(int limiter, size_t smem_optin) {
  constexpr int MINB = FV_STAGE_MIN_BLOCKS;
  if (limiter == FV_LIM_VANLEER)
    return StageKernels<DIM, FV_LIM_VANLEER, MAXT, MINB, AnyShape>::set_attributes(smem_optin);
  if (limiter == FV_LIM_NONE)
    return StageKernels<DIM, FV_LIM_NONE, MAXT, MINB, AnyShape>::set_attributes(smem_optin);
  return StageKernels<DIM, FV_LIM_MINMOD, MAXT, MINB, AnyShape>::set_attributes(smem_optin);
}

// Launches the kernel compiled for shape SH when the stage's limiter, tile and
// threads are its own; false when they are not.
template <int DIM, int LIM, int MINB, class SH>
bool launch_shape(int mode, const CUtensorMap *tmap, const StageArgs &a, int threads, cudaStream_t st,
                  cudaError_t *e) {
  if (a.limiter != LIM || threads != SH::THREADS || a.tile[0] != SH::TX || a.tile[1] != SH::TY || a.tile[2] != SH::TZ)
    return false;
  *e = StageKernels<DIM, LIM, SH::THREADS, MINB, SH>::launch(mode, tmap, a, threads, st);
  return true;
}

}  // namespace fvk
