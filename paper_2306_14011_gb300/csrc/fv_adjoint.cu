// Discrete adjoint of the residual: out = sum_d scale_d J_d(U)^T lam, with J_d
// the Jacobian of the axis-d flux differences, plus a linear combination of up
// to three arrays (the reverse of the SSP-RK3 stage combinations).
//
// lam^T R = sum over faces f of ds (lam_{f-1} - lam_f) . F_f, F_f the flux
// between cells f-1 and f from their MUSCL states.  One CTA per tile computes,
// for every face whose stencil touches the tile, the cotangents of its left and
// right states (roe_F_vjp).  A cell c with limited slope s_c lends q_c + h s_c to
// the face above it and q_c - h s_c to the one below (h = eps/2), so with QLb
// and QRb the cotangents those faces send back,
//   q_c receives  QLb + QRb  and  s_c receives  t_c = h (QLb - QRb),
// and minmod passes t_c to the one difference it picked: +t_c to q_c and -t_c
// to q_{c-1} when it is q_c - q_{c-1}, -t_c to q_c and +t_c to q_{c+1} when it is
// q_{c+1} - q_c.  A thread walks a run of faces and forms, between two faces, the
// cell's own sum and t_c; each cell then gathers its two neighbours' t, so no
// atomics are needed.  Halo: 3 cells of U.  With transmissive boundaries the
// faces outside [0, n] do not exist, and the boundary cells also collect what
// was sent to their ghost copies (whose slopes pick nothing: a ghost's
// difference to its source is zero).
//
// What bounds it (2D, 1024^2): 285 FP64 instructions per cell and the integer
// work of the flux's products; before this form -- cotangents to four stencil
// cells kept per face, slopes evaluated twice per cell, products emulated bit
// for bit -- it took 340 and 0.96 ms.
#include "../../include/fv.h"
#include "fv_adjoint.cuh"
#include "fv_stage.cuh"

namespace fvk {

namespace {

struct AdjGeom {
  int UX, UY, UZ, uplane;  // U box with halo 3
  int cmax;                // cells along an axis pass: the tile and one more on either side, at most
  int np;                  // face runs of an axis pass, at most
  int cells;
};

__host__ __device__ constexpr int adj_run_length(int fn, int nline, int threads) { return (fn * nline + threads - 1) / threads; }

__host__ __device__ inline AdjGeom adj_geom(int dim, const int tile[3], int threads) {
  AdjGeom g;
  const int tx = tile[0], ty = tile[1], tz = dim == 3 ? tile[2] : 1;
  g.UX = tx + 6;
  g.UY = ty + 6;
  g.UZ = dim == 3 ? tz + 6 : 1;
  g.uplane = g.UX * g.UY * g.UZ;
  g.cells = tx * ty * tz;
  g.cmax = g.np = 0;
  for (int d = 0; d < dim; ++d) {
    const int t = d == 0 ? tx : (d == 1 ? ty : tz), nline = g.cells / t;
    // runs of K = ceil(faces / threads) faces: fewer than threads + nline, for
    // the ragged tiles' smaller counts too
    const int faces = (t + 3) * nline, items = faces < threads + nline ? faces : threads + nline;
    g.cmax = g.cmax > (t + 2) * nline ? g.cmax : (t + 2) * nline;
    g.np = g.np > items ? g.np : items;
  }
  return g;
}

// U box of 3 cells around the valid tile, every variable, plain loads with the
// boundary index map (corners included; they are never read).
template <int DIM>
__device__ void load_box(double *dst, const AdjArgs &a, const int o[3], const int ext[3], const AdjGeom &G) {
  constexpr int NV = DIM + 2;
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];
  const int ex = ext[0] + 6, ey = ext[1] + 6, ez = DIM == 3 ? ext[2] + 6 : 1;
  const int cnt = ex * ey * ez;
  for (int c = threadIdx.x; c < cnt; c += blockDim.x) {
    const int i = c % ex, r = c / ex, j = r % ey, k = r / ey;
    const int gx = ghost_source(o[0] - 3 + i, a.n[0], a.bc[0][0], a.bc[0][1]);
    const int gy = ghost_source(o[1] - 3 + j, a.n[1], a.bc[1][0], a.bc[1][1]);
    const int gz = DIM == 3 ? ghost_source(o[2] - 3 + k, a.n[2], a.bc[2][0], a.bc[2][1]) : 0;
    const long long s = ((long long)gz * a.n[1] + gy) * a.n[0] + gx;
    const int d = (k * G.UY + j) * G.UX + i;
#pragma unroll
    for (int v = 0; v < NV; ++v) dst[v * G.uplane + d] = a.U[v * N + s];
  }
}

// Faces along axis D, then the cells' gather.  The axis is a run-time argument:
// the kernel runs one copy of this (long) code for every axis; the variables are
// taken normal-first by their place in memory.  Per cell of the pass (index
// m * nline + line, m = 0 .. ext + 1 for the cells -1 .. ext along D): own[v] its
// own sum, tb[v] = t_c, pick the picked differences (2 bits per variable).
// HALF: h is 1/2 (eps = 1), so h * x is an exponent decrement on the integer
// pipe (scale_pow2) instead of an FP64 product.
template <int DIM, bool HALF>
__device__ __forceinline__ void adj_axis(const double *Ubox, double *own, double *tb, double *first, double *last,
                                         double *acc, int *pick, int *last_pick, const AdjArgs &a, const int o[3],
                                         const int ext[3], const AdjGeom &G, double scale, const int D) {
  constexpr int NV = DIM + 2;
  constexpr int NT = DIM - 1;
  const bool along_z = DIM == 3 && D == 2;
  auto of = [=](int x, int y, int z) { return D == 0 ? x : (along_z ? z : y); };
  int perm[NV];  // the variable in each normal-first place
  perm[0] = 0;
  perm[1] = 1 + D;
  perm[2] = D == 0 ? 2 : 1;
  if (DIM == 3) perm[3] = D == 2 ? 2 : 3;
  perm[NV - 1] = NV - 1;
  const int e2 = DIM == 3 ? ext[2] : 1;
  const int eD = of(ext[0], ext[1], e2), nD = of(a.n[0], a.n[1], a.n[2]), oD = of(o[0], o[1], o[2]);
  const int la = D == 0 ? ext[1] : ext[0];  // line = ca + la * cb over the two other axes
  const int nline = of(ext[1] * e2, ext[0] * e2, ext[0] * ext[1]);
  const int fn = eD + 3;
  const int K = adj_run_length(fn, nline, (int)blockDim.x), nrun = (fn + K - 1) / K;
  const int us = of(1, G.UX, G.UX * G.UY);  // U stencil stride
  const long long N = (long long)a.n[0] * a.n[1] * a.n[2];
  const long long gs = D == 0 ? 1 : (along_z ? (long long)a.n[0] * a.n[1] : a.n[0]);
  const double h = a.half_eps;
  const bool lo_trans = a.bc[D][0] == FV_BC_TRANSMISSIVE, hi_trans = a.bc[D][1] == FV_BC_TRANSMISSIVE;

  // the cell between two faces: what they send back to its state and slope
  auto cell = [&](int v, double QLb, double QRb, int pk, int at) {
    const double diff = QLb - QRb;
    const double t = HALF ? scale_pow2<-1>(diff) : h * diff;
    // +t, -t or nothing for the cell itself
    const double to_self = isel(pk == 0, 0.0, isel(pk == 1, t, mul_sign(t, -1.0)));
    own[v * G.cmax + at] = (QLb + QRb) + to_self;
    tb[v * G.cmax + at] = t;
  };

  for (int item = threadIdx.x; item < nrun * nline; item += blockDim.x) {
    const int run = item / nline, line = item - run * nline;
    const int m0 = run * K, m1 = min(m0 + K, fn);
    const int cb = DIM == 3 ? line / la : 0, ca = line - cb * la;
    // U stencil of local face m (global oD - 1 + m, between cells m - 2 and m - 1
    // of the tile): box coordinates m .. m + 3 along D
    const int i = D == 0 ? m0 : ca + 3, j = D == 1 ? m0 : (D == 0 ? ca : cb) + 3, k = DIM == 2 ? 0 : (D == 2 ? m0 : cb + 3);
    const double *p = Ubox + (k * G.UY + j) * G.UX + i;
    // the line's first cell in lam
    const long long g0 = D == 0 ? ((long long)(o[2] + cb) * a.n[1] + (o[1] + ca)) * a.n[0]
                                : (D == 1 ? (long long)(o[2] + cb) * a.n[1] * a.n[0] + (o[0] + ca)
                                          : (long long)(o[1] + cb) * a.n[0] + (o[0] + ca));
    // lam of cell c along D: beyond a transmissive side 0 (a ghost carries no residual)
    auto lam = [&](int c, double (&x)[NV]) {
      const bool none = (c < 0 && lo_trans) || (c >= nD && hi_trans);
      const long long at = g0 + gs * ghost_source(c, nD, a.bc[D][0], a.bc[D][1]);
#pragma unroll
      for (int v = 0; v < NV; ++v) x[v] = none ? 0.0 : a.lam[perm[v] * N + at];
    };
    double left[NV], d0[NV], l0[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) muscl_start<FV_LIM_MINMOD>(p + perm[v] * G.uplane, us, left[v], d0[v], h);
    lam(oD - 2 + m0, l0);
    int before = 0;  // the picks of the cell below the face
#pragma unroll 1
    for (int m = m0; m < m1; ++m, p += us) {
      const int fg = oD - 1 + m;
      double QL[NV], QR[NV], Gb[NV], bL[NV], bR[NV];
      int picks = 0;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const double dm = d0[v];
        muscl_step<FV_LIM_MINMOD>(p + perm[v] * G.uplane, us, left[v], d0[v], h, 0.0, 0.0, QL[v], QR[v]);
        picks |= minmod_pick(dm, d0[v]) << (2 * v);
      }
      double l1[NV];
      lam(fg, l1);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Gb[v] = l0[v] - l1[v];
        l0[v] = l1[v];
      }
      const bool real = !((lo_trans && fg < 0) || (hi_trans && fg > nD));
      if (real) {
        roe_F_vjp<NT>(QL, QR, a.g1, a.efix, a.inv2efix, Gb, bL, bR);
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) bL[v] = bR[v] = 0.0;
      }
      if (m == m0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) first[v * G.np + item] = bL[v];
      } else {
        const int at = (m - 1) * nline + line;
        pick[at] = before;
#pragma unroll
        for (int v = 0; v < NV; ++v) cell(v, bL[v], last[v * G.np + item], (before >> (2 * v)) & 3, at);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) last[v * G.np + item] = bR[v];
      before = picks;
    }
    last_pick[item] = before;
  }
  __syncthreads();
  for (int item = threadIdx.x; item < (nrun - 1) * nline; item += blockDim.x) {
    const int run = item / nline, line = item - run * nline;
    const int at = ((run + 1) * K - 1) * nline + line, pk = last_pick[item];
    pick[at] = pk;
#pragma unroll
    for (int v = 0; v < NV; ++v) cell(v, first[v * G.np + item + nline], last[v * G.np + item], (pk >> (2 * v)) & 3, at);
  }
  __syncthreads();
  // gather, and after the last axis the result
  const int ncell = ext[0] * ext[1] * e2;
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
    const int i = c % ext[0], rr = c / ext[0], j = DIM == 3 ? rr % ext[1] : rr, k = DIM == 3 ? rr / ext[1] : 0;
    const int m = of(i, j, k);  // the tile's cell m is the pass's cell m + 1
    const int line = of(j + la * k, i + la * k, i + la * j);
    const int at = (m + 1) * nline + line;
    const int pa = pick[at + nline], pb = pick[at - nline];
    const bool lo = lo_trans && oD + m == 0, hi = hi_trans && oD + m == nD - 1;
    const long long gi = ((long long)(o[2] + k) * a.n[1] + (o[1] + j)) * a.n[0] + (o[0] + i);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double *O = own + v * G.cmax + at, *t = tb + v * G.cmax + at;
      const double from_above = isel(((pa >> (2 * v)) & 3) == 1, mul_sign(t[nline], -1.0), 0.0);
      const double from_below = isel(((pb >> (2 * v)) & 3) == 2, t[-nline], 0.0);
      double s = (O[0] + from_above) + from_below;
      if (lo) s += O[-nline];  // the ghost next to a transmissive side is a copy of this cell
      if (hi) s += O[nline];
      const int pv = perm[v];
      double r = D == 0 ? scale * s : fma(scale, s, acc[pv * G.cells + c]);
      if (D < DIM - 1) {
        acc[pv * G.cells + c] = r;
      } else {
        if (a.A) r = fma(a.cA, a.A[pv * N + gi], r);
        if (a.B) r = fma(a.cB, a.B[pv * N + gi], r);
        if (a.C) r = fma(a.cC, a.C[pv * N + gi], r);
        a.out[pv * N + gi] = r;
      }
    }
  }
  if (D < DIM - 1) __syncthreads();
}

// 2D: two CTAs of 192 threads per SM, 168 registers (more of the smaller CTAs);
// 3D: the 8x8x8 tile's shared memory (222 KB) leaves one CTA, of 384 threads.
template <int DIM, bool HALF>
__global__ void __launch_bounds__(DIM == 2 ? kAdjThreads2d : kAdjThreads3d, DIM == 2 ? 2 : 1) adjoint_kernel(const AdjArgs a) {
  constexpr int NV = DIM + 2;
  extern __shared__ unsigned char smem_raw[];
  double *Ubox = aligned_smem(smem_raw);
  const AdjGeom G = adj_geom(DIM, a.tile, (int)blockDim.x);
  double *own = Ubox + NV * G.uplane, *tb = own + NV * G.cmax, *first = tb + NV * G.cmax, *last = first + NV * G.np;
  double *acc = last + NV * G.np;
  int *pick = reinterpret_cast<int *>(acc + NV * G.cells), *last_pick = pick + G.cmax;
  int b = blockIdx.x;
  const int bx = b % a.ntile[0];
  b /= a.ntile[0];
  const int by = b % a.ntile[1];
  const int bz = b / a.ntile[1];
  const int o[3] = {bx * a.tile[0], by * a.tile[1], DIM == 3 ? bz * a.tile[2] : 0};
  int ext[3];
  ext[0] = min(a.tile[0], a.n[0] - o[0]);
  ext[1] = min(a.tile[1], a.n[1] - o[1]);
  ext[2] = DIM == 3 ? min(a.tile[2], a.n[2] - o[2]) : 1;
  load_box<DIM>(Ubox, a, o, ext, G);
  __syncthreads();
#pragma unroll 1
  for (int D = 0; D < DIM; ++D)
    adj_axis<DIM, HALF>(Ubox, own, tb, first, last, acc, pick, last_pick, a, o, ext, G, a.scale[D], D);
}

}  // namespace

size_t adjoint_smem_bytes(int dim, const int tile[3], int threads) {
  const AdjGeom G = adj_geom(dim, tile, threads);
  const int nv = dim + 2;
  return 128 + sizeof(double) * (size_t)nv * (G.uplane + 2 * G.cmax + 2 * G.np + G.cells) + sizeof(int) * (size_t)(G.cmax + G.np);
}

template <int DIM, bool HALF>
cudaError_t launch_adjoint_kernel(const AdjArgs &a, unsigned blocks, int threads, size_t smem, cudaStream_t st) {
  const cudaError_t e = allow_full_smem((const void *)adjoint_kernel<DIM, HALF>);
  if (e == cudaSuccess) adjoint_kernel<DIM, HALF><<<blocks, threads, smem, st>>>(a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_adjoint(int dim, const AdjArgs &a, int threads, cudaStream_t st) {
  const size_t smem = adjoint_smem_bytes(dim, a.tile, threads);
  const unsigned blocks = (unsigned)((long long)a.ntile[0] * a.ntile[1] * a.ntile[2]);
  const bool half = a.half_eps == 0.5;
  if (dim == 2)
    return half ? launch_adjoint_kernel<2, true>(a, blocks, threads, smem, st)
                : launch_adjoint_kernel<2, false>(a, blocks, threads, smem, st);
  return half ? launch_adjoint_kernel<3, true>(a, blocks, threads, smem, st)
              : launch_adjoint_kernel<3, false>(a, blocks, threads, smem, st);
}

}  // namespace fvk
