// Surrogate network of the autotuner (paper Sec. 3.3, Table "para-setting"):
// a fully connected FP64 regressor with ReLU hidden layers and an identity
// output, trained by minibatch Adam on 1/2 mean squared error plus an L2
// penalty alpha/(2B) ||W||^2.
//
// Training is one cooperative kernel for all epochs.  A minibatch is two
// phases between grid barriers: (A) each CTA takes some of the batch's rows
// through the network and back, with their activations in shared memory and the
// weights from L2, and leaves activations and deltas in device memory; (B) each
// CTA sums its weights' gradients over the rows and updates them (and the
// transposed copy that the backward pass reads, coalesced).  What bounds it
// is FP64 (3 x 12 k FMA per row: 14 us a minibatch of 200 at the DFMA stream's
// rate on all SMs) and the two barriers; as one kernel per layer and operation,
// 14 launches a minibatch, it took 260 us, and now 49.  Every sum has a fixed order:
// results are deterministic run to run.
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/fv.h"
#include "fv_device.cuh"
#include "fv_internal.h"

namespace fvk {

namespace {

constexpr int kMaxLayers = 8;
constexpr int kMaxWidth = 1024;

// out[r][j] = act(sum_i in[r][i] W[i][j] + b[j])
__global__ void dense_forward(const double *in, long rows, int fin, int fout, const double *W, const double *b,
                              double *out, int relu) {
  const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (t >= rows * fout) return;
  const long r = t / fout;
  const int j = (int)(t - r * fout);
  const double *x = in + r * fin;
  double acc = b[j];
  for (int i = 0; i < fin; ++i) acc = fma(x[i], W[(long)i * fout + j], acc);
  out[t] = (relu && acc < 0.0) ? 0.0 : acc;
}

inline unsigned nblocks(long work, int threads) { return (unsigned)((work + threads - 1) / threads); }

struct Net {
  int nl;
  int sizes[kMaxLayers + 1];
  long woff[kMaxLayers], boff[kMaxLayers];
  long nparams;
};

bool make_net(int nl, const int *sizes, Net &net) {
  if (nl < 1 || nl > kMaxLayers || !sizes) return false;
  net.nl = nl;
  long off = 0;
  for (int l = 0; l <= nl; ++l) {
    if (sizes[l] < 1 || sizes[l] > kMaxWidth) return false;
    net.sizes[l] = sizes[l];
  }
  if (sizes[nl] != 1) return false;
  for (int l = 0; l < nl; ++l) {
    net.woff[l] = off;
    off += (long)sizes[l] * sizes[l + 1];
    net.boff[l] = off;
    off += sizes[l + 1];
  }
  net.nparams = off;
  return true;
}

constexpr int kTrainThreads = 256;
// Bound on a grid-barrier wait: 2 s, and 1 us per row of a minibatch.  A CTA may wait
// while another sums its parameters' gradients over the whole batch (about 45 ns a row).
constexpr uint64_t kTrainBarrierNs = 2000000000ull, kTrainRowNs = 1000ull;

struct TrainArgs {
  Net net;
  double *params, *wt;            // weights and biases; W_l transposed at woff[l]
  double *m, *v;                  // Adam moments
  const double *X, *y;
  const int *order;               // [epochs][n]
  long n;
  int B, epochs;
  double *acts[kMaxLayers + 1];   // [l >= 1]: [B][sizes[l]] activations
  double *delta[kMaxLayers];      // [l]: [B][sizes[l + 1]] deltas
  double *row_loss;               // [2][B] delta^2, of even and odd minibatches
  double *w2_part;                // per CTA: its share of sum W^2 before the update
  const double *lr;               // [epochs * batches] step sizes with the bias corrections
  double *loss;                   // [epochs]
  int *state;                     // [0] epochs run, [1] stop, [2] barrier timed out
  unsigned *bar;                  // barrier count, generation
  double alpha, b1, b2, eps, tol;
  int n_iter_no_change;
};

// Grid-wide barrier of a cooperative launch (bounded).  False in every thread
// of the CTA if the wait timed out, here or in a CTA that has left.
__device__ bool train_barrier(const TrainArgs &a) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned *gen = a.bar + 1;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(a.bar, 1u) == gridDim.x - 1) {
      atomicExch(a.bar, 0u);
      __threadfence();
      atomicAdd(a.bar + 1, 1u);
    } else if (!spin_while_equal(gen, g, kTrainBarrierNs + kTrainRowNs * (uint64_t)a.B)) {
      atomicExch(a.state + 2, 1);
      ok = 0;
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// out[r][j] = sum_i in[r][i] W[i][j] (+ bias[j] or 0) for the CTA's nr <= R rows:
// thread (part, j) sums a share of the i for all rows, then the shares are added
// in order.  in, out: shared memory, strides si and so; W: device memory written
// in this kernel, read past L1.
template <int R>
__device__ void cta_matvec(const double *in, int si, int fin, const double *W, const double *bias, int fout,
                           double *out, int so, double *red) {
  const int parts = max(1, min((int)blockDim.x / fout, 8)), per = (fin + parts - 1) / parts;
  for (int j0 = 0; j0 < fout; j0 += blockDim.x) {
    const int t = threadIdx.x, part = parts > 1 ? t / fout : 0, j = j0 + (parts > 1 ? t - part * fout : t);
    if (part < parts && j < fout) {
      double acc[R];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = (part == 0 && bias) ? __ldcg(bias + j) : 0.0;
      const int i1 = min(fin, (part + 1) * per);
      int i = part * per;
      for (; i + 16 <= i1; i += 16) {
        double w[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) w[q] = __ldcg(W + (long)(i + q) * fout + j);
#pragma unroll
        for (int q = 0; q < 16; ++q)
#pragma unroll
          for (int r = 0; r < R; ++r) acc[r] = fma(in[r * si + i + q], w[q], acc[r]);
      }
#pragma unroll 8
      for (; i < i1; ++i) {
        const double w = __ldcg(W + (long)i * fout + j);
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = fma(in[r * si + i], w, acc[r]);
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (parts == 1)
          out[r * so + j] = acc[r];
        else
          red[(r * parts + part) * fout + j] = acc[r];
      }
    }
    __syncthreads();
    if (parts > 1) {
      for (int q = threadIdx.x; q < R * fout; q += blockDim.x) {
        const int r = q / fout, jj = q - r * fout;
        double s = red[(r * parts) * fout + jj];
        for (int p = 1; p < parts; ++p) s += red[(r * parts + p) * fout + jj];
        out[r * so + jj] = s;
      }
      __syncthreads();
    }
  }
}

// R rows of one minibatch per CTA and turn.
template <int R>
__global__ void __launch_bounds__(kTrainThreads) train_kernel(const TrainArgs a) {
  extern __shared__ double sm[];
  const Net &net = a.net;
  int at[kMaxLayers + 1], width = 0, maxw = 0;  // a row's activations in shared memory
  for (int l = 0; l <= net.nl; ++l) {
    at[l] = width;
    width += net.sizes[l];
    maxw = net.sizes[l] > maxw ? net.sizes[l] : maxw;
  }
  double *act = sm, *dl = act + (long)R * width, *dn = dl + (long)R * maxw, *red = dn + (long)R * maxw;  // red: R * threads
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
  // the transposed weights
  for (int l = 0; l < net.nl; ++l)
    for (int q = tid; q < net.sizes[l] * net.sizes[l + 1]; q += nthr) {
      const int i = q / net.sizes[l + 1], j = q - i * net.sizes[l + 1];
      a.wt[net.woff[l] + (long)j * net.sizes[l] + i] = a.params[net.woff[l] + q];
    }
  if (!train_barrier(a)) return;
  double best = INFINITY;
  int stall = 0;
  long step = 0;
  for (int ep = 0; ep < a.epochs; ++ep) {
    double total = 0.0;  // CTA 0, thread 0: the epoch's loss
    for (long s0 = 0; s0 < a.n; s0 += a.B, ++step) {
      const int rows = (int)min((long)a.B, a.n - s0);
      const int *idx = a.order + (long)ep * a.n + s0;
      // ---- (A) rows forward and back
      for (int r0 = blockIdx.x * R; r0 < rows; r0 += gridDim.x * R) {
        const int nr = min(R, rows - r0);
        for (int q = threadIdx.x; q < R * net.sizes[0]; q += blockDim.x) {
          const int r = q / net.sizes[0], i = q - r * net.sizes[0];
          act[r * width + i] = a.X[(long)idx[r0 + min(r, nr - 1)] * net.sizes[0] + i];
        }
        __syncthreads();
        for (int l = 0; l < net.nl; ++l) {
          const int fi = net.sizes[l], fo = net.sizes[l + 1];
          cta_matvec<R>(act + at[l], width, fi, a.params + net.woff[l], a.params + net.boff[l], fo, act + at[l + 1],
                        width, red);
          for (int q = threadIdx.x; q < nr * fo; q += blockDim.x) {
            const int r = q / fo, j = q - r * fo;
            double x = act[r * width + at[l + 1] + j];
            if (l < net.nl - 1) {
              x = x < 0.0 ? 0.0 : x;
              act[r * width + at[l + 1] + j] = x;
            }
            a.acts[l + 1][(long)(r0 + r) * fo + j] = x;
          }
          __syncthreads();
        }
        if ((int)threadIdx.x < R) {
          const int r = threadIdx.x;
          const double e = act[r * width + at[net.nl]] - a.y[idx[r0 + min(r, nr - 1)]];
          dl[r * maxw] = e;
          if (r < nr) {
            a.delta[net.nl - 1][r0 + r] = e;
            a.row_loss[(step & 1) * a.B + r0 + r] = e * e;
          }
        }
        __syncthreads();
        for (int l = net.nl - 1; l > 0; --l) {
          const int fi = net.sizes[l], fo = net.sizes[l + 1];
          cta_matvec<R>(dl, maxw, fo, a.wt + net.woff[l], nullptr, fi, dn, maxw, red);
          for (int q = threadIdx.x; q < R * fi; q += blockDim.x) {
            const int r = q / fi, i = q - r * fi;
            const double x = act[r * width + at[l] + i] > 0.0 ? dn[r * maxw + i] : 0.0;  // ReLU derivative
            dl[r * maxw + i] = x;
            if (r < nr) a.delta[l - 1][(long)(r0 + r) * fi + i] = x;
          }
          __syncthreads();
        }
      }
      if (!train_barrier(a)) return;
      // ---- (B) gradients, Adam (efficient form: lr carries the bias corrections)
      // A CTA takes 32 consecutive parameters, a lane each; its warps share the rows.
      const double lr = a.lr[step];
      const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
      constexpr int kWarps = kTrainThreads / 32;
      double w2 = 0.0;
      for (long k0 = blockIdx.x * 32; k0 < net.nparams; k0 += (long)gridDim.x * 32) {
        const long k = k0 + lane;
        int l = 0;
        while (l + 1 < net.nl && k >= net.woff[l + 1]) ++l;
        const int fi = net.sizes[l], fo = net.sizes[l + 1], q = (int)(k - net.woff[l]);
        const int i = q / fo, j = q - i * fo;  // i = fi: the bias
        const bool weight = i < fi;
        if (k < net.nparams) {
          const double *D = a.delta[l] + j, *A = (l == 0 ? a.X : a.acts[l]) + (weight ? i : 0);
          double g[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) g[u] = 0.0;
          int r = warp;
          for (; r + 7 * kWarps < rows; r += 8 * kWarps) {
            double x[8], d[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int rr = r + u * kWarps;
              d[u] = __ldcg(D + (long)rr * fo);
              x[u] = __ldcg(A + (long)(l == 0 ? idx[rr] : rr) * fi);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) g[u] = fma(isel(weight, x[u], 1.0), d[u], g[u]);
          }
          for (; r < rows; r += kWarps) {
            const double d = __ldcg(D + (long)r * fo), x = __ldcg(A + (long)(l == 0 ? idx[r] : r) * fi);
            g[0] = fma(isel(weight, x, 1.0), d, g[0]);
          }
          red[threadIdx.x] = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]));
        }
        __syncthreads();
        if (warp == 0 && k < net.nparams) {
          double acc = red[lane];
#pragma unroll
          for (int w = 1; w < kWarps; ++w) acc += red[w * 32 + lane];
          const double w = __ldcg(a.params + k);
          if (weight) {
            acc += a.alpha * w;
            w2 = fma(w, w, w2);
          }
          const double g = acc / rows;
          const double mt = a.b1 * __ldcg(a.m + k) + (1.0 - a.b1) * g;
          const double vt = a.b2 * __ldcg(a.v + k) + (1.0 - a.b2) * g * g;
          a.m[k] = mt;
          a.v[k] = vt;
          const double wn = w - lr * mt / (sqrt(vt) + a.eps);
          a.params[k] = wn;
          if (weight) a.wt[net.woff[l] + (long)j * fi + i] = wn;
        }
        __syncthreads();
      }
      // this CTA's share of sum W^2, in a fixed order
      red[threadIdx.x] = w2;
      __syncthreads();
      for (int off = kTrainThreads / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
      }
      if (threadIdx.x == 0) a.w2_part[blockIdx.x] = red[0];
      if (!train_barrier(a)) return;
      // loss of the batch: 1/2 sum delta^2 + alpha/2 sum W^2.  CTA 0 sums it while
      // the others go on: they write the other half of row_loss next, and
      // w2_part only past a barrier that CTA 0 has to reach first
      if (blockIdx.x == 0) {
        double s = 0.0;
        for (int r = threadIdx.x; r < rows; r += blockDim.x) s += 0.5 * __ldcg(a.row_loss + (step & 1) * a.B + r);
        for (int q = threadIdx.x; q < (int)gridDim.x; q += blockDim.x) s += 0.5 * a.alpha * __ldcg(a.w2_part + q);
        red[threadIdx.x] = s;
        __syncthreads();
        for (int off = kTrainThreads / 2; off > 0; off >>= 1) {
          if ((int)threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
          __syncthreads();
        }
        total += red[0];
        __syncthreads();
      }
    }
    // stop once the epoch loss failed to improve by tol for more than n_iter_no_change epochs
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      const double lh = total / (double)a.n;
      a.loss[ep] = lh;
      stall = lh > best - a.tol ? stall + 1 : 0;
      best = lh < best ? lh : best;
      a.state[0] = ep + 1;
      if (a.n_iter_no_change > 0 && stall > a.n_iter_no_change) a.state[1] = 1;
    }
    if (!train_barrier(a)) return;
    if (__ldcg(a.state + 1)) return;
  }
}

// ---------------------------------------------------------------- forward pass on the integer pipes
//
// A layer is a matrix product, and the FP64 pipe does 5.3e11 multiply-adds a
// second; in one kernel per layer scoring was bound by it.  So the sums run in integers: the
// weights of an output (a column) and the activations of a row become
// fixed-point numbers of 77 bits below the largest one's exponent, as three
// balanced 26-bit limbs, exact for every value within 2^-24 of the largest.  Of
// the nine limb products the six that reach above 2^-77 of the largest product
// are summed, in three 64-bit accumulators (at most 3 x 1024 products below
// 2^50 each).  With the largest activation and weight in [1, 2) the sum S of a
// K-term row then has an absolute error below K 2^-73; it is taken where |S| >=
// 2^-18, that is an error below K 2^-55 |S|, less than an FP64 chain's.  Every
// other output (a sum that cancels or whose large factors meet small ones, and
// infinities, NaN and results near the ends of the range) is the FP64 chain of
// dense_forward, output by output.
//
// A CTA takes 16 rows through all layers, a thread 4 rows x 2 outputs of a
// layer at a time: per input 48 multiply-adds for 18 words of operands, from
// shared memory (activations, read by a warp as one line per limb) and L2
// (weights, each read once per CTA).  Scoring 200,000 rows of 14 features
// through (128, 64, 32): 4.30 -> 2.29 ms, bound by the 32 x 32 + 64-bit
// multiply-adds (six per product: 6.3e12 a second).
constexpr int kLimbBits = 26;
constexpr int kPredictThreads = 128, kPredictRows = 16;

// Where it pays, else one FP64 kernel per layer (dense_forward), us against it:
// four CTAs per SM ([14, 200, 200, 1], two: 200,000 rows 12,000 / 14,400, but
// 8000 rows 793 / 776); a wave of CTAs ([14, 128, 64, 32, 1]: 8000 rows 284 / 353,
// 2000 rows 246 / 224; [14, 64, 64, 1]: 8000 rows 212 / 245, 4000 rows 206 / 201);
// sums long enough for the conversions (32 inputs per output on average: 200,000
// rows of [14, 64, 64, 1] 1080 / 1960, [14, 32, 32, 1] 590 / 750); and two thirds
// of the products behind the first layer, whose inputs are the caller's and may
// be so far apart in scale that every sum is left to FP64 (features from 2^-40 to
// 2^40: [14, 128, 64, 32, 1] 2650 / 4300, but [64, 64, 1] 1950 / 1630).
constexpr size_t kPredictSmem = 55 * 1024;
inline bool predict_in_integers(const Net &net, long n, size_t smem) {
  long macs = 0, outputs = 0;
  for (int l = 0; l < net.nl; ++l) {
    macs += (long)net.sizes[l] * net.sizes[l + 1];
    outputs += net.sizes[l + 1];
  }
  return smem <= kPredictSmem && n >= 8192 && n <= 0x7fffffffl * kPredictRows && macs >= 32 * outputs &&
         3l * net.sizes[0] * net.sizes[1] <= macs;
}

// The exponent field of a value, 1 for subnormal numbers, 0 for zeros.
__device__ __forceinline__ int exponent_of(double v) {
  const int e = (__double2hiint(v) >> 20) & 0x7ff;
  return e == 0 && !izero(v) ? 1 : e;
}

// v = (l2 2^52 + l1 2^26 + l0) 2^(E - 1099), truncated below, for finite v of
// exponent field at most E (E >= 1); |l| <= 2^25.
__device__ __forceinline__ void to_limbs(double v, int E, int (&l)[3]) {
  const unsigned long long b = (unsigned long long)dbits(v);
  const int raw = (int)(b >> 52) & 0x7ff, e = raw ? raw : 1, d = E - e;
  unsigned long long m = (b & 0xfffffffffffffull) | (raw ? 0x10000000000000ull : 0ull);
  const int up = d < 24 ? 24 - d : 0, down = d > 24 ? d - 24 : 0;
  m = down < 64 ? m >> down : 0ull;
  const unsigned long long lo = m << up, hi = up ? m >> (64 - up) : 0ull;
  constexpr int mask = (1 << kLimbBits) - 1, half = 1 << (kLimbBits - 1);
  int l0 = (int)lo & mask;
  unsigned long long q = (lo >> kLimbBits) | (hi << (64 - kLimbBits));
  if (l0 >= half) l0 -= mask + 1, ++q;
  int l1 = (int)q & mask;
  q >>= kLimbBits;
  if (l1 >= half) l1 -= mask + 1, ++q;
  const int s = (long long)b < 0 ? -1 : 1;
  l[0] = s * l0;
  l[1] = s * l1;
  l[2] = s * (int)q;
}

// (s[2] 2^52 + s[1] 2^26 + s[0]) 2^(Ea + Ew - 2146), rounded to double, into
// *out; false where its error may exceed an FP64 chain's (see above).
__device__ __forceinline__ bool from_sums(const long long (&s)[3], int Ea, int Ew, double *out) {
  if (Ea == 2047 || Ew == 2047) return false;  // infinities and NaN
  *out = 0.0;
  if (Ea == 0 || Ew == 0) return true;         // all activations or all weights are zero
  const __int128 sum = ((__int128)s[2] << (2 * kLimbBits)) + ((__int128)s[1] << kLimbBits) + s[0];
  const bool neg = sum < 0;
  const unsigned __int128 a = neg ? -(unsigned __int128)sum : (unsigned __int128)sum;
  const unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
  if (hi < (1ull << 18)) return false;         // below 2^82: 2^100 is the largest factors' product in [1, 4)
  const int lz = __clzll((long long)hi);       // 17 .. 45
  const unsigned long long T = (hi << lz) | (lo >> (64 - lz));
  const int field = (127 - lz) - 100 + Ea + Ew - 1023;
  if (field < 1 || field > 2045) return false;
  const unsigned long long bits = ((unsigned long long)(field - 1) << 52) + (T >> 11) + ((T >> 10) & 1ull);
  *out = __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
  return true;
}

struct PredictArgs {
  Net net;
  const double *params, *X;
  double *out;
  long n;
  int *limbs;               // layer l at loff[l]: [fin][3][outputs rounded up to even]
  int *exps;                // [column over all layers]: exponent field of its largest weight
  long loff[kMaxLayers];
  int coff[kMaxLayers + 1];
  int width[2], maxin;      // widest even and odd level, widest layer input
};

__host__ __device__ constexpr int even(int n) { return (n + 1) & ~1; }

// One warp per output column: its exponent and the limbs of its weights.
__global__ void __launch_bounds__(128) weight_limbs(const PredictArgs a) {
  const int col = (int)(blockIdx.x * 4 + threadIdx.x / 32), lane = threadIdx.x & 31;
  if (col >= a.coff[a.net.nl]) return;
  int l = 0;
  while (col >= a.coff[l + 1]) ++l;
  const int j = col - a.coff[l], fi = a.net.sizes[l], fo = a.net.sizes[l + 1], fop = even(fo);
  const double *W = a.params + a.net.woff[l];
  int E = 0;
  if (j < fo)
    for (int i = lane; i < fi; i += 32) E = max(E, exponent_of(W[(long)i * fo + j]));
  E = __reduce_max_sync(0xffffffffu, E);
  if (lane == 0) a.exps[col] = E;
  for (int i = lane; i < fi; i += 32) {
    int q[3] = {0, 0, 0};
    if (E > 0 && E < 2047) to_limbs(W[(long)i * fo + j], E, q);
    for (int c = 0; c < 3; ++c) a.limbs[a.loff[l] + ((long)i * 3 + c) * fop + j] = q[c];
  }
}

// dense_forward's sum for one output, from the CTA's activations.
static __device__ __noinline__ double dense_fp64(const double *x, const double *W, const double *b, int fi, int fo,
                                                 int j) {
  double acc = b[j];
  for (int i = 0; i < fi; ++i) acc = fma(x[i * kPredictRows], W[(long)i * fo + j], acc);
  return acc;
}

__global__ void __launch_bounds__(kPredictThreads, 4) predict_kernel(const PredictArgs a) {
  constexpr int R = kPredictRows;
  extern __shared__ __align__(16) unsigned char raw[];
  double *const level[2] = {reinterpret_cast<double *>(raw), reinterpret_cast<double *>(raw) + R * a.width[0]};
  int *const limb = reinterpret_cast<int *>(reinterpret_cast<double *>(raw) + R * (a.width[0] + a.width[1]));
  __shared__ int row_exp[2][R];
  const int t = threadIdx.x;
  const long row0 = (long)blockIdx.x * R;
  const int rows = (int)min((long)R, a.n - row0);
  if (t < 2 * R) row_exp[t / R][t % R] = 0;
  __syncthreads();
  for (int q = t; q < R * a.net.sizes[0]; q += kPredictThreads) {
    const int r = q / a.net.sizes[0], i = q - r * a.net.sizes[0];
    const double v = r < rows ? a.X[row0 * a.net.sizes[0] + q] : 0.0;
    level[0][i * R + r] = v;
    atomicMax(&row_exp[0][r], exponent_of(v));
  }
  for (int l = 0; l < a.net.nl; ++l) {
    const int fi = a.net.sizes[l], fo = a.net.sizes[l + 1], fop = even(fo);
    const double *in = level[l & 1];
    double *dst = level[(l + 1) & 1];
    const int *Ea = row_exp[l & 1];
    const bool last = l == a.net.nl - 1;
    __syncthreads();  // this level's activations and exponents are there; the limbs before are read
    if (t < R) row_exp[(l + 1) & 1][t] = 0;
    for (int q = t; q < R * fi; q += kPredictThreads) {
      const int i = q / R, r = q % R, E = Ea[r];
      int c[3] = {0, 0, 0};
      if (E > 0 && E < 2047) to_limbs(in[q], E, c);
      for (int k = 0; k < 3; ++k) limb[(i * 3 + k) * R + r] = c[k];
    }
    __syncthreads();
    const double *W = a.params + a.net.woff[l], *b = a.params + a.net.boff[l];
    // a layer of few outputs splits its inputs over `parts` neighbouring lanes:
    // integer sums are exact in any order
    const int tiles = (R / 4) * (fop / 2);
    int parts = 1;
    while (parts < 32 && 2 * parts * tiles <= kPredictThreads) parts *= 2;
    const int part = t & (parts - 1);
    int top[4] = {0, 0, 0, 0};
    const int rg = t / parts % (R / 4);  // the same rows for all of a thread's tiles
    for (int q0 = 0; q0 < tiles; q0 += kPredictThreads / parts) {
      const int q = q0 + t / parts, j0 = q / (R / 4) * 2;
      if (parts == 1 && q >= tiles) break;
      const int mine = q < tiles ? fi : 0;  // (with parts > 1 all lanes take part in the sums below)
      const int *w = a.limbs + a.loff[l] + (long)part * 3 * fop + j0;
      const int *x = limb + part * 3 * R + rg * 4;
      long long s[4][2][3] = {};
#pragma unroll 2
      for (int i = part; i < mine; i += parts, w += 3 * parts * fop, x += 3 * parts * R) {
        int wl[3][2], xl[3][4];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const int2 v = __ldg(reinterpret_cast<const int2 *>(w + k * fop));
          wl[k][0] = v.x, wl[k][1] = v.y;
          const int4 u = *reinterpret_cast<const int4 *>(x + k * R);
          xl[k][0] = u.x, xl[k][1] = u.y, xl[k][2] = u.z, xl[k][3] = u.w;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            s[r][c][2] += (long long)xl[2][r] * wl[2][c];
            s[r][c][1] += (long long)xl[2][r] * wl[1][c];
            s[r][c][1] += (long long)xl[1][r] * wl[2][c];
            s[r][c][0] += (long long)xl[2][r] * wl[0][c];
            s[r][c][0] += (long long)xl[1][r] * wl[1][c];
            s[r][c][0] += (long long)xl[0][r] * wl[2][c];
          }
      }
      for (int m = parts / 2; m > 0; m /= 2) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int k = 0; k < 3; ++k) s[r][c][k] += __shfl_xor_sync(0xffffffffu, s[r][c][k], m);
      }
      if (part != 0 || q >= tiles) continue;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int j = j0 + c;
        if (j >= fo) continue;
        const int Ew = __ldg(a.exps + a.coff[l] + j);
        const double bias = b[j];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int row = rg * 4 + r;
          double v;
          if (from_sums(s[r][c], Ea[row], Ew, &v))
            v += bias;
          else
            v = dense_fp64(in + row, W, b, fi, fo, j);
          if (last) {
            if (row < rows) a.out[row0 + row] = v;
          } else {
            v = v < 0.0 ? 0.0 : v;
            dst[j * R + row] = v;
            top[r] = max(top[r], exponent_of(v));
          }
        }
      }
    }
    if (!last && part == 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (top[r]) atomicMax(&row_exp[(l + 1) & 1][rg * 4 + r], top[r]);
    }
  }
}

}  // namespace

// Forward pass over `rows` inputs in chunks; act0/act1: ping-pong buffers of
// chunk * max width doubles.
cudaError_t mlp_forward(const Net &net, const double *params, const double *X, long n, double *out, double *act0,
                        double *act1, long chunk, cudaStream_t st) {
  for (long r0 = 0; r0 < n; r0 += chunk) {
    const long rows = (n - r0 < chunk) ? n - r0 : chunk;
    const double *in = X + r0 * net.sizes[0];
    for (int l = 0; l < net.nl; ++l) {
      const bool last = l == net.nl - 1;
      double *dst = last ? out + r0 : ((l & 1) ? act1 : act0);
      const int fo = net.sizes[l + 1];
      dense_forward<<<nblocks(rows * fo, 256), 256, 0, st>>>(in, rows, net.sizes[l], fo, params + net.woff[l], params + net.boff[l], dst,
                                                             last ? 0 : 1);
      in = dst;
    }
  }
  return cudaGetLastError();
}

}  // namespace fvk

using namespace fvk;

extern "C" int fv_mlp_predict(int nl, const int *sizes, const double *params, const double *X, long n, double *out,
                              void *stream) {
  Net net;
  if (!make_net(nl, sizes, net) || !params || !X || !out || n < 0) return FV_EINVAL;
  if (n == 0) return FV_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaErrorMemoryAllocation;
  void *buf = nullptr;
  PredictArgs a;
  long limbs = 0;
  memset(&a, 0, sizeof(a));
  a.net = net;
  a.params = params;
  a.X = X;
  a.out = out;
  a.n = n;
  for (int l = 0; l < nl; ++l) {
    a.loff[l] = limbs;
    a.coff[l + 1] = a.coff[l] + even(sizes[l + 1]);
    limbs += 3l * sizes[l] * even(sizes[l + 1]);
    a.maxin = sizes[l] > a.maxin ? sizes[l] : a.maxin;
    a.width[l & 1] = sizes[l] > a.width[l & 1] ? sizes[l] : a.width[l & 1];
  }
  const size_t smem = (size_t)kPredictRows * (8 * (a.width[0] + a.width[1]) + 12 * a.maxin);
  if (predict_in_integers(net, n, smem)) {
    e = allow_full_smem((const void *)predict_kernel);
    if (e == cudaSuccess) e = cudaMalloc(&buf, sizeof(int) * (limbs + a.coff[nl]));
    if (e == cudaSuccess) {
      a.limbs = static_cast<int *>(buf);
      a.exps = a.limbs + limbs;
      weight_limbs<<<nblocks(a.coff[nl], 4), 128, 0, st>>>(a);
      predict_kernel<<<nblocks(n, kPredictRows), kPredictThreads, smem, st>>>(a);
      e = cudaGetLastError();
    }
  } else {
    int maxw = 1;
    for (int l = 1; l < nl; ++l) maxw = sizes[l] > maxw ? sizes[l] : maxw;
    const long chunk = n < 65536 ? n : 65536;
    e = cudaMalloc(&buf, sizeof(double) * 2 * chunk * maxw);
    double *act = static_cast<double *>(buf);
    if (e == cudaSuccess) e = mlp_forward(net, params, X, n, out, act, act + chunk * maxw, chunk, st);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(buf);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? FV_ENOMEM : FV_ECUDA;
  }
  return FV_OK;
}

extern "C" int fv_mlp_train(int nl, const int *sizes, double *params, const double *X, const double *y, long n,
                            const int *order, int epochs, const fv_mlp_hyper *h, double *loss_out,
                            int *epochs_run, void *stream) {
  Net net;
  if (!make_net(nl, sizes, net) || !params || !X || !y || !order || !h || n < 1 || epochs < 0 || h->batch < 1 ||
      !(h->lr > 0.0) || !(h->beta1 >= 0.0 && h->beta1 < 1.0) || !(h->beta2 >= 0.0 && h->beta2 < 1.0) ||
      !(h->eps > 0.0) || !(h->alpha >= 0.0))
    return FV_EINVAL;
  if (epochs_run) *epochs_run = 0;
  if (epochs == 0) return FV_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int B = h->batch < n ? h->batch : (int)n;
  long width = 0;
  int maxw = 1;
  for (int l = 0; l <= nl; ++l) {
    width += sizes[l];
    maxw = sizes[l] > maxw ? sizes[l] : maxw;
  }
  // grid: up to three CTAs per SM (train 4.0 ms for 80 minibatches of 200 rows
  // against 5.1 with one); rows of a CTA's turn: one, or two for larger batches
  int dev = 0, sms = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return FV_ECUDA;
  }
  auto smem = [&](int R) {
    return sizeof(double) * (size_t)R * ((size_t)width + 2 * (size_t)maxw + kTrainThreads);
  };
  const bool two = B > 3 * sms && smem(2) + 1024 <= (size_t)optin;
  void (*const kernel)(const TrainArgs) = two ? train_kernel<2> : train_kernel<1>;
  const size_t sm = smem(two ? 2 : 1);
  if (sm + 1024 > (size_t)optin) return FV_EUNSUPPORTED;  // (never: widths up to 1024, 8 layers take 108 KB)
  int per_sm = 0;
  if (allow_full_smem((const void *)kernel) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kTrainThreads, sm) != cudaSuccess || per_sm < 1) {
    (void)cudaGetLastError();
    return FV_ECUDA;
  }
  const int grid = (per_sm < 3 ? per_sm : 3) * sms;
  // workspace
  const long batches = (n + B - 1) / B;
  const size_t np = (size_t)net.nparams;
  const size_t nd = 3 * np + (size_t)B * (2 * (size_t)width + 2) + grid + (size_t)epochs + (size_t)epochs * batches;
  double *ws = nullptr;
  if (cudaMalloc(&ws, sizeof(double) * nd + 64) != cudaSuccess) {
    (void)cudaGetLastError();
    return FV_ENOMEM;
  }
  TrainArgs a;
  memset(&a, 0, sizeof(a));
  a.net = net;
  a.params = params;
  double *p = ws;
  a.m = p;
  a.v = p + np;
  a.wt = p + 2 * np;
  p += 3 * np;
  for (int l = 1; l <= nl; ++l) {
    a.acts[l] = p;
    p += (size_t)B * sizes[l];
    a.delta[l - 1] = p;
    p += (size_t)B * sizes[l];
  }
  a.row_loss = p;
  p += 2 * B;
  a.w2_part = p;
  p += grid;
  a.loss = p;
  p += epochs;
  double *lr = p;
  p += (size_t)epochs * batches;
  a.lr = lr;
  a.state = reinterpret_cast<int *>(p);
  a.bar = reinterpret_cast<unsigned *>(p) + 4;
  a.X = X;
  a.y = y;
  a.order = order;
  a.n = n;
  a.B = B;
  a.epochs = epochs;
  a.alpha = h->alpha;
  a.b1 = h->beta1;
  a.b2 = h->beta2;
  a.eps = h->eps;
  a.tol = h->tol;
  a.n_iter_no_change = h->n_iter_no_change;
  std::vector<double> hlr, hloss;
  try {
    hlr.resize((size_t)epochs * batches);
    hloss.resize(epochs);
  } catch (const std::bad_alloc &) {
    cudaFree(ws);
    return FV_ENOMEM;
  }
  for (size_t t = 1; t <= hlr.size(); ++t)
    hlr[t - 1] = h->lr * std::sqrt(1.0 - std::pow(h->beta2, (double)t)) / (1.0 - std::pow(h->beta1, (double)t));
  int state[3] = {0, 0, 0};
  cudaError_t e = cudaMemsetAsync(a.m, 0, sizeof(double) * 2 * np, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.state, 0, 64, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(lr, hlr.data(), sizeof(double) * hlr.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, a);
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(hloss.data(), a.loss, sizeof(double) * epochs, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(state, a.state, sizeof(state), cudaMemcpyDeviceToHost, st);
  const cudaError_t es = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = es;
  cudaFree(ws);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return FV_ECUDA;
  }
  if (loss_out)
    for (int q = 0; q < state[0]; ++q) loss_out[q] = hloss[q];
  if (epochs_run) *epochs_run = state[0];
  return state[2] ? FV_ETIMEOUT : FV_OK;
}
