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
// 14 launches a minibatch, it took 200 us.  Every sum has a fixed order:
// results are deterministic run to run.
#include <cmath>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/fv.h"
#include "fv_device.cuh"
#include "fv_internal.h"

namespace fvk {

namespace {

constexpr int kMaxLayers = 8;
constexpr int kMaxWidth = 1024;

// out[r][j] = act(sum_i in[row(r)][i] W[i][j] + b[j]); row(r) = idx[r] if idx.
__global__ void dense_forward(const double *in, const int *idx, long rows, int fin, int fout, const double *W,
                              const double *b, double *out, int relu) {
  const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (t >= rows * fout) return;
  const long r = t / fout;
  const int j = (int)(t - r * fout);
  const long src = idx ? (long)idx[r] : r;
  const double *x = in + src * fin;
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
constexpr uint64_t kTrainBarrierNs = 2000000000ull;  // 2 s bound on a grid-barrier wait

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
    } else if (!spin_while_equal(gen, g, kTrainBarrierNs)) {
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
      dense_forward<<<nblocks(rows * fo, 256), 256, 0, st>>>(in, nullptr, rows, net.sizes[l], fo,
                                                             params + net.woff[l], params + net.boff[l], dst,
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
  int maxw = 1;
  for (int l = 1; l < nl; ++l) maxw = sizes[l] > maxw ? sizes[l] : maxw;
  const long chunk = n < 65536 ? n : 65536;
  double *buf = nullptr;
  if (cudaMalloc(&buf, sizeof(double) * 2 * chunk * maxw) != cudaSuccess) {
    (void)cudaGetLastError();
    return FV_ENOMEM;
  }
  cudaError_t e = mlp_forward(net, params, X, n, out, buf, buf + chunk * maxw, chunk, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(buf);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return FV_ECUDA;
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
  if (cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess ||
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
  std::vector<double> hlr((size_t)epochs * batches), hloss(epochs);
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
