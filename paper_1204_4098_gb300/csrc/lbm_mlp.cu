// Warm-start network: a 4 -> 64 -> 64 -> 3 tanh MLP trained and evaluated
// by hand-written kernels.
//
//   h1 = tanh(x W1 + b1),  h2 = tanh(h1 W2 + b2),  y = h2 W3 + b3,
//   L  = mean over samples and outputs of (y - t)^2,  Adam updates.
//
// Parameters are one flat FP32 vector W1[4][64], b1[64], W2[64][64], b2[64],
// W3[64][3], b3[3] (4675 values).  Training runs as ONE launch of a cluster of
// 8 CTAs for all epochs.  The network is far too small for tensor cores to
// matter.  The paper has no network; it serves the warm start of the parameter
// sweeps.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <string>

#include "lbm.h"
#include "lbm_internal.h"

namespace cg = cooperative_groups;

namespace lbm {

constexpr int kIn = 4, kHid = 64, kOut = 3;
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kIn * kHid;    // 256
constexpr int kOffW2 = kOffB1 + kHid;          // 320
constexpr int kOffB2 = kOffW2 + kHid * kHid;   // 4416
constexpr int kOffW3 = kOffB2 + kHid;          // 4480
constexpr int kOffB3 = kOffW3 + kHid * kOut;   // 4672
constexpr int kNParams = kOffB3 + kOut;        // 4675
constexpr int kMaxBatch = 128;                 // largest minibatch

// ---------------------------------------------------------------------------
// training: one cluster of 8 CTAs for the whole run
// ---------------------------------------------------------------------------
// A minibatch is ~1.7 MFMA in short dependent phases, so what counts is how
// many SMs share each phase and what it costs to hand over between them.  CTA
// r of the cluster carries samples 16 r .. 16 r + 15 forward and backward with
// its own copy of the weights (one thread per few outputs of a layer), and
// owns hidden columns 8 r .. 8 r + 7: it sums the gradients of their weights
// over the whole minibatch and applies Adam, the moments in registers.  Two
// hand-overs per minibatch go through distributed shared memory: activations
// and their derivatives to the owners of the columns, updated weights to
// every copy, each closed by a cluster barrier.  Every sum runs in the order
// of one thread going through it alone (inputs, then samples, ascending), so
// results do not depend on the split.  One CTA of 128 threads, a sample per
// thread and 37 parameters each in the second half, took 72 us per minibatch
// of 128 against 7.6 us here.
constexpr int kClusterCtas = 8;
constexpr int kTrainThreads = 256;
constexpr int kCtaSamples = kMaxBatch / kClusterCtas;  // 16
constexpr int kCols = kHid / kClusterCtas;             // hidden columns a CTA owns
constexpr int kPad = kHid + 4;  // padded row: 16-byte aligned, rows 4 banks apart

struct TrainSmem {
  float W1[kIn * kHid], b1[kHid], W2[kHid * kPad], b2[kHid], W3t[kOut * kHid], b3[kOut + 1];
  float H1[kMaxBatch * kPad];       // every sample
  float H2[kCtaSamples * kPad];     // this CTA's samples
  float DZ2[kCtaSamples * kPad];
  float H2c[kMaxBatch * kCols];     // this CTA's columns of every sample
  float DZ2c[kMaxBatch * kCols];
  float DZ1c[kMaxBatch * kCols];
  float X[kMaxBatch * kIn];         // every sample
  float DY[kMaxBatch * 4];
  float G[kHid * kCols];            // gradients of this CTA's columns of W2
  float T[kCtaSamples * 4];         // this CTA's samples
  float sq[kMaxBatch];              // squared errors (CTA 0)
  float red[kMaxBatch / 32];
};

// Where parameter p of the flat vector lives in a CTA's copy of the weights (an
// offset in floats from the start of TrainSmem and of PredictSmem, which begin
// alike; W3 transposed for vector loads).
__device__ __forceinline__ int weight_slot(int p) {
  constexpr int o1 = 0, ob1 = o1 + kIn * kHid, o2 = ob1 + kHid, ob2 = o2 + kHid * kPad,
                o3 = ob2 + kHid, ob3 = o3 + kHid * kOut;
  if (p < kOffB1) return o1 + p;
  if (p < kOffW2) return ob1 + (p - kOffB1);
  if (p < kOffB2) return o2 + (p - kOffW2) / kHid * kPad + (p - kOffW2) % kHid;
  if (p < kOffW3) return ob2 + (p - kOffB2);
  if (p < kOffB3) return o3 + (p - kOffW3) % kOut * kHid + (p - kOffW3) / kOut;
  return ob3 + (p - kOffB3);
}

// mode 0: train `epochs` epochs over `order` (epochs x n sample indices) with
// Adam; mode 1: one full-batch gradient of the first `n` samples (n <= 128)
// into grad_out, no update.  loss_out gets the last minibatch's loss.
__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(kTrainThreads)
mlp_train_kernel(float* params, float* adam_m, float* adam_v, const float* __restrict__ X,
                 const float* __restrict__ Y, int n, const int* __restrict__ order, int epochs,
                 int batch, float lr, int t0, int mode, float* grad_out, float* loss_out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem& s = *reinterpret_cast<TrainSmem*>(smem_raw);
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = int(cluster.block_rank());
  for (int p = tid; p < kNParams; p += kTrainThreads)
    reinterpret_cast<float*>(&s)[weight_slot(p)] = params[p];

  // The parameters this thread owns (-1: none): two neighbours of the CTA's
  // columns of W2, and in warps 4 .. 7 one of its columns of W1, of b1 or b2,
  // of W3, and (CTA 0) of b3.
  constexpr int kOwn = 3;
  int own[kOwn];
  own[0] = kOffW2 + (tid >> 2) * kHid + kCols * rank + 2 * (tid & 3);
  own[1] = own[0] + 1;
  own[2] = -1;
  if (warp == 4) {
    own[2] = kOffW1 + lane / kCols * kHid + kCols * rank + lane % kCols;
  } else if (warp == 5 && lane < 2 * kCols) {
    own[2] = (lane < kCols ? kOffB1 : kOffB2) + kCols * rank + lane % kCols;
  } else if (warp == 6 && lane < kCols * kOut) {
    own[2] = kOffW3 + kCols * kOut * rank + lane;
  } else if (warp == 7 && lane < kOut && rank == 0) {
    own[2] = kOffB3 + lane;
  }
  float m[kOwn], v[kOwn];
#pragma unroll
  for (int q = 0; q < kOwn; ++q) {
    m[q] = (mode == 0 && own[q] >= 0) ? adam_m[own[q]] : 0.f;
    v[q] = (mode == 0 && own[q] >= 0) ? adam_v[own[q]] : 0.f;
  }
  const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
  float b1t = powf(beta1, float(t0)), b2t = powf(beta2, float(t0));
  const int per_epoch = (n + batch - 1) / batch;
  const int steps = mode == 0 ? epochs * per_epoch : 1;

  // a minibatch's rows travel in registers (thread b: sample b) from the end
  // of the minibatch before, their indices from one minibatch earlier still
  // (a row's address waits for its index)
  float4 xin = make_float4(0.f, 0.f, 0.f, 0.f);
  float tin[kOut] = {0.f, 0.f, 0.f};
  int next = 0;  // this thread's sample of the minibatch that load_rows takes
  auto load_index = [&](int st) {
    if (mode != 0 || st >= steps || tid >= kMaxBatch) return;
    const int e = st / per_epoch, k0 = (st % per_epoch) * batch;
    if (tid < min(batch, n - k0)) next = order[size_t(e) * n + k0 + tid];
  };
  auto load_rows = [&](int st) {
    if (st >= steps || tid >= kMaxBatch) return;
    const int k0 = (st % per_epoch) * batch;
    const int nb = mode == 0 ? min(batch, n - k0) : n;
    if (tid >= nb) return;
    const int idx = mode == 0 ? next : tid;
    xin = reinterpret_cast<const float4*>(X)[idx];
    if (tid / kCtaSamples == rank)
#pragma unroll
      for (int k = 0; k < kOut; ++k) tin[k] = Y[size_t(idx) * kOut + k];
  };
  load_index(0);
  load_rows(0);
  load_index(1);
  cluster.sync();  // every CTA of the cluster runs: its shared memory may be written

  for (int st = 0; st < steps; ++st) {
    const int k0 = (st % per_epoch) * batch;
    const int nb = mode == 0 ? min(batch, n - k0) : n;
    const int first = kCtaSamples * rank;                      // this CTA's samples
    const float scale = 2.f / float(nb * kOut);
    const int mine = max(0, min(kCtaSamples, nb - first));
    if (tid < nb) reinterpret_cast<float4*>(s.X)[tid] = xin;
    if (tid >= first && tid < first + mine)
#pragma unroll
      for (int k = 0; k < kOut; ++k) s.T[(tid - first) * 4 + k] = tin[k];
    __syncthreads();
    // hidden layer 1: thread = sample b, columns j .. j + 3; to every CTA
    {
      const int b = tid >> 4, j = (tid & 15) * 4;
      if (b < mine) {
        float h[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float z = s.b1[j + q];
#pragma unroll
          for (int i = 0; i < kIn; ++i)
            z = fmaf(s.X[(first + b) * kIn + i], s.W1[i * kHid + j + q], z);
          h[q] = tanhf(z);
        }
        const float4 hv = make_float4(h[0], h[1], h[2], h[3]);
        float* const at = &s.H1[(first + b) * kPad + j];
#pragma unroll
        for (int r = 0; r < kClusterCtas; ++r)
          *reinterpret_cast<float4*>(cluster.map_shared_rank(at, r)) = hv;
      }
    }
    __syncthreads();
    // hidden layer 2: thread = samples 2 warp, 2 warp + 1, columns 2 lane, 2 lane + 1
    {
      const int b = 2 * warp, j = 2 * lane;
      if (b < mine) {
        const float* const ha = &s.H1[(first + b) * kPad];
        const float* const hb = ha + kPad;  // (past the last sample: unused)
        float z[2][2] = {{s.b2[j], s.b2[j + 1]}, {s.b2[j], s.b2[j + 1]}};
#pragma unroll
        for (int i = 0; i < kHid; i += 4) {
          const float4 a4 = *reinterpret_cast<const float4*>(ha + i);
          const float4 b4 = *reinterpret_cast<const float4*>(hb + i);
          const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float2 w = *reinterpret_cast<const float2*>(&s.W2[(i + q) * kPad + j]);
            z[0][0] = fmaf(av[q], w.x, z[0][0]);
            z[0][1] = fmaf(av[q], w.y, z[0][1]);
            z[1][0] = fmaf(bv[q], w.x, z[1][0]);
            z[1][1] = fmaf(bv[q], w.y, z[1][1]);
          }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (b + q < mine) {
            const float2 h = make_float2(tanhf(z[q][0]), tanhf(z[q][1]));
            *reinterpret_cast<float2*>(&s.H2[(b + q) * kPad + j]) = h;
            *reinterpret_cast<float2*>(cluster.map_shared_rank(
                &s.H2c[(first + b + q) * kCols + j % kCols], j / kCols)) = h;
          }
      }
    }
    __syncthreads();
    // outputs and their derivatives: thread = sample b, output k (of four lanes)
    if (tid < 4 * kCtaSamples) {
      const int b = tid >> 2, k = tid & 3, kk = k < kOut ? k : 0;
      float y = s.b3[kk];
#pragma unroll
      for (int j = 0; j < kHid; j += 4) {
        const float4 h = *reinterpret_cast<const float4*>(&s.H2[b * kPad + j]);
        const float4 w = *reinterpret_cast<const float4*>(&s.W3t[kk * kHid + j]);
        y = fmaf(h.x, w.x, y);
        y = fmaf(h.y, w.y, y);
        y = fmaf(h.z, w.z, y);
        y = fmaf(h.w, w.w, y);
      }
      const float d = y - s.T[b * 4 + kk];
      const float d1 = __shfl_down_sync(0xffffffffu, d, 1), d2 = __shfl_down_sync(0xffffffffu, d, 2);
      if (b < mine) {
        const float dy = scale * d;
        float* const at = &s.DY[(first + b) * 4 + k];
        if (k < kOut)
#pragma unroll
          for (int r = 0; r < kClusterCtas; ++r) *cluster.map_shared_rank(at, r) = dy;
        if (k == 0)
          *cluster.map_shared_rank(&s.sq[first + b], 0) =
              fmaf(d2, d2, fmaf(d1, d1, fmaf(d, d, 0.f)));
      }
    }
    __syncthreads();
    // through layer 2: thread = sample b, columns j .. j + 3
    {
      const int b = tid >> 4, j = (tid & 15) * 4;
      if (b < mine) {
        const float4 h4 = *reinterpret_cast<const float4*>(&s.H2[b * kPad + j]);
        const float hv[4] = {h4.x, h4.y, h4.z, h4.w};
        float g[4] = {0.f, 0.f, 0.f, 0.f}, dz[4];
#pragma unroll
        for (int k = 0; k < kOut; ++k) {
          const float dy = s.DY[(first + b) * 4 + k];
          const float4 w = *reinterpret_cast<const float4*>(&s.W3t[k * kHid + j]);
          g[0] = fmaf(dy, w.x, g[0]);
          g[1] = fmaf(dy, w.y, g[1]);
          g[2] = fmaf(dy, w.z, g[2]);
          g[3] = fmaf(dy, w.w, g[3]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) dz[q] = g[q] * (1.f - hv[q] * hv[q]);
        const float4 dv = make_float4(dz[0], dz[1], dz[2], dz[3]);
        *reinterpret_cast<float4*>(&s.DZ2[b * kPad + j]) = dv;
        *reinterpret_cast<float4*>(cluster.map_shared_rank(
            &s.DZ2c[(first + b) * kCols + j % kCols], j / kCols)) = dv;
      }
    }
    __syncthreads();
    // through layer 1: thread = samples 2 warp, 2 warp + 1, rows lane, lane + 32
    {
      const int b = 2 * warp;
      if (b < mine) {
        const float* const da = &s.DZ2[b * kPad];
        const float* const db = da + kPad;  // (past the last sample: unused)
        float g[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
        for (int j = 0; j < kHid; j += 4) {
          const float4 a4 = *reinterpret_cast<const float4*>(da + j);
          const float4 b4 = *reinterpret_cast<const float4*>(db + j);
          const float4 w0 = *reinterpret_cast<const float4*>(&s.W2[lane * kPad + j]);
          const float4 w1 = *reinterpret_cast<const float4*>(&s.W2[(lane + 32) * kPad + j]);
          const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
          const float w0v[4] = {w0.x, w0.y, w0.z, w0.w}, w1v[4] = {w1.x, w1.y, w1.z, w1.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            g[0][0] = fmaf(av[q], w0v[q], g[0][0]);
            g[0][1] = fmaf(av[q], w1v[q], g[0][1]);
            g[1][0] = fmaf(bv[q], w0v[q], g[1][0]);
            g[1][1] = fmaf(bv[q], w1v[q], g[1][1]);
          }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (b + q < mine)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              const int i = lane + 32 * r;
              const float h = s.H1[(first + b + q) * kPad + i];
              *cluster.map_shared_rank(&s.DZ1c[(first + b + q) * kCols + i % kCols], i / kCols) =
                  g[q][r] * (1.f - h * h);
            }
      }
    }
    load_rows(st + 1);
    load_index(st + 2);
    cluster.sync();  // every sample's activations and derivatives are in place

    // gradients of the owned parameters over the minibatch, then Adam
    b1t *= beta1;
    b2t *= beta2;
    float gs = 0.f;  // of own[2]
    auto sums = [&](int count) {  // over the samples 0 .. count - 1
      if (warp < 4) {
        const float* const h = &s.H1[tid & 63];
        const float* const dz = &s.DZ2c[4 * (tid >> 6)];
        float g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 16
        for (int b = 0; b < count; ++b) {
          const float4 d = *reinterpret_cast<const float4*>(dz + b * kCols);
          const float hv = h[b * kPad];
          g[0] = fmaf(hv, d.x, g[0]);
          g[1] = fmaf(hv, d.y, g[1]);
          g[2] = fmaf(hv, d.z, g[2]);
          g[3] = fmaf(hv, d.w, g[3]);
        }
        // (W2's sums are taken four columns a thread, its updates two)
        *reinterpret_cast<float4*>(&s.G[(tid & 63) * kCols + 4 * (tid >> 6)]) =
            make_float4(g[0], g[1], g[2], g[3]);
      } else if (own[2] < 0) {
        return;
      } else if (warp == 4) {
#pragma unroll 16
        for (int b = 0; b < count; ++b)
          gs = fmaf(s.X[b * kIn + lane / kCols], s.DZ1c[b * kCols + lane % kCols], gs);
      } else if (warp == 5) {
        const float* const d = lane < kCols ? &s.DZ1c[lane] : &s.DZ2c[lane - kCols];
#pragma unroll 16
        for (int b = 0; b < count; ++b) gs += d[b * kCols];
      } else if (warp == 6) {
#pragma unroll 16
        for (int b = 0; b < count; ++b)
          gs = fmaf(s.H2c[b * kCols + lane / kOut], s.DY[b * 4 + lane % kOut], gs);
      } else {
#pragma unroll 16
        for (int b = 0; b < count; ++b) gs += s.DY[b * 4 + lane];
      }
    };
    if (nb == kMaxBatch) sums(kMaxBatch);
    else sums(nb);
    __syncthreads();
    const float2 g2 = *reinterpret_cast<const float2*>(&s.G[2 * tid]);
    const float g[kOwn] = {g2.x, g2.y, gs};
    if (mode == 1) {
#pragma unroll
      for (int q = 0; q < kOwn; ++q)
        if (own[q] >= 0) grad_out[own[q]] = g[q];
    } else {
      float w[kOwn];
#pragma unroll
      for (int q = 0; q < kOwn; ++q) {
        if (own[q] < 0) continue;
        m[q] = fmaf(beta1, m[q], (1.f - beta1) * g[q]);
        v[q] = fmaf(beta2, v[q], (1.f - beta2) * g[q] * g[q]);
        const float mh = m[q] / (1.f - b1t), vh = v[q] / (1.f - b2t);
        w[q] = reinterpret_cast<float*>(&s)[weight_slot(own[q])] - lr * mh / (sqrtf(vh) + eps);
      }
      float* const at = reinterpret_cast<float*>(&s) + weight_slot(own[0]);
#pragma unroll
      for (int r = 0; r < kClusterCtas; ++r)
        *reinterpret_cast<float2*>(cluster.map_shared_rank(at, r)) = make_float2(w[0], w[1]);
      if (own[2] >= 0) {
        float* const one = reinterpret_cast<float*>(&s) + weight_slot(own[2]);
#pragma unroll
        for (int r = 0; r < kClusterCtas; ++r) *cluster.map_shared_rank(one, r) = w[2];
      }
    }
    if (st == steps - 1 && rank == 0 && loss_out) {
      // the last minibatch's loss
      float sq = tid < nb ? s.sq[tid] : 0.f;
      for (int o = 16; o > 0; o >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, o);
      if (tid < kMaxBatch && lane == 0) s.red[warp] = sq;
      __syncthreads();
      if (tid == 0) {
        float t = 0.f;
        for (int w = 0; w < kMaxBatch / 32; ++w) t += s.red[w];
        *loss_out = t / float(nb * kOut);
      }
    }
    cluster.sync();  // every copy of the weights is updated; the buffers are free
  }
#pragma unroll
  for (int q = 0; q < kOwn; ++q) {
    const int p = own[q];
    if (p < 0) continue;
    params[p] = reinterpret_cast<float*>(&s)[weight_slot(p)];
    if (mode == 0) {
      adam_m[p] = m[q];
      adam_v[p] = v[q];
    }
  }
}

// y = network(x).  A CTA stages the weights once and takes groups of 16
// samples in turn, spread over its threads as in training; sums run in the
// same order.  (One sample per thread put 256 samples on one SM, each thread
// 4096 multiply-adds deep.)  X and Y may be mapped host memory.
constexpr int kPredictSamples = 16;
struct PredictSmem {
  float W1[kIn * kHid], b1[kHid], W2[kHid * kPad], b2[kHid], W3t[kOut * kHid], b3[kOut + 1];
  float X[kPredictSamples * kIn];
  float H1[kPredictSamples * kPad];
  float H2[kPredictSamples * kPad];
};
static_assert(offsetof(PredictSmem, W3t) == offsetof(TrainSmem, W3t) &&
                  offsetof(PredictSmem, b3) == offsetof(TrainSmem, b3),
              "weight_slot serves both");

__global__ void __launch_bounds__(kTrainThreads)
mlp_predict_kernel(const float* __restrict__ params, const float* __restrict__ X, int n,
                   float* Y) {
  __shared__ __align__(16) PredictSmem s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int groups = (n + kPredictSamples - 1) / kPredictSamples;
  float xin = 0.f;  // the group's inputs: thread = one value
  auto load = [&](int g) {
    const size_t at = size_t(g) * kPredictSamples * kIn + tid;
    if (g < groups && tid < kPredictSamples * kIn && at < size_t(n) * kIn) xin = X[at];
  };
  load(blockIdx.x);
  for (int p = tid; p < kNParams; p += kTrainThreads)
    reinterpret_cast<float*>(&s)[weight_slot(p)] = params[p];
  for (int g = blockIdx.x; g < groups; g += gridDim.x) {
    const int first = g * kPredictSamples, mine = min(kPredictSamples, n - first);
    if (tid < kPredictSamples * kIn) s.X[tid] = xin;
    __syncthreads();
    load(g + gridDim.x);
    {
      const int b = tid >> 4, j = (tid & 15) * 4;
      float h[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float z = s.b1[j + q];
#pragma unroll
        for (int i = 0; i < kIn; ++i) z = fmaf(s.X[b * kIn + i], s.W1[i * kHid + j + q], z);
        h[q] = tanhf(z);
      }
      *reinterpret_cast<float4*>(&s.H1[b * kPad + j]) = make_float4(h[0], h[1], h[2], h[3]);
    }
    __syncthreads();
    {
      const int b = 2 * warp, j = 2 * lane;
      const float* const ha = &s.H1[b * kPad];
      const float* const hb = ha + kPad;
      float z[2][2] = {{s.b2[j], s.b2[j + 1]}, {s.b2[j], s.b2[j + 1]}};
#pragma unroll
      for (int i = 0; i < kHid; i += 4) {
        const float4 a4 = *reinterpret_cast<const float4*>(ha + i);
        const float4 b4 = *reinterpret_cast<const float4*>(hb + i);
        const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 w = *reinterpret_cast<const float2*>(&s.W2[(i + q) * kPad + j]);
          z[0][0] = fmaf(av[q], w.x, z[0][0]);
          z[0][1] = fmaf(av[q], w.y, z[0][1]);
          z[1][0] = fmaf(bv[q], w.x, z[1][0]);
          z[1][1] = fmaf(bv[q], w.y, z[1][1]);
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q)
        *reinterpret_cast<float2*>(&s.H2[(b + q) * kPad + j]) =
            make_float2(tanhf(z[q][0]), tanhf(z[q][1]));
    }
    __syncthreads();
    if (tid < mine * kOut) {
      const int b = tid / kOut, k = tid % kOut;
      float y = s.b3[k];
#pragma unroll
      for (int j = 0; j < kHid; j += 4) {
        const float4 h = *reinterpret_cast<const float4*>(&s.H2[b * kPad + j]);
        const float4 w = *reinterpret_cast<const float4*>(&s.W3t[k * kHid + j]);
        y = fmaf(h.x, w.x, y);
        y = fmaf(h.y, w.y, y);
        y = fmaf(h.z, w.z, y);
        y = fmaf(h.w, w.w, y);
      }
      Y[size_t(first) * kOut + tid] = y;
    }
    // (the next group's writes to X and H1 come before its own barriers, after
    // every read of them; H2 is rewritten two barriers on)
  }
}

}  // namespace lbm

using namespace lbm;

struct lbm_mlp {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float* d_params = nullptr;
  float* d_m = nullptr;
  float* d_v = nullptr;
  float* d_scratch = nullptr;  // gradient / loss
  // predict: samples of a small call in mapped host memory, of a larger one on
  // the device; kept for the next call, at most kStageMost samples.  One call
  // at a time holds them (stage_mutex); one that another thread makes meanwhile
  // takes buffers of its own.
  std::mutex stage_mutex;
  float* h_stage = nullptr;    // kStageSamples x (4 + 3), page-locked
  float* d_stage = nullptr;    // stage_samples x (4 + 3)
  int stage_samples = 0;
  int sm_count = 0;
  int adam_t = 0;
  std::string err;
};

namespace {

lbm_status mfail(lbm_mlp* m, lbm_status st, const std::string& msg) {
  if (m) m->err = msg;
  return st;
}

#define LBM_MCUDA(m, call)                                                               \
  do {                                                                                   \
    cudaError_t e_ = (call);                                                             \
    if (e_ != cudaSuccess)                                                               \
      return mfail(m, LBM_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));   \
  } while (0)

struct MDeviceGuard {
  int prev = -1;
  explicit MDeviceGuard(int dev) {
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
  }
  ~MDeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

constexpr int kStageSamples = 4096;      // through mapped host memory up to here
constexpr int kStageMost = 1 << 18;      // largest device staging that is kept (7 MB)

// A temporary device buffer.
struct DevBuf {
  void* p = nullptr;
  ~DevBuf() { cudaFree(p); }
};

}  // namespace

extern "C" {

int lbm_mlp_num_params(void) { return kNParams; }

lbm_status lbm_mlp_create(int device, void* cuda_stream, lbm_mlp** out) {
  if (!out) return LBM_E_INVAL;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return LBM_E_CUDA;
  MDeviceGuard guard(device);
  lbm_mlp* m = new lbm_mlp();
  m->device = device;
  if (cuda_stream) {
    m->stream = static_cast<cudaStream_t>(cuda_stream);
  } else if (cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking) == cudaSuccess) {
    m->own_stream = true;
  } else {
    delete m;
    return LBM_E_CUDA;
  }
  bool ok = cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, device) ==
                cudaSuccess &&
            cudaMalloc(&m->d_params, kNParams * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->d_m, kNParams * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->d_v, kNParams * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->d_scratch, (kNParams + 1) * sizeof(float)) == cudaSuccess &&
            cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(sizeof(TrainSmem))) == cudaSuccess &&
            cudaMemsetAsync(m->d_params, 0, kNParams * sizeof(float), m->stream) == cudaSuccess &&
            cudaMemsetAsync(m->d_m, 0, kNParams * sizeof(float), m->stream) == cudaSuccess &&
            cudaMemsetAsync(m->d_v, 0, kNParams * sizeof(float), m->stream) == cudaSuccess &&
            cudaStreamSynchronize(m->stream) == cudaSuccess;
  if (!ok) {
    lbm_mlp_destroy(m);
    return LBM_E_NOMEM;
  }
  *out = m;
  return LBM_OK;
}

lbm_status lbm_mlp_destroy(lbm_mlp* m) {
  if (!m) return LBM_OK;
  MDeviceGuard guard(m->device);
  if (m->stream) cudaStreamSynchronize(m->stream);
  cudaFree(m->d_params);
  cudaFree(m->d_m);
  cudaFree(m->d_v);
  cudaFree(m->d_scratch);
  cudaFree(m->d_stage);
  if (m->h_stage) cudaFreeHost(m->h_stage);
  if (m->own_stream && m->stream) cudaStreamDestroy(m->stream);
  delete m;
  return LBM_OK;
}

const char* lbm_mlp_last_error(const lbm_mlp* m) { return m ? m->err.c_str() : ""; }

lbm_status lbm_mlp_set_params(lbm_mlp* m, const float* params) {
  if (!m || !params) return mfail(m, LBM_E_INVAL, "null argument");
  MDeviceGuard guard(m->device);
  LBM_MCUDA(m, cudaMemcpyAsync(m->d_params, params, kNParams * sizeof(float),
                               cudaMemcpyHostToDevice, m->stream));
  LBM_MCUDA(m, cudaMemsetAsync(m->d_m, 0, kNParams * sizeof(float), m->stream));
  LBM_MCUDA(m, cudaMemsetAsync(m->d_v, 0, kNParams * sizeof(float), m->stream));
  LBM_MCUDA(m, cudaStreamSynchronize(m->stream));
  m->adam_t = 0;
  return LBM_OK;
}

lbm_status lbm_mlp_get_params(lbm_mlp* m, float* params) {
  if (!m || !params) return mfail(m, LBM_E_INVAL, "null argument");
  MDeviceGuard guard(m->device);
  LBM_MCUDA(m, cudaMemcpyAsync(params, m->d_params, kNParams * sizeof(float),
                               cudaMemcpyDeviceToHost, m->stream));
  LBM_MCUDA(m, cudaStreamSynchronize(m->stream));
  return LBM_OK;
}

lbm_status lbm_mlp_gradient(lbm_mlp* m, const float* X, const float* Y, int n, float* grad,
                            float* loss) {
  if (!m || !X || !Y || !grad || n < 1 || n > kMaxBatch)
    return mfail(m, LBM_E_INVAL, "need 1 <= n <= 128 and non-null arrays");
  MDeviceGuard guard(m->device);
  DevBuf dx, dy;
  LBM_MCUDA(m, cudaMalloc(&dx.p, size_t(n) * kIn * sizeof(float)));
  LBM_MCUDA(m, cudaMalloc(&dy.p, size_t(n) * kOut * sizeof(float)));
  LBM_MCUDA(m, cudaMemcpyAsync(dx.p, X, size_t(n) * kIn * sizeof(float), cudaMemcpyHostToDevice,
                               m->stream));
  LBM_MCUDA(m, cudaMemcpyAsync(dy.p, Y, size_t(n) * kOut * sizeof(float), cudaMemcpyHostToDevice,
                               m->stream));
  mlp_train_kernel<<<kClusterCtas, kTrainThreads, sizeof(TrainSmem), m->stream>>>(
      m->d_params, m->d_m, m->d_v, static_cast<float*>(dx.p), static_cast<float*>(dy.p), n,
      nullptr, 1, n, 0.f, m->adam_t, 1, m->d_scratch, m->d_scratch + kNParams);
  LBM_MCUDA(m, cudaGetLastError());
  count_launches(1);
  LBM_MCUDA(m, cudaMemcpyAsync(grad, m->d_scratch, kNParams * sizeof(float),
                               cudaMemcpyDeviceToHost, m->stream));
  float l = 0.f;
  LBM_MCUDA(m, cudaMemcpyAsync(&l, m->d_scratch + kNParams, sizeof(float), cudaMemcpyDeviceToHost,
                               m->stream));
  LBM_MCUDA(m, cudaStreamSynchronize(m->stream));
  if (loss) *loss = l;
  return LBM_OK;
}

lbm_status lbm_mlp_train(lbm_mlp* m, const float* X, const float* Y, int n, const int* order,
                         int epochs, int batch, float lr, float* final_loss) {
  if (!m || !X || !Y || !order || n < 1 || epochs < 1 || batch < 1 || batch > kMaxBatch ||
      !(lr > 0.f))
    return mfail(m, LBM_E_INVAL, "need n, epochs >= 1, 1 <= batch <= 128, lr > 0");
  for (size_t k = 0; k < size_t(epochs) * n; ++k)
    if (order[k] < 0 || order[k] >= n) return mfail(m, LBM_E_INVAL, "order index out of range");
  MDeviceGuard guard(m->device);
  DevBuf dx, dy, dord;
  LBM_MCUDA(m, cudaMalloc(&dx.p, size_t(n) * kIn * sizeof(float)));
  LBM_MCUDA(m, cudaMalloc(&dy.p, size_t(n) * kOut * sizeof(float)));
  LBM_MCUDA(m, cudaMalloc(&dord.p, size_t(epochs) * n * sizeof(int)));
  LBM_MCUDA(m, cudaMemcpyAsync(dx.p, X, size_t(n) * kIn * sizeof(float), cudaMemcpyHostToDevice,
                               m->stream));
  LBM_MCUDA(m, cudaMemcpyAsync(dy.p, Y, size_t(n) * kOut * sizeof(float), cudaMemcpyHostToDevice,
                               m->stream));
  LBM_MCUDA(m, cudaMemcpyAsync(dord.p, order, size_t(epochs) * n * sizeof(int),
                               cudaMemcpyHostToDevice, m->stream));
  mlp_train_kernel<<<kClusterCtas, kTrainThreads, sizeof(TrainSmem), m->stream>>>(
      m->d_params, m->d_m, m->d_v, static_cast<float*>(dx.p), static_cast<float*>(dy.p), n,
      static_cast<int*>(dord.p), epochs, batch, lr, m->adam_t, 0, nullptr,
      m->d_scratch + kNParams);
  LBM_MCUDA(m, cudaGetLastError());
  count_launches(1);
  float l = 0.f;
  LBM_MCUDA(m, cudaMemcpyAsync(&l, m->d_scratch + kNParams, sizeof(float), cudaMemcpyDeviceToHost,
                               m->stream));
  LBM_MCUDA(m, cudaStreamSynchronize(m->stream));
  m->adam_t += epochs * ((n + batch - 1) / batch);
  if (final_loss) *final_loss = l;
  return LBM_OK;
}

lbm_status lbm_mlp_predict(lbm_mlp* m, const float* X, int n, float* Y) {
  if (!m || !X || !Y || n < 1) return mfail(m, LBM_E_INVAL, "bad argument");
  MDeviceGuard guard(m->device);
  const size_t xb = size_t(n) * kIn * sizeof(float), yb = size_t(n) * kOut * sizeof(float);
  const int groups = (n + kPredictSamples - 1) / kPredictSamples;
  const int grid = std::min(groups, 4 * m->sm_count);
  const std::unique_lock<std::mutex> stage(m->stage_mutex, std::try_to_lock);
  if (n <= kStageSamples && stage && !m->h_stage &&
      cudaMallocHost(&m->h_stage, size_t(kStageSamples) * (kIn + kOut) * sizeof(float)) !=
          cudaSuccess) {
    cudaGetLastError();  // (no page-locked memory to be had: through the device's)
    m->h_stage = nullptr;
  }
  if (n <= kStageSamples && stage && m->h_stage) {
    // small calls: the kernel reads and writes page-locked host memory, so the
    // call is one launch and one wait (256 samples: 58 -> 22 us against two
    // allocations, two copies and one CTA per 256 samples)
    float* const hx = m->h_stage;
    float* const hy = m->h_stage + size_t(kStageSamples) * kIn;
    std::memcpy(hx, X, xb);
    mlp_predict_kernel<<<grid, kTrainThreads, 0, m->stream>>>(m->d_params, hx, n, hy);
    LBM_MCUDA(m, cudaGetLastError());
    count_launches(1);
    LBM_MCUDA(m, cudaStreamSynchronize(m->stream));
    std::memcpy(Y, hy, yb);
    return LBM_OK;
  }
  DevBuf temp;  // beyond the staging that is kept, or beside a call that holds it
  float* dx = nullptr;
  if (n <= kStageMost && stage) {
    if (m->stage_samples < n) {
      cudaFree(m->d_stage);  // (waits for the work that reads it)
      m->d_stage = nullptr;
      m->stage_samples = 0;
      LBM_MCUDA(m, cudaMalloc(&m->d_stage, xb + yb));
      m->stage_samples = n;
    }
    dx = m->d_stage;
  } else {
    LBM_MCUDA(m, cudaMalloc(&temp.p, xb + yb));
    dx = static_cast<float*>(temp.p);
  }
  float* const dy = dx + size_t(n) * kIn;
  LBM_MCUDA(m, cudaMemcpyAsync(dx, X, xb, cudaMemcpyHostToDevice, m->stream));
  mlp_predict_kernel<<<grid, kTrainThreads, 0, m->stream>>>(m->d_params, dx, n, dy);
  LBM_MCUDA(m, cudaGetLastError());
  count_launches(1);
  LBM_MCUDA(m, cudaMemcpyAsync(Y, dy, yb, cudaMemcpyDeviceToHost, m->stream));
  LBM_MCUDA(m, cudaStreamSynchronize(m->stream));
  return LBM_OK;
}

}  // extern "C"
