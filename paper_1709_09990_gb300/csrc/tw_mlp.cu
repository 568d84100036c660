// The 12-32-1 ReLU network that proposes a starting bound for the k sweep.
// The paper has no learned component; the proposal only changes which decide
// runs are made first, and the answer is always certified by decide runs.
//
// Parameters (449 fp32): W1 [32][12] row-major, b1[32], W2[32], b2.
//   z = W1 x + b1, h = relu(z), yhat = W2 . h + b2
//   loss = (1/B) sum_b (yhat_b - y_b)^2, g_b = 2 (yhat_b - y_b) / B
//   dW2 = sum_b g_b h_b, db2 = sum_b g_b, dz_b = g_b W2 * [z_b > 0],
//   dW1 = sum_b dz_b x_b^T, db1 = sum_b dz_b
// Gradients are reduced in a fixed order (per 128-sample tile, then per block,
// then over blocks), so results are deterministic.  Adam: Kingma & Ba (2015).
#include <cuda_runtime.h>

#include "tw_internal.h"

namespace tw {
namespace {

constexpr int kIn = 12;
constexpr int kHid = 32;
constexpr int kParams = kHid * kIn + kHid + kHid + 1;  // 449
constexpr int kTile = 128;

struct TileScratch {
  float x[kTile][kIn];
  float h[kTile][kHid];
  float dz[kTile][kHid];
  float g[kTile];
  float sq[kTile];
};

// Forward + backward of samples [s0, s0 + cnt) (cnt <= kTile) into the tile
// scratch; idx (or nullptr = identity) maps tile rows to sample indices.
__device__ void tile_forward_backward(const float* __restrict__ P, const float* __restrict__ x,
                                      const float* __restrict__ y, const int32_t* idx, int s0, int cnt,
                                      float inv_b, TileScratch& T) {
  for (int t = threadIdx.x; t < kTile; t += blockDim.x) {
    if (t >= cnt) {
      T.g[t] = 0.f;
      T.sq[t] = 0.f;
      for (int j = 0; j < kHid; ++j) {
        T.h[t][j] = 0.f;
        T.dz[t][j] = 0.f;
      }
      for (int i = 0; i < kIn; ++i) T.x[t][i] = 0.f;
      continue;
    }
    const int s = idx ? idx[s0 + t] : (s0 + t);
    float xi[kIn];
    for (int i = 0; i < kIn; ++i) {
      xi[i] = x[(size_t)s * kIn + i];
      T.x[t][i] = xi[i];
    }
    const float* W1 = P;
    const float* b1 = P + kHid * kIn;
    const float* W2 = b1 + kHid;
    const float b2 = W2[kHid];
    float out = b2;
    float z[kHid];
    for (int j = 0; j < kHid; ++j) {
      float a = b1[j];
      for (int i = 0; i < kIn; ++i) a = fmaf(W1[j * kIn + i], xi[i], a);
      z[j] = a;
      const float hj = a > 0.f ? a : 0.f;
      T.h[t][j] = hj;
      out = fmaf(W2[j], hj, out);
    }
    const float diff = out - y[s];
    const float g = 2.f * diff * inv_b;
    T.g[t] = g;
    T.sq[t] = diff * diff;
    for (int j = 0; j < kHid; ++j) T.dz[t][j] = z[j] > 0.f ? g * W2[j] : 0.f;
  }
  __syncthreads();
}

// acc[p] += gradient contribution of the tile for parameter p (fixed order).
__device__ void tile_accumulate(const TileScratch& T, float* acc) {
  for (int p = threadIdx.x; p < kParams; p += blockDim.x) {
    float a = 0.f;
    if (p < kHid * kIn) {
      const int j = p / kIn, i = p % kIn;
      for (int t = 0; t < kTile; ++t) a = fmaf(T.dz[t][j], T.x[t][i], a);
    } else if (p < kHid * kIn + kHid) {
      const int j = p - kHid * kIn;
      for (int t = 0; t < kTile; ++t) a += T.dz[t][j];
    } else if (p < kHid * kIn + 2 * kHid) {
      const int j = p - kHid * kIn - kHid;
      for (int t = 0; t < kTile; ++t) a = fmaf(T.g[t], T.h[t][j], a);
    } else {
      for (int t = 0; t < kTile; ++t) a += T.g[t];
    }
    acc[p] += a;
  }
  __syncthreads();
}

__global__ void mlp_forward_kernel(const float* __restrict__ P, const float* __restrict__ x, int batch,
                                   float* __restrict__ yhat) {
  __shared__ float sP[kParams];
  for (int p = threadIdx.x; p < kParams; p += blockDim.x) sP[p] = P[p];
  __syncthreads();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  float xi[kIn];
  for (int i = 0; i < kIn; ++i) xi[i] = x[(size_t)b * kIn + i];
  const float* b1 = sP + kHid * kIn;
  const float* W2 = b1 + kHid;
  float out = W2[kHid];
  for (int j = 0; j < kHid; ++j) {
    float a = b1[j];
    for (int i = 0; i < kIn; ++i) a = fmaf(sP[j * kIn + i], xi[i], a);
    out = fmaf(W2[j], a > 0.f ? a : 0.f, out);
  }
  yhat[b] = out;
}

// Stage 1: block blk reduces samples [blk*per, (blk+1)*per) into partial[blk].
__global__ void mlp_grad_partial_kernel(const float* __restrict__ P, const float* __restrict__ x,
                                        const float* __restrict__ y, int batch, int per, float* partial) {
  __shared__ float sP[kParams];
  __shared__ float sAcc[kParams];
  __shared__ TileScratch T;
  for (int p = threadIdx.x; p < kParams; p += blockDim.x) {
    sP[p] = P[p];
    sAcc[p] = 0.f;
  }
  __syncthreads();
  const float inv_b = 1.f / (float)batch;
  const int lo = blockIdx.x * per;
  const int hi = min(batch, lo + per);
  for (int s0 = lo; s0 < hi; s0 += kTile) {
    tile_forward_backward(sP, x, y, nullptr, s0, min(kTile, hi - s0), inv_b, T);
    tile_accumulate(T, sAcc);
  }
  for (int p = threadIdx.x; p < kParams; p += blockDim.x) partial[(size_t)blockIdx.x * kParams + p] = sAcc[p];
}

// Stage 2: grad[p] = sum over blocks of partial[blk][p], in block order.
__global__ void mlp_grad_final_kernel(const float* __restrict__ partial, int blocks, float* __restrict__ grad) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kParams) return;
  float a = 0.f;
  for (int b = 0; b < blocks; ++b) a += partial[(size_t)b * kParams + p];
  grad[p] = a;
}

__device__ __forceinline__ void adam_update(float& p, float g, float& m, float& v, float lr, float beta1, float beta2,
                                            float eps, float c1, float c2) {
  m = beta1 * m + (1.f - beta1) * g;
  v = beta2 * v + (1.f - beta2) * g * g;
  const float mhat = m / c1;
  const float vhat = v / c2;
  p -= lr * mhat / (sqrtf(vhat) + eps);
}

__global__ void mlp_adam_kernel(float* P, const float* __restrict__ G, float* M, float* V, float lr, float beta1,
                                float beta2, float eps, float c1, float c2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kParams) return;
  float pp = P[p], m = M[p], v = V[p];
  adam_update(pp, G[p], m, v, lr, beta1, beta2, eps, c1, c2);
  P[p] = pp;
  M[p] = m;
  V[p] = v;
}

// ---- training ---------------------------------------------------------------
//
// The whole run in one CTA: for each epoch and minibatch, forward, backward
// (fixed-order reduction) and an Adam step, all on chip.  A step is a chain: the
// next one needs its weights, so its latency is the kernel's time (2000 samples,
// 60 epochs, minibatches of 256: 480 steps in 2.48 ms, 5.2 us a step at 45% of
// the issue slots; 8.6 ms with one thread per sample and one per parameter,
// whose sums read two words from shared memory per multiply-add).  Up to two
// tiles of 128 samples are worked on at once:
//  F. four lanes per sample, 8 hidden units each, two samples per lane, so a
//     weight read serves two samples (four, with half the threads, is 10%
//     slower); the output sum runs through the four lanes in the order of the
//     units.
//  A. per tile, 48 lanes hold 2 x 4 blocks of the W1 gradient (two shared-memory
//     reads for 8 multiply-adds), one warp the other gradients, one lane the
//     loss; every sum runs over the tile's samples in order.
//  U. thread p owns parameter p and its Adam moments in registers.
// The next pass's samples are fetched during A.  Every sum has the order of
// tile_accumulate: sample by sample within a tile, then tile by tile.
constexpr int kTrainThreads = 512;
constexpr int kRow = kHid + 4;               // padded rows of h and dz
constexpr int kQuarter = kHid / 4 * kIn + 8;  // padded 8-unit blocks of W1
struct TrainShared {
  float w1[4 * kQuarter];
  float b1[kHid], w2[kHid], b2[4];
  float x[2 * kTile * kIn];
  float h[2 * kTile * kRow];
  float dz[2 * kTile * kRow];
  float g[2 * kTile];
  float sq[2 * kTile];
  float part[2][kParams + 1];  // per tile: the gradient sums, then the loss sum
};

// Sample idx's features (float4 loads when x is 16-byte aligned).
__device__ __forceinline__ void load_features(const float* __restrict__ x, int idx, bool aligned, float (&xi)[kIn]) {
  const float* r = x + (size_t)idx * kIn;
  if (aligned) {
#pragma unroll
    for (int i = 0; i < kIn; i += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(r + i));
      xi[i] = v.x;
      xi[i + 1] = v.y;
      xi[i + 2] = v.z;
      xi[i + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < kIn; ++i) xi[i] = __ldg(r + i);
  }
}

__global__ void __launch_bounds__(kTrainThreads) mlp_train_kernel(float* P, float* M, float* V,
                                                                 const float* __restrict__ x,
                                                                 const float* __restrict__ y, int batch_total,
                                                                 int minibatch, int epochs,
                                                                 const int32_t* __restrict__ perm, float lr,
                                                                 float* loss_out) {
  extern __shared__ __align__(16) unsigned char train_smem[];
  TrainShared& T = *reinterpret_cast<TrainShared*>(train_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool aligned = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
  const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
  // U: this thread's parameter and where F reads it
  const bool owner = tid < kParams;
  float prm = owner ? P[tid] : 0.f, mom = owner ? M[tid] : 0.f, var = owner ? V[tid] : 0.f, acc = 0.f;
  float* place = tid < kHid * kIn
                     ? &T.w1[(tid / kIn / 8) * kQuarter + (tid / kIn % 8) * kIn + tid % kIn]
                     : (tid < kHid * kIn + kHid ? &T.b1[tid - kHid * kIn]
                                                : (tid < kHid * kIn + 2 * kHid ? &T.w2[tid - kHid * kIn - kHid] : T.b2));
  if (owner) *place = prm;
  // F: this lane's units 8q .. 8q+7 and samples t0, t0 + 8 of the pass
  const int q = lane & 3;
  const int t0 = warp * 16 + (lane >> 2);
  // The passes in order; `at` = first entry of perm, `cnt` = samples (0: none left).
  // A pass's sample numbers are fetched two passes ahead and its features one
  // ahead (fetching both one ahead is 6% slower: A waits for the numbers).
  struct Pass {
    int e, mb0, s0, cnt;
    size_t at;
  };
  auto measure = [&](Pass& p) {
    const int mb = min(minibatch, batch_total - p.mb0);
    p.cnt = p.e < epochs ? min(2 * kTile, mb - p.s0) : 0;
    p.at = (size_t)p.e * batch_total + p.mb0 + p.s0;
  };
  auto advance = [&](Pass& p) {
    const int mb = min(minibatch, batch_total - p.mb0);
    p.s0 += 2 * kTile;
    if (p.s0 >= mb) {
      p.s0 = 0;
      p.mb0 += mb;
      if (p.mb0 >= batch_total) {
        p.mb0 = 0;
        ++p.e;
      }
    }
    measure(p);
  };
  float xs[2][kIn], ys[2];
  int num[2];
  auto fetch_numbers = [&](const Pass& p) {
#pragma unroll
    for (int u = 0; u < 2; ++u) num[u] = t0 + 8 * u < p.cnt ? __ldg(&perm[p.at + t0 + 8 * u]) : -1;
  };
  auto fetch_features = [&]() {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (num[u] >= 0) {
        load_features(x, num[u], aligned, xs[u]);
        ys[u] = __ldg(&y[num[u]]);
      } else {
        ys[u] = 0.f;
#pragma unroll
        for (int i = 0; i < kIn; ++i) xs[u][i] = 0.f;
      }
    }
  };
  Pass ahead{0, 0, 0, 0, 0};
  measure(ahead);
  fetch_numbers(ahead);
  fetch_features();
  advance(ahead);
  fetch_numbers(ahead);
  float b1t = 1.f, b2t = 1.f;
  for (int e = 0; e < epochs; ++e) {
    float loss = 0.f;  // (thread kParams sums it)
    for (int mb0 = 0; mb0 < batch_total; mb0 += minibatch) {
      const int mb = min(minibatch, batch_total - mb0);
      const float inv_b = 1.f / (float)mb;
      for (int s0 = 0; s0 < mb; s0 += 2 * kTile) {
        const int cnt = min(2 * kTile, mb - s0);
        __syncthreads();  // the weights are in place, the last pass's tiles are free
        // ---- F
        float z[2][8];
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          const float b = T.b1[8 * q + jj];
          z[0][jj] = z[1][jj] = b;
          const float4* wr = reinterpret_cast<const float4*>(&T.w1[q * kQuarter + jj * kIn]);
#pragma unroll
          for (int i4 = 0; i4 < kIn / 4; ++i4) {
            const float4 wv = wr[i4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              z[u][jj] = fmaf(wv.x, xs[u][4 * i4], z[u][jj]);
              z[u][jj] = fmaf(wv.y, xs[u][4 * i4 + 1], z[u][jj]);
              z[u][jj] = fmaf(wv.z, xs[u][4 * i4 + 2], z[u][jj]);
              z[u][jj] = fmaf(wv.w, xs[u][4 * i4 + 3], z[u][jj]);
            }
          }
        }
        float w2[8];
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) w2[jj] = T.w2[8 * q + jj];
        float out[2] = {T.b2[0], T.b2[0]};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
#pragma unroll
          for (int jj = 0; jj < 8; ++jj)
#pragma unroll
            for (int u = 0; u < 2; ++u) out[u] = fmaf(w2[jj], z[u][jj] > 0.f ? z[u][jj] : 0.f, out[u]);
#pragma unroll
          for (int u = 0; u < 2; ++u) out[u] = __shfl_sync(0xffffffffu, out[u], (lane & ~3) | r);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int t = t0 + 8 * u;
          if (t >= cnt) continue;  // (A reads the pass's samples only)
          const float diff = out[u] - ys[u];
          const float g = 2.f * diff * inv_b;
          float4* hr = reinterpret_cast<float4*>(&T.h[t * kRow + 8 * q]);
          float4* dr = reinterpret_cast<float4*>(&T.dz[t * kRow + 8 * q]);
#pragma unroll
          for (int j4 = 0; j4 < 2; ++j4) {
            const float* zz = &z[u][4 * j4];
            const float* ww = &w2[4 * j4];
            hr[j4] = make_float4(zz[0] > 0.f ? zz[0] : 0.f, zz[1] > 0.f ? zz[1] : 0.f, zz[2] > 0.f ? zz[2] : 0.f,
                                 zz[3] > 0.f ? zz[3] : 0.f);
            dr[j4] = make_float4(zz[0] > 0.f ? g * ww[0] : 0.f, zz[1] > 0.f ? g * ww[1] : 0.f,
                                 zz[2] > 0.f ? g * ww[2] : 0.f, zz[3] > 0.f ? g * ww[3] : 0.f);
          }
          if (q < 3) {
            reinterpret_cast<float4*>(&T.x[t * kIn])[q] =
                q == 0 ? make_float4(xs[u][0], xs[u][1], xs[u][2], xs[u][3])
                       : (q == 1 ? make_float4(xs[u][4], xs[u][5], xs[u][6], xs[u][7])
                                 : make_float4(xs[u][8], xs[u][9], xs[u][10], xs[u][11]));
          } else {
            T.g[t] = g;
            T.sq[t] = diff * diff;
          }
        }
        __syncthreads();
        fetch_features();  // of the next pass
        advance(ahead);
        fetch_numbers(ahead);
        // ---- A: warps 0-1, 4, 6 work on the first tile, 2-3, 5, 7 on the second
        const int tile = warp < 4 ? warp >> 1 : warp & 1;
        const int n_t = min(kTile, cnt - tile * kTile);
        if (warp < 4) {
          const int c = (warp & 1) * 32 + lane;
          if (c < 48 && n_t > 0) {
            const int jg = c & 15, ig = c >> 4;
            const float* dz = &T.dz[tile * kTile * kRow + 2 * jg];
            const float* xr = &T.x[tile * kTile * kIn + 4 * ig];
            float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 8
            for (int t = 0; t < n_t; ++t) {
              const float2 d = *reinterpret_cast<const float2*>(dz + t * kRow);
              const float4 v = *reinterpret_cast<const float4*>(xr + t * kIn);
              s[0][0] = fmaf(d.x, v.x, s[0][0]);
              s[0][1] = fmaf(d.x, v.y, s[0][1]);
              s[0][2] = fmaf(d.x, v.z, s[0][2]);
              s[0][3] = fmaf(d.x, v.w, s[0][3]);
              s[1][0] = fmaf(d.y, v.x, s[1][0]);
              s[1][1] = fmaf(d.y, v.y, s[1][1]);
              s[1][2] = fmaf(d.y, v.z, s[1][2]);
              s[1][3] = fmaf(d.y, v.w, s[1][3]);
            }
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
              for (int b = 0; b < 4; ++b) T.part[tile][(2 * jg + a) * kIn + 4 * ig + b] = s[a][b];
          }
        } else if (warp < 6) {
          float sb1 = 0.f, sw2 = 0.f, sb2 = 0.f;
#pragma unroll 8
          for (int t = 0; t < n_t; ++t) {
            const int row = tile * kTile + t;
            const float g = T.g[row];
            sb1 += T.dz[row * kRow + lane];
            sw2 = fmaf(g, T.h[row * kRow + lane], sw2);
            sb2 += g;
          }
          T.part[tile][kHid * kIn + lane] = sb1;
          T.part[tile][kHid * kIn + kHid + lane] = sw2;
          if (lane == 0) T.part[tile][kHid * kIn + 2 * kHid] = sb2;
        } else if (warp < 8 && lane == 0) {
          float l = 0.f;
#pragma unroll 8
          for (int t = 0; t < n_t; ++t) l += T.sq[tile * kTile + t];
          T.part[tile][kParams] = l;
        }
        __syncthreads();
        // ---- U
        if (tid <= kParams) {
          float& sum = owner ? acc : loss;
          sum += T.part[0][tid];
          if (cnt > kTile) sum += T.part[1][tid];
        }
      }
      b1t *= beta1;
      b2t *= beta2;
      if (owner) {
        adam_update(prm, acc, mom, var, lr, beta1, beta2, eps, 1.f - b1t, 1.f - b2t);
        *place = prm;
        acc = 0.f;
      }
    }
    if (tid == kParams && loss_out) loss_out[e] = loss / (float)batch_total;
  }
  if (owner) {
    P[tid] = prm;
    M[tid] = mom;
    V[tid] = var;
  }
}

}  // namespace

cudaError_t launch_mlp_forward(const float* params, const float* x, int batch, float* yhat, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  mlp_forward_kernel<<<(batch + 255) / 256, 256, 0, s>>>(params, x, batch, yhat);
  return cudaGetLastError();
}

cudaError_t launch_mlp_grad(const float* params, const float* x, const float* y, int batch, float* grad,
                            float* partial, int partial_blocks, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  const int per = ((batch + partial_blocks - 1) / partial_blocks + kTile - 1) / kTile * kTile;
  const int blocks = (batch + per - 1) / per;
  mlp_grad_partial_kernel<<<blocks, 256, 0, s>>>(params, x, y, batch, per, partial);
  mlp_grad_final_kernel<<<(kParams + 255) / 256, 256, 0, s>>>(partial, blocks, grad);
  return cudaGetLastError();
}

cudaError_t launch_mlp_adam(float* params, const float* grad, float* m, float* v, int t, float lr, float beta1,
                            float beta2, float eps, cudaStream_t s) {
  const float c1 = 1.f - powf(beta1, (float)t);
  const float c2 = 1.f - powf(beta2, (float)t);
  mlp_adam_kernel<<<(kParams + 255) / 256, 256, 0, s>>>(params, grad, m, v, lr, beta1, beta2, eps, c1, c2);
  return cudaGetLastError();
}

cudaError_t launch_mlp_train(float* params, float* m, float* v, const float* x, const float* y, int batch_total,
                             int minibatch, int epochs, const int32_t* perm, float lr, float* loss_out,
                             cudaStream_t s) {
  if (batch_total <= 0 || epochs <= 0) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(TrainShared));
  if (e != cudaSuccess) return e;
  mlp_train_kernel<<<1, kTrainThreads, sizeof(TrainShared), s>>>(params, m, v, x, y, batch_total, minibatch, epochs,
                                                                 perm, lr, loss_out);
  return cudaGetLastError();
}

}  // namespace tw
