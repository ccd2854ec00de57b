// Training of the troubled-cell indicator in FP32: loss and gradient of the
// network nin -> 64 -> 64 -> 1 (ReLU, sigmoid, weighted cross-entropy; layout of
// the flat weights in dg_mlp.cu) and Adam steps on shuffled mini-batches.
//
// A gradient is two launches. k_train_tile does the forward and backward passes
// of 32 samples per block entirely in shared memory and leaves the block's
// share of the gradient in its own row of a scratch matrix; k_train_reduce sums
// the rows in a fixed order and applies the Adam update. (As eight kernels with
// one thread per weight walking the batch serially, a 4096-sample step took
// 1.15 ms, 0.90 of it in the weight gradients; now 0.032 ms: 25 us in the tiles,
// latency-bound with one 8-warp block per SM, and 7 us in the sum over 128 rows.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

#include "dg_mlp.cuh"

namespace dgmhd {

namespace {

constexpr int HID = 64;
constexpr int TB = 32;        // samples per tile
constexpr int NTT = 256;      // threads per block
constexpr int SS = TB + 4;    // row stride of the [feature][sample] arrays (16-byte rows, no bank conflicts)
constexpr int KC = 128;       // inputs per pass over W1 and X
constexpr int WS = HID + 2;   // row stride of the transposed weights
constexpr int MAXBLK = 304;   // blocks (and scratch rows) at most: two per SM

struct TrainSmem {
  float w1t[KC][WS];    // W1 transposed, the current inputs
  float w2t[HID][WS];   // W2 transposed
  float w2[HID][WS];    // W2
  float xt[KC][SS];     // inputs [k][sample]
  float h1[HID][SS];    // relu(Z1)
  float d2[HID][SS];    // Z2, then delta2
  float d1[HID][SS];    // delta1
  float w3[HID], b1[HID], b2[HID];
  float d3[TB];
  float part[8][TB];    // partial sums of the output layer
};

// acc[o][s]: two units o0, o0 + 1 by four samples s0.. of sum_k Wt[k][o] A[k][s]
__device__ __forceinline__ void layer(const float (*Wt)[WS], const float (*A)[SS], int K, int o0, int s0,
                                      float (&acc)[2][4]) {
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const float2 wv = *reinterpret_cast<const float2*>(&Wt[k][o0]);
    const float4 x = *reinterpret_cast<const float4*>(&A[k][s0]);
    acc[0][0] = fmaf(x.x, wv.x, acc[0][0]);
    acc[0][1] = fmaf(x.y, wv.x, acc[0][1]);
    acc[0][2] = fmaf(x.z, wv.x, acc[0][2]);
    acc[0][3] = fmaf(x.w, wv.x, acc[0][3]);
    acc[1][0] = fmaf(x.x, wv.y, acc[1][0]);
    acc[1][1] = fmaf(x.y, wv.y, acc[1][1]);
    acc[1][2] = fmaf(x.z, wv.y, acc[1][2]);
    acc[1][3] = fmaf(x.w, wv.y, acc[1][3]);
  }
}

// g[i][j] = sum_s D[o + 16 i][s] A[k + 16 j][s]: the tile's share of a weight gradient
template <int NJ>
__device__ __forceinline__ void outer(const float (*D)[SS], const float (*A)[SS], int o, int k, float (&g)[4][NJ]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) g[i][j] = 0.f;
#pragma unroll 2
  for (int s = 0; s < TB; s += 4) {
    float4 d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = *reinterpret_cast<const float4*>(&D[o + 16 * i][s]);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const float4 a = *reinterpret_cast<const float4*>(&A[k + 16 * j][s]);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        g[i][j] = fmaf(d[i].w, a.w, fmaf(d[i].z, a.z, fmaf(d[i].y, a.y, fmaf(d[i].x, a.x, g[i][j]))));
    }
  }
}

// One block per tile of 32 samples (grid-stride): thread t owns units 2 (t % 32)
// and + 1 of samples 4 (t / 32).. in the layers, a 4 x NJ patch of the weight
// gradients. prob: the samples' probabilities (for the loss), or NULL.
__global__ void __launch_bounds__(NTT) k_train_tile(const float* __restrict__ X, int ldx, const uint8_t* __restrict__ y,
                                                    const int64_t* __restrict__ perm, int64_t off, int nb, int nin,
                                                    const float* __restrict__ theta, float pos_weight, float inv_n,
                                                    float* __restrict__ part, float* __restrict__ prob) {
  extern __shared__ __align__(16) unsigned char smraw[];
  TrainSmem& sm = *reinterpret_cast<TrainSmem*>(smraw);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const float* W1 = theta;
  const float* b1 = W1 + HID * nin;
  const float* W2 = b1 + HID;
  const float* b2 = W2 + HID * HID;
  const float* w3 = b2 + HID;
  const int np = HID * nin + HID + HID * HID + HID + HID + 1;
  float* gW1 = part + (size_t)blockIdx.x * np;
  float* gb1 = gW1 + HID * nin;
  float* gW2 = gb1 + HID;
  float* gb2 = gW2 + HID * HID;
  float* gw3 = gb2 + HID;
  for (int i = t; i < HID * HID; i += NTT) {
    const float x = W2[i];
    sm.w2[i / HID][i % HID] = x;
    sm.w2t[i % HID][i / HID] = x;
  }
  if (t < HID) {
    sm.w3[t] = w3[t];
    sm.b1[t] = b1[t];
    sm.b2[t] = b2[t];
  }
  const float b3 = w3[HID];
  const int o0 = 2 * lane, s0 = 4 * warp;
  const int nchunk = (nin + KC - 1) / KC;
  const int ntile = (nb + TB - 1) / TB;
  bool first = true;
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x, first = false) {
    const int base = tile * TB;
    const int cnt = min(TB, nb - base);
    auto row = [&](int s) { return perm ? perm[off + base + s] : off + base + s; };
    // inputs [kb, kb + kl) of the tile, transposed; rows past the end and absent samples are zero
    auto stage_x = [&](int kb) {
      for (int s = warp; s < TB; s += 8) {
        const float* xr = X + (s < cnt ? row(s) : 0) * ldx + kb;
        for (int k = lane; k < KC; k += 32) sm.xt[k][s] = (s < cnt && kb + k < nin) ? xr[k] : 0.f;
      }
    };
    auto stage_w1 = [&](int kb) {
      for (int o = warp; o < HID; o += 8)
        for (int k = lane; k < KC; k += 32) sm.w1t[k][o] = kb + k < nin ? W1[(size_t)o * nin + kb + k] : 0.f;
    };
    __syncthreads();  // the weights are staged; the previous tile's reads are done
    // layer 1
    float acc[2][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      acc[0][e] = sm.b1[o0];
      acc[1][e] = sm.b1[o0 + 1];
    }
    for (int c = 0; c < nchunk; ++c) {
      if (c) __syncthreads();
      stage_x(c * KC);
      if (first || nchunk > 1) stage_w1(c * KC);
      __syncthreads();
      layer(sm.w1t, sm.xt, min(KC, nin - c * KC), o0, s0, acc);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
      *reinterpret_cast<float4*>(&sm.h1[o0 + e][s0]) =
          make_float4(fmaxf(acc[e][0], 0.f), fmaxf(acc[e][1], 0.f), fmaxf(acc[e][2], 0.f), fmaxf(acc[e][3], 0.f));
    __syncthreads();
    // layer 2
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      acc[0][e] = sm.b2[o0];
      acc[1][e] = sm.b2[o0 + 1];
    }
    layer(sm.w2t, sm.h1, HID, o0, s0, acc);
#pragma unroll
    for (int e = 0; e < 2; ++e)
      *reinterpret_cast<float4*>(&sm.d2[o0 + e][s0]) = make_float4(acc[e][0], acc[e][1], acc[e][2], acc[e][3]);
    __syncthreads();
    // output layer: warp w sums units 8 w .. 8 w + 7 of sample `lane`
    {
      float z = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) z = fmaf(fmaxf(sm.d2[8 * warp + k][lane], 0.f), sm.w3[8 * warp + k], z);
      sm.part[warp][lane] = z;
    }
    __syncthreads();
    if (t < TB) {
      float z = b3;
#pragma unroll
      for (int k = 0; k < 8; ++k) z += sm.part[k][t];
      const float p = 1.f / (1.f + expf(-z));
      float d = 0.f;
      if (t < cnt) {
        const float yy = y[row(t)] ? 1.f : 0.f;
        // weighted BCE: -(pw y log p + (1-y) log(1-p)); dL/dz = pw y (p - 1) + (1 - y) p
        d = (pos_weight * yy * (p - 1.f) + (1.f - yy) * p) * inv_n;
        if (prob) prob[base + t] = p;
      }
      sm.d3[t] = d;
    }
    __syncthreads();
    // delta2 = d3 w3 (Z2 > 0) over Z2; the output layer's gradient and b2's on the way:
    // thread t: unit t / 4, samples 8 (t % 4)..
    {
      const int k = t >> 2, q = 8 * (t & 3);
      const float wk = sm.w3[k];
      float g3 = 0.f, g2 = 0.f, s3 = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float z = sm.d2[k][q + e], d = sm.d3[q + e];
        const float dd = z > 0.f ? d * wk : 0.f;
        g3 = fmaf(d, fmaxf(z, 0.f), g3);
        g2 += dd;
        s3 += d;
        sm.d2[k][q + e] = dd;
      }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        g3 += __shfl_xor_sync(0xffffffffu, g3, o);
        g2 += __shfl_xor_sync(0xffffffffu, g2, o);
        s3 += __shfl_xor_sync(0xffffffffu, s3, o);
      }
      if ((t & 3) == 0) {
        gw3[k] = first ? g3 : gw3[k] + g3;
        gb2[k] = first ? g2 : gb2[k] + g2;
        if (k == 0) gw3[HID] = first ? s3 : gw3[HID] + s3;
      }
    }
    __syncthreads();
    // delta1 = W2^T delta2 (Z1 > 0)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[0][e] = acc[1][e] = 0.f;
    layer(sm.w2, sm.d2, HID, o0, s0, acc);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float4 h = *reinterpret_cast<const float4*>(&sm.h1[o0 + e][s0]);
      float4 d = make_float4(h.x > 0.f ? acc[e][0] : 0.f, h.y > 0.f ? acc[e][1] : 0.f, h.z > 0.f ? acc[e][2] : 0.f,
                             h.w > 0.f ? acc[e][3] : 0.f);
      *reinterpret_cast<float4*>(&sm.d1[o0 + e][s0]) = d;
    }
    __syncthreads();
    // weight gradients: thread t: rows (t / 16) + 16 i, columns (t % 16) + 16 j
    const int go = t >> 4, gk = t & 15;
    {
      float g[4][4];
      outer<4>(sm.d2, sm.h1, go, gk, g);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float* q = gW2 + (go + 16 * i) * HID + gk + 16 * j;
          *q = first ? g[i][j] : *q + g[i][j];
        }
    }
    for (int c = nchunk - 1; c >= 0; --c) {  // the last inputs are still staged
      if (c < nchunk - 1) {
        __syncthreads();
        stage_x(c * KC);
        __syncthreads();
      }
      float g[4][KC / 16];
      outer<KC / 16>(sm.d1, sm.xt, go, gk, g);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < KC / 16; ++j) {
          const int k = c * KC + gk + 16 * j;
          if (k < nin) {
            float* q = gW1 + (size_t)(go + 16 * i) * nin + k;
            *q = first ? g[i][j] : *q + g[i][j];
          }
        }
    }
    if (t < HID) {
      float s = 0.f;
#pragma unroll
      for (int e = 0; e < TB; ++e) s += sm.d1[t][e];
      gb1[t] = first ? s : gb1[t] + s;
    }
  }
}

struct Adam {
  float *th, *m, *v;  // NULL th: the gradient is written to `grad`
  float lr, c1, c2;
};

// Sums the nblk rows of the scratch matrix in a fixed order (eight interleaved
// partial sums per weight) into the gradient, or straight into an Adam step
// (beta 0.9 / 0.999, eps 1e-8). Blocks past the weights sum the loss.
__global__ void __launch_bounds__(256) k_train_reduce(const float* __restrict__ part, int nblk, int np, int nred,
                                                      float* __restrict__ grad, Adam a,
                                                      const float* __restrict__ prob, const uint8_t* __restrict__ y,
                                                      const int64_t* __restrict__ perm, int64_t off, int nb,
                                                      float pos_weight, float inv_n, double* __restrict__ loss) {
  __shared__ float red[8][32];
  __shared__ double redd[8];
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  if ((int)blockIdx.x < nred) {
    const int i = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (i < np)
      for (int b = q; b < nblk; b += 8) s += part[(size_t)b * np + i];
    red[q][lane] = s;
    __syncthreads();
    if (q || i >= np) return;
    float g = red[0][lane];
#pragma unroll
    for (int k = 1; k < 8; ++k) g += red[k][lane];
    if (!a.th) {
      grad[i] = g;
      return;
    }
    const float mi = 0.9f * a.m[i] + (1.f - 0.9f) * g;
    const float vi = 0.999f * a.v[i] + (1.f - 0.999f) * g * g;
    a.m[i] = mi;
    a.v[i] = vi;
    a.th[i] -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + 1e-8f);
    return;
  }
  const int s = (blockIdx.x - nred) * 256 + threadIdx.x;
  double l = 0.0;
  if (s < nb) {
    const bool yy = y[perm ? perm[off + s] : off + s] != 0;
    const double p = (double)prob[s];
    l = yy ? -(double)pos_weight * log(p + 1e-12) : -log(1.0 - p + 1e-12);
    l *= (double)inv_n;
  }
  for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if (lane == 0) redd[q] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) l += redd[k];
    atomicAdd(loss, l);
  }
}

// loss (nullable) += the mean weighted loss of the nb samples; the gradient
// into grad, or an Adam step
int gradient(const float* X, int ldx, const uint8_t* y, const int64_t* perm, int64_t off, int nb, int nin,
             const float* theta, float* grad, const Adam& a, double* loss, float pos_weight, float norm_n,
             void* scratch, cudaStream_t st) {
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(k_train_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)) !=
        cudaSuccess)
      return -3;
    attr = true;
  }
  const int np = mlp_n_params(nin);
  const int nblk = std::min((nb + TB - 1) / TB, MAXBLK);
  float* part = static_cast<float*>(scratch);
  float* prob = loss ? part + (size_t)nblk * np : nullptr;
  const float inv_n = 1.f / norm_n;
  k_train_tile<<<nblk, NTT, sizeof(TrainSmem), st>>>(X, ldx, y, perm, off, nb, nin, theta, pos_weight, inv_n, part,
                                                     prob);
  const int nred = (np + 31) / 32;
  k_train_reduce<<<nred + (loss ? (nb + 255) / 256 : 0), 256, 0, st>>>(part, nblk, np, nred, grad, a, prob, y, perm,
                                                                      off, nb, pos_weight, inv_n, loss);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace

size_t mlp_scratch_bytes(int nb, int nin) {
  const size_t nblk = (size_t)std::min((nb + TB - 1) / TB, MAXBLK);
  return (nblk * mlp_n_params(nin) + nb) * sizeof(float);
}

int mlp_loss_grad_dev(const float* X, int ldx, const uint8_t* y, int nb, int nin, const float* theta, float* grad,
                      double* loss, float pos_weight, void* scratch, cudaStream_t st) {
  return gradient(X, ldx, y, nullptr, 0, nb, nin, theta, grad, Adam{}, loss, pos_weight, (float)nb, scratch, st);
}

int mlp_train_dev(const float* X, int ldx, const uint8_t* y, int64_t n, int nin, float* theta, int epochs,
                  int batch, float lr, float pos_weight, uint64_t seed, double* last_loss, cudaStream_t st) {
  const int np = mlp_n_params(nin);
  // one allocation: shuffle (8-byte elements first), loss, Adam moments, scratch
  const size_t bytes = n * sizeof(int64_t) + sizeof(double) + 2 * (size_t)np * sizeof(float) +
                       mlp_scratch_bytes(batch, nin);
  unsigned char* mem = nullptr;
  if (cudaMalloc(&mem, bytes) != cudaSuccess) return -3;
  int64_t* perm = reinterpret_cast<int64_t*>(mem);
  double* dloss = reinterpret_cast<double*>(perm + n);
  float* m = reinterpret_cast<float*>(dloss + 1);
  float* v = m + np;
  void* scratch = v + np;
  int e = 0;
  if (cudaMemsetAsync(m, 0, 2 * (size_t)np * sizeof(float), st) != cudaSuccess) e = -3;
  std::vector<int64_t> hp(n);
  for (int64_t i = 0; i < n; ++i) hp[i] = i;
  std::mt19937_64 rng(seed);
  int t = 0;
  for (int ep = 0; ep < epochs && !e; ++ep) {
    // (the previous epoch's kernels may still run: the copy below follows them on the stream)
    std::shuffle(hp.begin(), hp.end(), rng);
    if (cudaMemcpyAsync(perm, hp.data(), n * sizeof(int64_t), cudaMemcpyHostToDevice, st)) e = -3;
    double* loss = ep == epochs - 1 ? dloss : nullptr;
    if (loss) cudaMemsetAsync(dloss, 0, sizeof(double), st);
    for (int64_t off = 0; off + batch <= n && !e; off += batch) {
      ++t;
      const float c1 = 1.f - powf(0.9f, (float)t), c2 = 1.f - powf(0.999f, (float)t);
      e = gradient(X, ldx, y, perm, off, batch, nin, theta, nullptr, Adam{theta, m, v, lr, c1, c2}, loss, pos_weight,
                   (float)batch, scratch, st);
    }
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) e = -3;
  if (!e && last_loss) {
    double l = 0.0;
    cudaMemcpy(&l, dloss, sizeof(double), cudaMemcpyDeviceToHost);
    const int64_t nbat = n / batch;
    *last_loss = nbat ? l / (double)nbat : 0.0;
  }
  cudaFree(mem);
  return e;
}

}  // namespace dgmhd
