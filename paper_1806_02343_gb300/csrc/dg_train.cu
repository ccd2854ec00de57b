// Training of the troubled-cell indicator in FP32: loss and gradient of the
// network nin -> 64 -> 64 -> 1 (ReLU, sigmoid, weighted cross-entropy; layout of
// the flat weights in dg_mlp.cu) and Adam steps on shuffled mini-batches.
//
// A gradient is two launches. k_train_pass does the forward and backward passes of
// 32 samples per block in shared memory and writes the activations and deltas as
// [unit][sample]; k_train_grad sums each weight's gradient over the samples, one
// thread per weight in the order of the samples, and applies the Adam update. Every
// sum is one chain in a fixed order -- inputs, units and samples ascending -- because
// Adam divides a gradient by its own size: where a weight's gradient cancels, the
// rounding of its sum decides the step, and a training of 32 steps from tile-wise
// sums ended 4e-5 away. (As eight kernels whose weight gradients read both factors
// from memory for every sample, a 4096-sample step took 1.15 ms; now 0.050 ms: 23 us
// in the passes, latency-bound with one 8-warp block per SM, 27 us in the chains.)
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
constexpr int MAXBLK = 304;   // blocks of the passes at most: two per SM
constexpr int GO = 4, GK = 16, GS = 256;  // a gradient block: GO x GK weights, chunks of GS samples
// samples per pair of launches: more than a mini-batch has, so that one pair is the
// rule; a gradient of more samples keeps scratch for this many (0.4 GB at 110 inputs)
// and its sums go on from pair to pair
constexpr int PART = 1 << 18;

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

// Scratch of nb samples: rows of ld = nb rounded up to a multiple of 4
struct Scratch {
  float *h1, *h2, *d1, *d2, *d3;  // [64][ld] four times, [ld]
  float* x;                       // [nin][ld]
  float* prob;                    // [nb]
  int ld;
  __host__ __device__ Scratch(float* s, int nb, int nin) : ld((nb + 3) / 4 * 4) {
    h1 = s;
    h2 = h1 + (size_t)HID * ld;
    d1 = h2 + (size_t)HID * ld;
    d2 = d1 + (size_t)HID * ld;
    d3 = d2 + (size_t)HID * ld;
    x = d3 + ld;
    prob = x + (size_t)nin * ld;
  }
  static size_t floats(int nb, int nin) { return (size_t)((nb + 3) / 4 * 4) * (4 * HID + 2 + nin); }
};

// One block per tile of 32 samples (grid-stride): thread t owns units 2 (t % 32)
// and + 1 of samples 4 (t / 32).. in the layers. want_prob: also the samples'
// probabilities (for the loss).
__global__ void __launch_bounds__(NTT) k_train_pass(const float* __restrict__ X, int ldx, const uint8_t* __restrict__ y,
                                                    const int64_t* __restrict__ perm, int64_t off, int nb, int nin,
                                                    const float* __restrict__ theta, float pos_weight, float inv_n,
                                                    Scratch out, bool want_prob) {
  extern __shared__ __align__(16) unsigned char smraw[];
  TrainSmem& sm = *reinterpret_cast<TrainSmem*>(smraw);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const float* W1 = theta;
  const float* b1 = W1 + HID * nin;
  const float* W2 = b1 + HID;
  const float* b2 = W2 + HID * HID;
  const float* w3 = b2 + HID;
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
    // a warp's lanes write the tile's samples of one unit
    auto put = [&](float* dst, const float (*src)[SS], int n, bool relu) {
      if (lane < cnt)
        for (int k = warp; k < n; k += 8) {
          const float x = src[k][lane];
          dst[(size_t)k * out.ld + base + lane] = relu ? fmaxf(x, 0.f) : x;
        }
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
      const int kl = min(KC, nin - c * KC);
      layer(sm.w1t, sm.xt, kl, o0, s0, acc);
      put(out.x + (size_t)c * KC * out.ld, sm.xt, kl, false);
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
    // output layer: one chain per sample
    if (t < TB) {
      float z = b3;
#pragma unroll 16
      for (int k = 0; k < HID; ++k) z = fmaf(fmaxf(sm.d2[k][t], 0.f), sm.w3[k], z);
      const float p = 1.f / (1.f + expf(-z));
      float d = 0.f;
      if (t < cnt) {
        const float yy = y[row(t)] ? 1.f : 0.f;
        // weighted BCE: -(pw y log p + (1-y) log(1-p)); dL/dz = pw y (p - 1) + (1 - y) p
        d = (pos_weight * yy * (p - 1.f) + (1.f - yy) * p) * inv_n;
        if (want_prob) out.prob[base + t] = p;
        out.d3[base + t] = d;
      }
      sm.d3[t] = d;
    }
    __syncthreads();
    put(out.h1, sm.h1, HID, false);
    put(out.h2, sm.d2, HID, true);
    __syncthreads();
    // delta2 = d3 w3 (Z2 > 0) over Z2
    for (int i = t; i < HID * TB; i += NTT) {
      const int k = i / TB, q = i % TB;
      sm.d2[k][q] = sm.d2[k][q] > 0.f ? sm.d3[q] * sm.w3[k] : 0.f;
    }
    __syncthreads();
    put(out.d2, sm.d2, HID, false);
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
    put(out.d1, sm.d1, HID, false);
  }
}

struct Adam {
  float *th, *m, *v;  // NULL th: the gradient is written to `grad`
  float lr, b1, b2, eps, c1, c2;
};

// Gradients of one layer: weight (o, k) of the patch of GO x GK weights is a chain
// over the samples of delta_o times input k (k == K: the bias, input 1). Both factors
// come through shared memory in chunks of GS samples, the next chunk's loads in
// flight during this one's sums.
struct Layer {
  const float* delta;  // [nout][ld]
  const float* act;    // [K][ld]
  int nout, K, w, b;   // outputs, inputs, and where the weights and the biases lie in theta
};

__device__ __forceinline__ void layer_grad(const Layer& L, int patch, int nb, int ld, bool go_on,
                                           float* __restrict__ grad, const Adam& a) {
  constexpr int NT = GO * GK, Q = GS / 4, N = (GO + GK) * Q / NT;  // 16-byte words per thread and chunk
  static_assert((GO * Q) % NT == 0 && (GK * Q) % NT == 0, "whole words per thread");
  __shared__ __align__(16) float T[GO + GK][GS + 4];
  const int t = threadIdx.x, kk = t % GK, oo = t / GK;
  const int nk = (L.K + GK) / GK;  // columns 0 .. K
  const int o0 = patch / nk * GO, k0 = patch % nk * GK;
  float4 r[N];
  // every load is unconditional (clamped indices), so that all are in flight
  auto fetch = [&](int b0) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int e = t + i * NT, q = e % Q, row = e / Q, s = min(b0 + 4 * q, ld - 4);
      const float* src = row < GO ? L.delta + (size_t)min(o0 + row, L.nout - 1) * ld
                                  : L.act + (size_t)min(k0 + row - GO, L.K - 1) * ld;
      r[i] = *reinterpret_cast<const float4*>(src + s);
    }
  };
  float g = 0.f;
  const int o = o0 + oo, k = k0 + kk;
  if (go_on && o < L.nout && k <= L.K) g = grad[k == L.K ? L.b + o : L.w + o * L.K + k];
  fetch(0);
  for (int b0 = 0; b0 < nb; b0 += GS) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int e = t + i * NT, q = e % Q, row = e / Q, s = b0 + 4 * q;
      float4 v = r[i];
      if (row >= GO && k0 + row - GO >= L.K) v = make_float4(1.f, 1.f, 1.f, 1.f);
      // samples past the end add zero
      if (s >= nb) v.x = 0.f;
      if (s + 1 >= nb) v.y = 0.f;
      if (s + 2 >= nb) v.z = 0.f;
      if (s + 3 >= nb) v.w = 0.f;
      *reinterpret_cast<float4*>(&T[row][4 * q]) = v;
    }
    __syncthreads();
    if (b0 + GS < nb) fetch(b0 + GS);
    // products and sums rounded separately
#pragma unroll 8
    for (int s = 0; s < GS; s += 4) {
      const float4 d = *reinterpret_cast<const float4*>(&T[oo][s]);
      const float4 x = *reinterpret_cast<const float4*>(&T[GO + kk][s]);
      g = __fadd_rn(g, __fmul_rn(d.x, x.x));
      g = __fadd_rn(g, __fmul_rn(d.y, x.y));
      g = __fadd_rn(g, __fmul_rn(d.z, x.z));
      g = __fadd_rn(g, __fmul_rn(d.w, x.w));
    }
  }
  if (o >= L.nout || k > L.K) return;
  const int i = k == L.K ? L.b + o : L.w + o * L.K + k;
  if (!a.th) {
    grad[i] = g;
    return;
  }
  const float mi = a.b1 * a.m[i] + (1.f - a.b1) * g;
  const float vi = a.b2 * a.v[i] + (1.f - a.b2) * g * g;
  a.m[i] = mi;
  a.v[i] = vi;
  a.th[i] -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
}

// Patches of the three layers, then (loss) blocks of 64 samples. go_on: the sums of
// the samples before these are in `grad`.
__global__ void __launch_bounds__(GO* GK) k_train_grad(Layer l1, Layer l2, Layer l3, int n1, int n2, int n3,
                                                       const int64_t* __restrict__ perm, int64_t off, int nb, int ld,
                                                       bool go_on, float* __restrict__ grad, Adam a,
                                                       const float* __restrict__ prob, const uint8_t* __restrict__ y,
                                                       float pos_weight, float inv_n, double* __restrict__ loss) {
  const int b = blockIdx.x;
  if (b < n1 + n2 + n3) {
    const Layer L = b < n1 ? l1 : b < n1 + n2 ? l2 : l3;
    layer_grad(L, b < n1 ? b : b < n1 + n2 ? b - n1 : b - n1 - n2, nb, ld, go_on, grad, a);
    return;
  }
  const int s = (b - n1 - n2 - n3) * GO * GK + threadIdx.x;
  double l = 0.0;
  if (s < nb) {
    const bool yy = y[perm ? perm[off + s] : off + s] != 0;
    const double p = (double)prob[s];
    l = yy ? -(double)pos_weight * log(p + 1e-12) : -log(1.0 - p + 1e-12);
    l *= (double)inv_n;
  }
  for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, l);
}

// loss (nullable) += the mean weighted loss of the nb samples; the gradient into
// grad, or an Adam step (grad: the sums, where nb > PART)
int gradient(const float* X, int ldx, const uint8_t* y, const int64_t* perm, int64_t off, int nb, int nin,
             const float* theta, float* grad, const Adam& a, double* loss, float pos_weight, float norm_n,
             void* scratch, cudaStream_t st) {
  raise_smem(k_train_pass, sizeof(TrainSmem));
  const Scratch sc(static_cast<float*>(scratch), std::min(nb, PART), nin);
  const float inv_n = 1.f / norm_n;
  const int w2 = HID * nin + HID, w3 = w2 + HID * HID + HID;
  const Layer l1{sc.d1, sc.x, HID, nin, 0, HID * nin}, l2{sc.d2, sc.h1, HID, HID, w2, w2 + HID * HID},
      l3{sc.d3, sc.h2, 1, HID, w3, w3 + HID};
  auto patches = [](const Layer& L) { return (L.nout + GO - 1) / GO * ((L.K + GK) / GK); };
  const int n1 = patches(l1), n2 = patches(l2), n3 = patches(l3);
  for (int b = 0; b < nb; b += PART) {
    const int n = std::min(PART, nb - b), nl = loss ? (n + GO * GK - 1) / (GO * GK) : 0;
    k_train_pass<<<std::min((n + TB - 1) / TB, MAXBLK), NTT, sizeof(TrainSmem), st>>>(
        X, ldx, y, perm, off + b, n, nin, theta, pos_weight, inv_n, sc, loss != nullptr);
    k_train_grad<<<n1 + n2 + n3 + nl, GO * GK, 0, st>>>(l1, l2, l3, n1, n2, n3, perm, off + b, n, sc.ld, b > 0, grad,
                                                        n == nb - b ? a : Adam{}, sc.prob, y, pos_weight, inv_n, loss);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace

size_t mlp_scratch_bytes(int nb, int nin) { return Scratch::floats(std::min(nb, PART), nin) * sizeof(float); }

int mlp_loss_grad_dev(const float* X, int ldx, const uint8_t* y, int nb, int nin, const float* theta, float* grad,
                      double* loss, float pos_weight, void* scratch, cudaStream_t st) {
  return gradient(X, ldx, y, nullptr, 0, nb, nin, theta, grad, Adam{}, loss, pos_weight, (float)nb, scratch, st);
}

int mlp_train_dev(const float* X, int ldx, const uint8_t* y, int64_t n, int nin, float* theta, int epochs,
                  int batch, float lr, float pos_weight, uint64_t seed, double* last_loss, cudaStream_t st) {
  const int np = mlp_n_params(nin);
  // one allocation: scratch (16-byte rows first), shuffle, loss, Adam moments, gradient sums
  const size_t bytes = n * sizeof(int64_t) + sizeof(double) + 3 * (size_t)np * sizeof(float) +
                       (mlp_scratch_bytes(batch, nin) + 7) / 8 * 8;
  unsigned char* mem = nullptr;
  if (cudaMalloc(&mem, bytes) != cudaSuccess) return -3;
  void* scratch = mem;
  int64_t* perm = reinterpret_cast<int64_t*>(mem + (mlp_scratch_bytes(batch, nin) + 7) / 8 * 8);
  double* dloss = reinterpret_cast<double*>(perm + n);
  float* m = reinterpret_cast<float*>(dloss + 1);
  float *v = m + np, *sums = v + np;
  int e = 0;
  if (cudaMemsetAsync(m, 0, 2 * (size_t)np * sizeof(float), st) != cudaSuccess) e = -3;
  cudaEvent_t copied = nullptr;  // behind the last copy of the shuffle
  if (cudaEventCreateWithFlags(&copied, cudaEventDisableTiming) != cudaSuccess) e = -3;
  std::vector<int64_t> hp(n);
  for (int64_t i = 0; i < n; ++i) hp[i] = i;
  std::mt19937_64 rng(seed);
  int t = 0;
  for (int ep = 0; ep < epochs && !e; ++ep) {
    // The copy below follows the previous epoch's kernels on the stream, and may read
    // hp as late as that (staging pageable memory first is allowed, not promised): the
    // next shuffle waits for it, while this epoch's kernels run.
    if (ep > 0 && cudaEventSynchronize(copied) != cudaSuccess) {
      e = -3;
      break;
    }
    std::shuffle(hp.begin(), hp.end(), rng);
    if (cudaMemcpyAsync(perm, hp.data(), n * sizeof(int64_t), cudaMemcpyHostToDevice, st) ||
        cudaEventRecord(copied, st) != cudaSuccess)
      e = -3;
    double* loss = ep == epochs - 1 ? dloss : nullptr;
    if (loss) cudaMemsetAsync(dloss, 0, sizeof(double), st);
    for (int64_t off = 0; off + batch <= n && !e; off += batch) {
      ++t;
      const float c1 = 1.f - powf(0.9f, (float)t), c2 = 1.f - powf(0.999f, (float)t);
      e = gradient(X, ldx, y, perm, off, batch, nin, theta, sums, Adam{theta, m, v, lr, 0.9f, 0.999f, 1e-8f, c1, c2},
                   loss, pos_weight, (float)batch, scratch, st);
    }
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) e = -3;
  if (copied) cudaEventDestroy(copied);
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
