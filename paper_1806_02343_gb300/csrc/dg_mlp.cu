// Learned troubled-cell indicator: features and BF16 tensor-core inference fused
// with the feature pass (the training kernels: dg_train.cu).
//
// Detection is its own step of the limiter (Sec. 4.2: first detect troubled
// cells, then limit them); this network replaces the TVB detection and only the
// cells it flags go through the characteristic TVB procedure.
//
// Features of a cell (nin = 8 n(d) + 10 D): Legendre coefficients of the 8 MHD
// variables (LDF B mapped exactly to per-component Legendre coefficients), each
// variable divided by s_v = |mean_v| + max_nb |mean_nb,v - mean_v| + 1e-12,
// then rho_nb / rho - 1 for the neighbours -x, +x, -y, +y (, -z, +z), then the
// degree-1 coefficient of each variable along each direction over M~ dx.
// Network: nin -> 64 -> 64 -> 1, ReLU, sigmoid. Weights (flat FP32):
// W1[64][nin], b1[64], W2[64][64], b2[64], w3[64], b3.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "dg_ldf.cuh"
#include "dg_mlp.cuh"
#include "dg_pos.cuh"
#include "dg_tc.cuh"

namespace dgmhd {

namespace {

constexpr int HID = 64;

// periodic face neighbour on the uniform mesh (cell counts stay below 2^31,
// so the index arithmetic is 32-bit)
__device__ __forceinline__ int64_t nbc(const Geom& g, int64_t c, int a, int dir) {
  const unsigned cc = (unsigned)c, nx = (unsigned)g.nx, ny = (unsigned)g.ny;
  const unsigned r = cc / nx;
  int ix = (int)(cc - r * nx), iy = (int)(r % ny), iz = (int)(r / ny);
  if (a == 0) { ix += dir; ix = ix < 0 ? ix + g.nx : (ix >= g.nx ? ix - g.nx : ix); }
  else if (a == 1) { iy += dir; iy = iy < 0 ? iy + g.ny : (iy >= g.ny ? iy - g.ny : iy); }
  else { iz += dir; iz = iz < 0 ? iz + g.nz : (iz >= g.nz ? iz - g.nz : iz); }
  return ((int64_t)iz * g.ny + iy) * g.nx + ix;
}

__device__ __forceinline__ int mrow(const Geom& g, int m) {
  if (g.glm) return m * g.n;
  if (m < 5) return m * g.n;
  if (g.D == 3) return g.ldf0 + (m - 5);
  return m < 7 ? g.ldf0 + (m - 5) : g.bz2d;
}

// Discretisation sizes seen by the feature code: RtDims reads them from the
// Geom at run time; CtDims<GLM, DEG> fixes them at compile time (3D), so the
// loops over variables and modes unroll and every row index is a constant.
struct RtDims {
  static constexpr bool SPARSE = false;
  const Geom& g;
  const MlpTabs& mt;
  __device__ int n() const { return g.n; }
  __device__ bool glm() const { return g.glm != 0; }
  __device__ int D() const { return g.D; }
  __device__ int ldf0() const { return g.ldf0; }
  __device__ int ndiv() const { return g.ndiv; }
  __device__ int bz2d() const { return g.bz2d; }
  __device__ int deg1(int a) const { return mt.deg1[a]; }
  __device__ int mrow(int k) const { return dgmhd::mrow(g, k); }
};

template <bool GLM, int DEG>
struct CtDims {
  static constexpr int N = (DEG + 1) * (DEG + 2) * (DEG + 3) / 6;
  // LDF basis size in 3D (Table A1): 3, 11, 26, 50 for degrees 0..3
  static constexpr int NDIV = DEG == 0 ? 3 : DEG == 1 ? 11 : DEG == 2 ? 26 : 50;
  // the LDF -> Legendre map's pattern is known for degrees 1 and 2
  static constexpr bool SPARSE = !GLM && (DEG == 1 || DEG == 2);
  __device__ static constexpr bool has(int j, int c, int l) {
    if constexpr (SPARSE) return ldf_has<DEG>(j, c, l);
    else return true;
  }
  __device__ static constexpr int n() { return N; }
  __device__ static constexpr bool glm() { return GLM; }
  __device__ static constexpr int D() { return 3; }
  __device__ static constexpr int ldf0() { return GLM ? -1 : 5 * N; }
  __device__ static constexpr int ndiv() { return GLM ? 0 : NDIV; }
  __device__ static constexpr int bz2d() { return -1; }
  // degree-1 modes in the basis order: (1,0,0), (0,1,0), (0,0,1)
  __device__ static constexpr int deg1(int a) { return 1 + a; }
  __device__ static constexpr int mrow(int k) { return (GLM || k < 5) ? k * N : 5 * N + (k - 5); }
};

// physical cell means of the 8 MHD variables from the raw mean rows
template <typename Dm>
__device__ __forceinline__ void phys_means(const Dm& dm, const MlpTabs& mt, const float* raw, float* m) {
#pragma unroll
  for (int k = 0; k < 5; ++k) m[k] = raw[k];
  if (dm.glm()) {
#pragma unroll
    for (int k = 5; k < 8; ++k) m[k] = raw[k];
  } else {
    m[5] = m[6] = m[7] = 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int cc = 0; cc < 3; ++cc)
        if (j < dm.D() && cc < dm.D()) m[5 + cc] += raw[5 + j] * mt.l2l[(j * 3 + cc) * MLP_MAXN + 0];
    if (dm.D() == 2) m[7] = raw[7];
  }
}

// State of one cell and of its face neighbours read straight from the state
// rows (FP32 form: the float mode-0 rows mirror the FP64 means exactly).
template <typename T>
struct GlobalSrc {
  const Geom& g;
  const T* w;
  int64_t c;
  __device__ float row(int r) const { return (float)w[(int64_t)r * g.stride + c]; }
  __device__ void nbraw(int a, int s, float* raw) const {
    const int64_t cn = nbc(g, c, a, s ? 1 : -1);
    for (int k = 0; k < 8; ++k) raw[k] = (float)w[(int64_t)mrow(g, k) * g.stride + cn];
  }
  __device__ float imdx(const MlpTabs& mt) const { return mt.inv_mdx; }
};

// Octree meshes (the per-side leaf lists of the context): the neighbour mean on side
// (a, s) is the average of the leaves across that side (one of the same level
// or coarser, or the 2^(D-1) finer ones), as the octree TVB procedure reads
// it; the slope scale is the leaf's own M~ dx_K. A side without a leaf (the
// edge of a partition's local mesh) reads the cell's own means.
struct AmrFeat {
  const int32_t* side_nb;    // the leaves across each side, in face-entry order (AmrHost::side_nb)
  const uint8_t* side_info;  // count | relation << 4 per leaf and side
  const double* dxc;
  double dxmin;  // the mesh's smallest cell (the one inv_mdx was made with)
  int on;
};

template <typename T>
struct AmrSrc {
  const Geom& g;
  const T* w;
  int64_t c;
  const AmrFeat& af;
  __device__ float row(int r) const { return (float)w[(int64_t)r * g.stride + c]; }
  __device__ void nbraw(int a, int s, float* raw) const {
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int sidx = 2 * a + (s ? 1 : 0);
    const int cnt = af.side_info[c * 6 + sidx] & 15;
    for (int k2 = 0; k2 < cnt; ++k2) {
      const int64_t cn = af.side_nb[c * 24 + sidx * 4 + k2];
      for (int k = 0; k < 8; ++k) acc[k] += (float)w[(int64_t)mrow(g, k) * g.stride + cn];
    }
    if (cnt == 0) {
      for (int k = 0; k < 8; ++k) raw[k] = (float)w[(int64_t)mrow(g, k) * g.stride + c];
      return;
    }
    const float inv = 1.f / (float)cnt;  // 1 or 2^(D-1): exact
    for (int k = 0; k < 8; ++k) raw[k] = acc[k] * inv;
  }
  __device__ float imdx(const MlpTabs& mt) const { return mt.inv_mdx * (float)(af.dxmin / af.dxc[c]); }
};

// features of one cell, written through put(k, value) for k in [0, nin)
// part < 0: every feature; else the work split between nparts (2 or 4)
// threads of the cell: part 0 writes the neighbour-density features; the
// Legendre variables go to the parts in order (GLM: 8 / nparts each; Powell:
// the 5 hydro variables), the LDF-mapped B to the last part (Powell).
template <typename Dm, typename Src, typename Put>
__device__ __forceinline__ void features_of(const Dm& dm, const MlpTabs& mt, const Src& src, Put put,
                                            int part = -1, int nparts = 2) {
  auto owner = [&](int v) {
    if (dm.glm()) return (v * nparts) >> 3;
    return nparts == 2 ? 0 : (v < 2 ? 0 : v < 4 ? 1 : 2);
  };
  const int ldf_part = nparts - 1;
  const int n = dm.n();
  float m[8];
  {
    float raw[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) raw[k] = src.row(dm.mrow(k));
    phys_means(dm, mt, raw, m);
  }
  float dmax[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (a >= dm.D()) break;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      float raw[8], mn[8];
      src.nbraw(a, s, raw);
      phys_means(dm, mt, raw, mn);
#pragma unroll
      for (int k = 0; k < 8; ++k) dmax[k] = fmaxf(dmax[k], fabsf(mn[k] - m[k]));
      if (part <= 0) put(8 * n + 2 * a + s, mn[0] / m[0] - 1.f);
    }
  }
  float inv[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) inv[k] = 1.f / (fabsf(m[k]) + dmax[k] + 1e-12f);
  const float imdx = src.imdx(mt);
  const int nleg = dm.glm() ? 8 : 5;
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    const bool leg = v < nleg || (!dm.glm() && dm.D() == 2 && v == 7);
    if (!leg) continue;
    if (part >= 0 && owner(v) != part) continue;
    const int r0 = (v == 7 && !dm.glm()) ? dm.bz2d() : v * n;
#pragma unroll
    for (int l = 0; l < n; ++l) {
      const float av = (l == 0) ? m[v] : src.row(r0 + l);
      put(v * n + l, av * inv[v]);
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (a < dm.D() && l == dm.deg1(a)) put(8 * n + 2 * dm.D() + 8 * a + v, av * imdx);
    }
  }
  if (!dm.glm() && (part < 0 || part == ldf_part)) {
    // LDF B -> per-component Legendre coefficients (exact map)
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) {
      if (cc >= dm.D()) break;
#pragma unroll
      for (int l = 0; l < n; ++l) {
        float acc = 0.f;
        if constexpr (Dm::SPARSE) {
          // only the map's non-zero entries (38 of 780 at degree 2), in the order of j
#pragma unroll
          for (int j = 0; j < Dm::ndiv(); ++j)
            if (Dm::has(j, cc, l)) acc += src.row(dm.ldf0() + j) * mt.l2l[(j * 3 + cc) * MLP_MAXN + l];
        } else {
          for (int j = 0; j < dm.ndiv(); ++j) acc += src.row(dm.ldf0() + j) * mt.l2l[(j * 3 + cc) * MLP_MAXN + l];
        }
        put((5 + cc) * n + l, acc * inv[5 + cc]);
#pragma unroll
        for (int a = 0; a < 3; ++a)
          if (a < dm.D() && l == dm.deg1(a)) put(8 * n + 2 * dm.D() + 8 * a + 5 + cc, acc * imdx);
      }
    }
  }
}

template <typename T, typename Put>
__device__ __forceinline__ void cell_features(const Geom& g, const MlpTabs& mt, const T* w, const double* /*wmean*/,
                                              int64_t c, const AmrFeat& af, Put put) {
  if (af.on) features_of(RtDims{g, mt}, mt, AmrSrc<T>{g, w, c, af}, put);
  else features_of(RtDims{g, mt}, mt, GlobalSrc<T>{g, w, c}, put);
}

template <typename T>
__global__ void k_features(Geom g, MlpTabs mt, const T* __restrict__ w, const double* __restrict__ wmean,
                           float* __restrict__ X, int ldx, AmrFeat af) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const int nin = 8 * g.n + 10 * g.D;
  float* xr = X + c * ldx;
  for (int k = nin; k < ldx; ++k) xr[k] = 0.f;
  cell_features(g, mt, w, wmean, c, af, [&](int k, float v) { xr[k] = v; });
}

// ---------------------------------------------------------------- inference (BF16 mma.sync)
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Network on the 32 cells of one warp: rows Xw[0..32) of bf16 features (row
// stride LD1) -> probabilities; writes the flags of the 32 cells to flw[0..32)
// and, for live cells, flag / prob. base = first cell of the warp.
template <int KP, int NTILE = 2>
__device__ __forceinline__ void infer_warp(const __nv_bfloat16* Xw, const __nv_bfloat16* W1s,
                                           const __nv_bfloat16* W2s, const float* bs, uint8_t* flw, int64_t base,
                                           int64_t ncell, float thresh, uint8_t* __restrict__ flag,
                                           float* __restrict__ prob) {
  constexpr int LD1 = KP + 8, LD2 = HID + 8;
  const int lane = threadIdx.x & 31;
  const int gq = lane >> 2, tq = lane & 3;
  for (int tile = 0; tile < NTILE; ++tile) {
    const __nv_bfloat16* Xt = Xw + tile * 16 * LD1;
    float h1[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      h1[j][0] = bs[8 * j + 2 * tq];
      h1[j][1] = bs[8 * j + 2 * tq + 1];
      h1[j][2] = bs[8 * j + 2 * tq];
      h1[j][3] = bs[8 * j + 2 * tq + 1];
    }
#pragma unroll
    for (int kk = 0; kk < KP / 16; ++kk) {
      uint32_t a[4];
      a[0] = *reinterpret_cast<const uint32_t*>(Xt + gq * LD1 + 16 * kk + 2 * tq);
      a[1] = *reinterpret_cast<const uint32_t*>(Xt + (gq + 8) * LD1 + 16 * kk + 2 * tq);
      a[2] = *reinterpret_cast<const uint32_t*>(Xt + gq * LD1 + 16 * kk + 8 + 2 * tq);
      a[3] = *reinterpret_cast<const uint32_t*>(Xt + (gq + 8) * LD1 + 16 * kk + 8 + 2 * tq);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t b[2];
        b[0] = *reinterpret_cast<const uint32_t*>(W1s + (8 * j + gq) * LD1 + 16 * kk + 2 * tq);
        b[1] = *reinterpret_cast<const uint32_t*>(W1s + (8 * j + gq) * LD1 + 16 * kk + 8 + 2 * tq);
        mma_bf16(h1[j], a, b);
      }
    }
    // ReLU; accumulator tiles 2kk, 2kk+1 form the A fragment of layer 2's k-step kk
    float h2[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      h2[j][0] = bs[HID + 8 * j + 2 * tq];
      h2[j][1] = bs[HID + 8 * j + 2 * tq + 1];
      h2[j][2] = bs[HID + 8 * j + 2 * tq];
      h2[j][3] = bs[HID + 8 * j + 2 * tq + 1];
    }
#pragma unroll
    for (int kk = 0; kk < HID / 16; ++kk) {
      uint32_t a[4];
      a[0] = pack_bf16(fmaxf(h1[2 * kk][0], 0.f), fmaxf(h1[2 * kk][1], 0.f));
      a[1] = pack_bf16(fmaxf(h1[2 * kk][2], 0.f), fmaxf(h1[2 * kk][3], 0.f));
      a[2] = pack_bf16(fmaxf(h1[2 * kk + 1][0], 0.f), fmaxf(h1[2 * kk + 1][1], 0.f));
      a[3] = pack_bf16(fmaxf(h1[2 * kk + 1][2], 0.f), fmaxf(h1[2 * kk + 1][3], 0.f));
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t b[2];
        b[0] = *reinterpret_cast<const uint32_t*>(W2s + (8 * j + gq) * LD2 + 16 * kk + 2 * tq);
        b[1] = *reinterpret_cast<const uint32_t*>(W2s + (8 * j + gq) * LD2 + 16 * kk + 8 + 2 * tq);
        mma_bf16(h2[j], a, b);
      }
    }
    // output layer: rows gq and gq+8 of the tile, reduced over the quad
    float o0 = 0.f, o1 = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float w0 = bs[2 * HID + 8 * j + 2 * tq], w1 = bs[2 * HID + 8 * j + 2 * tq + 1];
      o0 += fmaxf(h2[j][0], 0.f) * w0 + fmaxf(h2[j][1], 0.f) * w1;
      o1 += fmaxf(h2[j][2], 0.f) * w0 + fmaxf(h2[j][3], 0.f) * w1;
    }
    o0 += __shfl_xor_sync(0xffffffffu, o0, 1);
    o0 += __shfl_xor_sync(0xffffffffu, o0, 2);
    o1 += __shfl_xor_sync(0xffffffffu, o1, 1);
    o1 += __shfl_xor_sync(0xffffffffu, o1, 2);
    if (tq == 0) {
      const float b3 = bs[3 * HID];
      const int r0 = tile * 16 + gq;
      const int64_t c0 = base + r0;
      const float p0 = 1.f / (1.f + __expf(-(o0 + b3)));
      const float p1 = 1.f / (1.f + __expf(-(o1 + b3)));
      flw[r0] = p0 > thresh ? 1 : 0;
      flw[r0 + 8] = p1 > thresh ? 1 : 0;
      if (c0 < ncell) {
        if (flag) flag[c0] = p0 > thresh ? 1 : 0;
        if (prob) prob[c0] = p0;
      }
      if (c0 + 8 < ncell) {
        if (flag) flag[c0 + 8] = p1 > thresh ? 1 : 0;
        if (prob) prob[c0 + 8] = p1;
      }
    }
  }
}

// appends the warp's flagged live cells to list (ballot + one atomic per warp)
__device__ __forceinline__ void compact_warp(bool mine, int64_t c, int32_t* __restrict__ list,
                                             DevScalars* __restrict__ sc) {
  const int lane = threadIdx.x & 31;
  const unsigned bal = __ballot_sync(0xffffffffu, mine);
  const int cnt = __popc(bal);
  unsigned at = 0;
  if (lane == 0 && cnt) {
    at = atomicAdd(&sc->nflag, (unsigned)cnt);
    atomicAdd(&sc->cnt_flagged, (unsigned long long)cnt);
  }
  at = __shfl_sync(0xffffffffu, at, 0);
  if (mine) list[at + __popc(bal & ((1u << lane) - 1u))] = (int32_t)c;
}

// One warp infers 32 cells (two m16 tiles); KP = padded input width (multiple of 16).
// Shared layout: W1s[64][KP+8] bf16, W2s[64][72] bf16, Xs[warps][32][KP+8] bf16, biases f32,
// flags of the warp's 32 cells. Persistent: the weights are staged once per block and the
// block walks 128-cell tiles with a grid stride. With `list`, each warp appends its flagged
// cells (ballot + one atomic per warp) to list and counts them in sc.
template <typename T, int KP>
__global__ void __launch_bounds__(128) k_mlp_infer(Geom g, MlpTabs mt, const T* __restrict__ w,
                                                   const double* __restrict__ wmean,
                                                   const __nv_bfloat16* __restrict__ W1,
                                                   const __nv_bfloat16* __restrict__ W2,
                                                   const float* __restrict__ bias, float thresh,
                                                   uint8_t* __restrict__ flag, float* __restrict__ prob,
                                                   int32_t* __restrict__ list, DevScalars* __restrict__ sc,
                                                   AmrFeat af) {
  constexpr int LD1 = KP + 8, LD2 = HID + 8;
  extern __shared__ __align__(128) unsigned char smraw[];
  __nv_bfloat16* W1s = reinterpret_cast<__nv_bfloat16*>(smraw);
  __nv_bfloat16* W2s = W1s + HID * LD1;
  __nv_bfloat16* Xs = W2s + HID * LD2;
  float* bs = reinterpret_cast<float*>(Xs + 4 * 32 * LD1);  // b1[64], b2[64], w3[64], b3
  uint8_t* fl = reinterpret_cast<uint8_t*>(bs + 3 * HID + 1);  // [4][32]
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  for (int i = t; i < HID * KP; i += 128) W1s[(i / KP) * LD1 + i % KP] = W1[i];
  for (int i = t; i < HID * HID; i += 128) W2s[(i / HID) * LD2 + i % HID] = W2[i];
  for (int i = t; i < 3 * HID + 1; i += 128) bs[i] = bias[i];
  __syncthreads();
  const int nin = 8 * g.n + 10 * g.D;
  for (int64_t base = (int64_t)blockIdx.x * 128; base < g.ncell; base += (int64_t)gridDim.x * 128) {
    // features of this thread's cell (rows of Xs are private to the warp)
    const int64_t c = base + t;
    const bool live = c < g.ncell;
    {
      __nv_bfloat16* xr = Xs + (warp * 32 + lane) * LD1;
      for (int k = live ? nin : 0; k < KP; ++k) xr[k] = __float2bfloat16_rn(0.f);
      if (live) cell_features(g, mt, w, wmean, c, af, [&](int k, float v) { xr[k] = __float2bfloat16_rn(v); });
    }
    __syncwarp();
    infer_warp<KP>(Xs + warp * 32 * LD1, W1s, W2s, bs, fl + warp * 32, base + warp * 32, g.ncell, thresh, flag,
                   prob);
    __syncwarp();
    if (list) compact_warp(live && fl[warp * 32 + lane] != 0, c, list, sc);
    __syncwarp();
  }
}

__global__ void k_to_bf16(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, int rows, int cols,
                          int ldd) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= rows * ldd) return;
  const int r = i / ldd, k = i % ldd;
  dst[i] = __float2bfloat16_rn(k < cols ? src[r * cols + k] : 0.f);
}

// ---------------------------------------------------------------- tiled inference
// FP32 form on uniform 3D meshes whose x-rows hold whole 128-cell tiles, on the
// tensor core: two threads per cell build the features of their variables straight
// from coalesced loads (a row of a warp's 32 cells is one 128-byte line; the x, y, z
// neighbours' means are lines that other tiles of the same SMs read as rows) and
// store them, eight at a time, as the layer's BF16 operand. Each part reads only its
// own variables of the neighbours, and the FP32 positivity screen is summed from the
// same registers. 57 KB of shared memory at degree 2: four blocks per SM overlap
// their loads, their two layers and their epilogues. Bound by the loads' latency
// and the instruction issue. (Staging the 112 rows of a tile in shared memory by
// bulk copies took 57 KB more: two blocks per SM, each waiting for its copies, and
// 2-byte feature stores with 4-way bank conflicts: 3.91 ms per pass on 256^3 cells,
// GLM, degree 2, now 2.00 ms; 128^3, Powell, 0.51 and 0.28 ms.)

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

constexpr long long kWaitCycles = 2000000000ll;  // about one second at GB300 clocks

// feature words (two BF16 each) START .. START + CNT of cell `cell`: 16-byte
// stores where four words of a core-matrix row are complete
template <int START, int CNT, int KP>
__device__ __forceinline__ void put_words(__nv_bfloat16* Xs, int cell, const uint32_t* W) {
  sf::each<0, CNT>([&](auto K) {
    constexpr int k = decltype(K)::value, at = START + k, q0 = at / 4 * 4;  // q0: the quad's first word
    constexpr bool quad = q0 >= START && q0 + 4 <= START + CNT;
    __nv_bfloat16* d = Xs + tc::kmajor_index(cell, 2 * at, KP);
    if constexpr (!quad) *reinterpret_cast<uint32_t*>(d) = W[k];
    else if constexpr (at == q0) *reinterpret_cast<uint4*>(d) = make_uint4(W[k], W[k + 1], W[k + 2], W[k + 3]);
  });
}

// Features of `features_of` (same expressions, so the same BF16 values) of the
// variables of part P (GLM: 0-3, 4-7; Powell: the hydro variables, B), and of the
// same variables the terms of pos_screen_rows: dv (sum of |coefficients| beyond the
// mean, times the basis bound) and ms (mean). cn: the cell's neighbours.
template <bool GLM, int DEG, int KP, int P>
__device__ __forceinline__ void tile_features(const MlpTabs& mt, const PosScreen& ps, const float* __restrict__ w,
                                              int64_t S, int64_t c, const int64_t (&cn)[6], int cell,
                                              __nv_bfloat16* Xs, float* dv, float* ms) {
  using Dm = CtDims<GLM, DEG>;
  constexpr int N = Dm::N, SLOPE = 8 * N + 6;
  static_assert(N % 2 == 0, "pairs of features stay within a variable");
  if constexpr (GLM || P == 0) {
    constexpr int V0 = GLM ? 4 * P : 0, NV = GLM ? 4 : 5;
    const float* base = w + (int64_t)(V0 * N) * S;
    float m[NV], dmax[NV], nd[6];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      m[v] = base[(int64_t)(v * N) * S + c];
      dmax[v] = 0.f;
    }
#pragma unroll
    for (int q = 0; q < 6; ++q)
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const float x = base[(int64_t)(v * N) * S + cn[q]];
        dmax[v] = fmaxf(dmax[v], fabsf(x - m[v]));
        if (P == 0 && v == 0) nd[q] = x / m[0] - 1.f;
      }
    uint32_t W[NV * N / 2];
    float sl[3][NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const float inv = 1.f / (fabsf(m[v]) + dmax[v] + 1e-12f);
      float f[N], d = 0.f;
#pragma unroll
      for (int l = 0; l < N; ++l) {
        const float av = l == 0 ? m[v] : base[(int64_t)(v * N + l) * S + c];
        f[l] = av * inv;
        if (l > 0) d += fabsf(av);
        if (l >= 1 && l <= 3) sl[l - 1][v] = av * mt.inv_mdx;
      }
      dv[v] = d;
      ms[v] = m[v];
#pragma unroll
      for (int l = 0; l < N; l += 2) W[(v * N + l) / 2] = pack_bf16(f[l], f[l + 1]);
    }
    put_words<V0 * N / 2, NV * N / 2, KP>(Xs, cell, W);
    uint32_t x[3];
    if constexpr (P == 0) {
#pragma unroll
      for (int a = 0; a < 3; ++a) x[a] = pack_bf16(nd[2 * a], nd[2 * a + 1]);
      put_words<4 * N, 3, KP>(Xs, cell, x);
    } else {  // padding up to KP
      x[0] = 0u;
      put_words<(SLOPE + 24) / 2, 1, KP>(Xs, cell, x);
    }
    sf::each<0, 3>([&](auto A) {
      constexpr int a = decltype(A)::value;
      x[0] = pack_bf16(sl[a][0], sl[a][1]);
      x[1] = pack_bf16(sl[a][2], sl[a][3]);
      put_words<(SLOPE + 8 * a + V0) / 2, 2, KP>(Xs, cell, x);
      if constexpr (NV == 5) Xs[tc::kmajor_index(cell, SLOPE + 8 * a + 4, KP)] = __float2bfloat16_rn(sl[a][4]);
    });
  } else {
    constexpr int NDIV = Dm::NDIV;
    const float* base = w + (int64_t)(5 * N) * S;
    auto phys = [&](const float* raw, float* m) {
      m[0] = m[1] = m[2] = 0.f;
#pragma unroll
      for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) m[cc] += raw[j] * mt.l2l[(j * 3 + cc) * MLP_MAXN + 0];
    };
    float R[NDIV], m[3], dmax[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < NDIV; ++j) R[j] = base[(int64_t)j * S + c];
    phys(R, m);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      float raw[3], mn[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) raw[j] = base[(int64_t)j * S + cn[q]];
      phys(raw, mn);
#pragma unroll
      for (int k = 0; k < 3; ++k) dmax[k] = fmaxf(dmax[k], fabsf(mn[k] - m[k]));
    }
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) {
      dv[cc] = ms[cc] = 0.f;
#pragma unroll
      for (int j = 0; j < 3; ++j) ms[cc] += R[j] * ps.ldf_mean0[j * 3 + cc];
    }
#pragma unroll
    for (int j = 3; j < NDIV; ++j)
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) dv[cc] += fabsf(R[j]) * ps.ldf_maxabs[j * 3 + cc];
    uint32_t W[3 * N / 2], x[1];
    sf::each<0, 3>([&](auto CC) {
      constexpr int cc = decltype(CC)::value;
      const float inv = 1.f / (fabsf(m[cc]) + dmax[cc] + 1e-12f);
      float f[N];
      sf::each<0, N>([&](auto L) {
        constexpr int l = decltype(L)::value;
        float acc = 0.f;
        sf::each<0, NDIV>([&](auto J) {
          constexpr int j = decltype(J)::value;
          if constexpr (Dm::has(j, cc, l)) acc += R[j] * mt.l2l[(j * 3 + cc) * MLP_MAXN + l];
        });
        f[l] = acc * inv;
        if constexpr (l >= 1 && l <= 3) {
          constexpr int q = SLOPE + 8 * (l - 1) + 5 + cc;
          Xs[tc::kmajor_index(cell, q, KP)] = __float2bfloat16_rn(acc * mt.inv_mdx);
        }
      });
#pragma unroll
      for (int l = 0; l < N; l += 2) W[(cc * N + l) / 2] = pack_bf16(f[l], f[l + 1]);
    });
    put_words<5 * N / 2, 3 * N / 2, KP>(Xs, cell, W);
    x[0] = 0u;
    put_words<(SLOPE + 24) / 2, 1, KP>(Xs, cell, x);
  }
}

constexpr int kTileThreads = 256;  // two threads per cell of the 128-cell tile

template <int KP, bool GLM, int DEG>
__global__ void __launch_bounds__(kTileThreads, DEG <= 2 ? 4 : 2)
    k_mlp_tile(Geom g, const __grid_constant__ MlpTabs mt, const float* __restrict__ w,
               const __nv_bfloat16* __restrict__ W1, const __nv_bfloat16* __restrict__ W2,
               const float* __restrict__ bias, float thresh, uint8_t* __restrict__ flag, float* __restrict__ prob,
               int32_t* __restrict__ list, DevScalars* __restrict__ sc, int32_t* __restrict__ plist,
               const __grid_constant__ PosScreen ps) {
  constexpr int NTH = kTileThreads, CG = NTH / 128, CW = HID / CG, N1 = GLM ? 4 : 3;
  extern __shared__ __align__(128) unsigned char smraw[];
  // tensor-core operands in the K-major core-matrix layout (dg_tc.cuh)
  __nv_bfloat16* W1s = reinterpret_cast<__nv_bfloat16*>(smraw);  // [HID][KP]
  __nv_bfloat16* W2s = W1s + HID * KP;                           // [HID][HID]
  __nv_bfloat16* Xs = W2s + HID * HID;  // [128][KP] features; then layer 1's output [128][HID]
  float* scr = reinterpret_cast<float*>(Xs + 128 * KP);  // [2][N1][128] part 1's dv and ms
  float* part = scr + 2 * N1 * 128;                      // [CG][128] partial sums of the output layer
  float* bs = part + CG * 128;                           // b1[64], b2[64], w3[64], b3
  uint64_t* bar = reinterpret_cast<uint64_t*>(bs + 3 * HID + 2);  // MMA completion
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 1);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int cell = t & 127, fpart = t >> 7;  // warp-uniform part
  for (int i = t; i < HID * KP; i += NTH) W1s[tc::kmajor_index(i / KP, i % KP, KP)] = W1[i];
  for (int i = t; i < HID * HID; i += NTH) W2s[tc::kmajor_index(i / HID, i % HID, HID)] = W2[i];
  for (int i = t; i < 3 * HID + 1; i += NTH) bs[i] = bias[i];
  if (t == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // 128 tensor-memory columns: layer 1's accumulator [128 x 64], then layer 2's
  if (warp == 0) tc::tmem_alloc(tslot, 128);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tm = *tslot;
  constexpr uint32_t IDESC = tc::idesc_bf16_f32(128, HID);
  const int64_t S = g.stride;
  const unsigned ntile = (unsigned)(g.ncell / 128), tpr = (unsigned)g.nx / 128u;
  // bounded wait of every thread on an mbarrier phase; false on timeout (all threads agree)
  auto wait_all = [&](unsigned parity) {
    bool ok = false;
    const long long t0 = clock64();
    while (!(ok = mbar_try_wait(bar, parity)))
      if (clock64() - t0 > kWaitCycles) break;
    return __syncthreads_and(ok) != 0;
  };
  int mma_pending = -1;  // parity of an MMA commit not yet observed (timeout path), else -1
  for (unsigned tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    const int64_t c0 = (int64_t)tile * 128, c = c0 + cell;
    int64_t cn[6];
    {
      const unsigned rowi = tile / tpr, xt = tile - rowi * tpr;
      const int iz = (int)(rowi / (unsigned)g.ny), iy = (int)(rowi - (unsigned)iz * (unsigned)g.ny);
      const int x = (int)(xt * 128u) + cell;
      const int64_t pl = (int64_t)g.nx * g.ny;
      cn[0] = x == 0 ? c + g.nx - 1 : c - 1;
      cn[1] = x == g.nx - 1 ? c - (g.nx - 1) : c + 1;
      cn[2] = iy == 0 ? c + pl - g.nx : c - g.nx;
      cn[3] = iy == g.ny - 1 ? c - (pl - g.nx) : c + g.nx;
      cn[4] = iz == 0 ? c + pl * (g.nz - 1) : c - pl;
      cn[5] = iz == g.nz - 1 ? c - pl * (g.nz - 1) : c + pl;
    }
    float dv[5], ms[5];
    if (fpart == 0) {
      tile_features<GLM, DEG, KP, 0>(mt, ps, w, S, c, cn, cell, Xs, dv, ms);
    } else {
      tile_features<GLM, DEG, KP, 1>(mt, ps, w, S, c, cn, cell, Xs, dv, ms);
#pragma unroll
      for (int k = 0; k < N1; ++k) {
        scr[k * 128 + cell] = dv[k];
        scr[(N1 + k) * 128 + cell] = ms[k];
      }
    }
    tc::fence_proxy_async();  // the features, written by every thread, become tensor-core operands
    __syncthreads();
    // layer 1 on the tensor core: D1[128 x 64] = X[128 x KP] W1^T (FP32 in tensor memory)
    if (t == 0) {
      tc::fence_after_sync();
#pragma unroll
      for (int kk = 0; kk < KP / 16; ++kk)
        tc::mma_bf16(tm, tc::smem_desc(tc::smem_u32(Xs + kk * 128), 128, KP * 16),
                     tc::smem_desc(tc::smem_u32(W1s + kk * 128), 128, KP * 16), IDESC, kk > 0);
      tc::commit(bar);
    }
    mma_pending = 0;
    bool sfail = false;
    if (plist && fpart == 0) {
      // FP32 positivity screen, while the tensor core runs layer 1; only the cells
      // the indicator does not flag are listed from it (the TVB kernel screens the
      // flagged ones after limiting them)
      constexpr int N0 = GLM ? 4 : 5;
      float d8[8], m8[8];
#pragma unroll
      for (int k = 0; k < N0; ++k) {
        d8[k] = dv[k];
        m8[k] = ms[k];
      }
#pragma unroll
      for (int k = N0; k < 8; ++k) {
        d8[k] = scr[(k - N0) * 128 + cell];
        m8[k] = scr[(N1 + k - N0) * 128 + cell];
      }
      sfail = !pos_screen_bound(ps, m8, d8);
    }
    if (!wait_all(0)) {
      if (t == 0) atomicOr(&sc->status, 8);
      break;
    }
    mma_pending = -1;
    tc::fence_after_sync();
    // epilogue 1: warp w reads lanes 32 (w % 4).. of columns CW (w / 4)..; bias,
    // ReLU, BF16 into layer 2's A operand (over the features: layer 1 is done)
    const int quarter = warp & 3, colh = warp >> 2, row = 32 * quarter + lane;
    const uint32_t tlane = (uint32_t)(32 * quarter) << 16;
    {
      float v[CW];
      tc::ld32(tm + tlane + CW * colh, v);
      // 16-byte stores of eight BF16 values: the 8 rows of a core matrix fill 128 contiguous bytes
#pragma unroll
      for (int j = 0; j < CW / 8; ++j) {
        uint4 pk;
        uint32_t* pw = reinterpret_cast<uint32_t*>(&pk);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = CW * colh + 8 * j + 2 * e;
          pw[e] = pack_bf16(fmaxf(v[8 * j + 2 * e] + bs[k], 0.f), fmaxf(v[8 * j + 2 * e + 1] + bs[k + 1], 0.f));
        }
        *reinterpret_cast<uint4*>(Xs + tc::kmajor_index(row, CW * colh + 8 * j, HID)) = pk;
      }
    }
    tc::fence_before_sync();
    tc::fence_proxy_async();
    __syncthreads();
    // layer 2: D2[128 x 64] = H1[128 x 64] W2^T, in columns 64..127
    if (t == 0) {
      tc::fence_after_sync();
#pragma unroll
      for (int kk = 0; kk < HID / 16; ++kk)
        tc::mma_bf16(tm + HID, tc::smem_desc(tc::smem_u32(Xs + kk * 128), 128, HID * 16),
                     tc::smem_desc(tc::smem_u32(W2s + kk * 128), 128, HID * 16), IDESC, kk > 0);
      tc::commit(bar);
    }
    mma_pending = 1;
    if (!wait_all(1)) {
      if (t == 0) atomicOr(&sc->status, 8);
      break;
    }
    mma_pending = -1;
    tc::fence_after_sync();
    // epilogue 2: bias, ReLU and this warp's share of the output layer's dot product
    {
      float v[CW];
      tc::ld32(tm + tlane + HID + CW * colh, v);
      float o = 0.f;
#pragma unroll
      for (int j = 0; j < CW; ++j) o += fmaxf(v[j] + bs[HID + CW * colh + j], 0.f) * bs[2 * HID + CW * colh + j];
      part[colh * 128 + row] = o;
    }
    tc::fence_before_sync();
    __syncthreads();
    // output and lists, by the first part's four warps; the other part goes on to the
    // next tile (it writes `part` again only behind that tile's barriers)
    if (fpart == 0) {
      float z = bs[3 * HID];
#pragma unroll
      for (int gq = 0; gq < CG; ++gq) z += part[gq * 128 + t];
      const float p = 1.f / (1.f + __expf(-z));
      const bool hit = p > thresh;
      if (flag) flag[c] = hit ? 1 : 0;
      if (prob) prob[c] = p;
      if (list) compact_warp(hit, c, list, sc);
      if (plist) append_cells(!hit && sfail, c, plist, &sc->npos);
    }
  }
  if (mma_pending >= 0) {
    // a commit not observed in time: wait once more (bounded) before the columns are freed
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, (unsigned)mma_pending))
      if (clock64() - t0 > kWaitCycles) break;
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tm, 128);
}

}  // namespace

static AmrFeat amr_feat(const Ctx& c) {
  return AmrFeat{c.amr.side_nb, c.amr.side_info, c.amr.dxc, c.g.dx, c.amr.on ? 1 : 0};
}

int mlp_build_tables(Ctx& c) {
  const Basis& B = *c.hb;
  const Geom& g = c.g;
  MlpTabs mt;
  std::memset(&mt, 0, sizeof(mt));
  if (g.n > MLP_MAXN || 8 * g.n + 10 * g.D > MLP_MAXIN) return -7;
  for (int a = 0; a < g.D; ++a)
    for (int l = 0; l < g.n; ++l) {
      const auto& k = B.modes[l];
      if (k[0] + k[1] + k[2] == 1 && k[a] == 1) mt.deg1[a] = l;
    }
  mt.inv_mdx = (float)(1.0 / (c.p.Mtilde * g.dx));
  if (!g.glm) {
    // <phi_j,c, P_l> / M_l by exact monomial integration
    const auto& ms = B.ms;
    for (int j = 0; j < g.ndiv && j < 64; ++j)
      for (int cc = 0; cc < g.D; ++cc)
        for (int l = 0; l < g.n; ++l) {
          double s = 0.0;
          for (size_t i = 0; i < ms.exps.size(); ++i) {
            const double a = B.ldf[j][cc][i];
            if (a == 0.0) continue;
            for (size_t k = 0; k < ms.exps.size(); ++k) {
              const double b = B.leg[l][k];
              if (b == 0.0) continue;
              double t = a * b;
              for (int ax = 0; ax < g.D; ++ax) {
                const int e = ms.exps[i][ax] + ms.exps[k][ax];
                t *= (e & 1) ? 0.0 : 2.0 / (e + 1.0);
              }
              s += t;
            }
          }
          mt.l2l[(j * 3 + cc) * MLP_MAXN + l] = (float)(s / B.leg_mass[l]);
        }
  }
  c.mlp = mt;
  return 0;
}

int mlp_features_launch(Ctx& c, const void* w, const double* wmean, float* X, int ldx, cudaStream_t st) {
  const Geom& g = c.g;
  const unsigned nb = (unsigned)((g.ncell + 127) / 128);
  if (c.p.precision == DG_PREC_FP32MIX)
    k_features<float><<<nb, 128, 0, st>>>(g, c.mlp, (const float*)w, nullptr, X, ldx, amr_feat(c));
  else
    k_features<double><<<nb, 128, 0, st>>>(g, c.mlp, (const double*)w, nullptr, X, ldx, amr_feat(c));
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mlp_set_weights(Ctx& c, const float* theta_dev, int nin, float thresh) {
  const Geom& g = c.g;
  if (nin != 8 * g.n + 10 * g.D) return -1;
  const int kp = (nin + 15) / 16 * 16;
  if (kp != 64 && kp != 80 && kp != 112 && kp != 192) return -7;
  if (!c.mlp_w1) {
    if (cudaMalloc(&c.mlp_w1, (size_t)HID * kp * 2) || cudaMalloc(&c.mlp_w2, (size_t)HID * HID * 2) ||
        cudaMalloc(&c.mlp_bias, (3 * HID + 1) * sizeof(float)))
      return -3;
  }
  const float* W1 = theta_dev;
  const float* b1 = W1 + HID * nin;
  const float* W2 = b1 + HID;
  const float* b2 = W2 + HID * HID;
  const float* w3 = b2 + HID;
  k_to_bf16<<<(HID * kp + 255) / 256, 256>>>(W1, (__nv_bfloat16*)c.mlp_w1, HID, nin, kp);
  k_to_bf16<<<(HID * HID + 255) / 256, 256>>>(W2, (__nv_bfloat16*)c.mlp_w2, HID, HID, HID);
  cudaMemcpy(c.mlp_bias, b1, HID * sizeof(float), cudaMemcpyDeviceToDevice);
  cudaMemcpy(c.mlp_bias + HID, b2, HID * sizeof(float), cudaMemcpyDeviceToDevice);
  cudaMemcpy(c.mlp_bias + 2 * HID, w3, (HID + 1) * sizeof(float), cudaMemcpyDeviceToDevice);
  c.mlp_kp = kp;
  c.mlp_thresh = thresh;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : -3;
}

template <int KP, bool GLM>
static constexpr size_t tile_smem() {
  return (size_t)HID * KP * 2 + (size_t)HID * HID * 2 + (size_t)128 * KP * 2 +
         (2 * (GLM ? 4 : 3) * 128 + 2 * 128 + 3 * HID + 2) * sizeof(float) + 16;
}

// the tiled kernel applies: FP32 form, uniform 3D mesh, x-rows of whole 128-cell
// tiles (other meshes keep k_mlp_infer: the two sum the layers in another order,
// and a probability near the threshold must not change sides with the kernel)
static bool tile_ok(const Ctx& c) {
  const Geom& g = c.g;
  return c.p.precision == DG_PREC_FP32MIX && !c.amr.on && g.D == 3 && g.nx % 128 == 0;
}

template <int KP, bool GLM, int DEG>
static void tile_launch(Ctx& c, const void* w, uint8_t* flag, float* prob, cudaStream_t st, int32_t* list,
                        int32_t* plist) {
  constexpr size_t sm = tile_smem<KP, GLM>();
  const auto k = k_mlp_tile<KP, GLM, DEG>;
  raise_smem(k, sm);
  // persistent: the weights are staged once per block. At most four blocks per
  // SM: each holds 128 of the SM's 512 tensor-memory columns
  const int per_sm = DEG <= 2 ? 4 : 2;
  const unsigned nb = (unsigned)std::min<int64_t>(c.g.ncell / 128, (int64_t)c.nsm * per_sm);
  k<<<nb, kTileThreads, sm, st>>>(c.g, c.mlp, (const float*)w, (const __nv_bfloat16*)c.mlp_w1,
                                  (const __nv_bfloat16*)c.mlp_w2, c.mlp_bias, c.mlp_thresh, flag, prob, list, c.sc,
                                  plist, c.pscr);
}

template <typename T, int KP>
static void infer_launch(Ctx& c, const void* w, const double* wmean, uint8_t* flag, float* prob, cudaStream_t st,
                         int32_t* list, int32_t* plist, bool* screened) {
  if constexpr (sizeof(T) == 4) {
    if (tile_ok(c)) {
      // compile-time feature code for the scheme and degree (KP follows the degree)
      constexpr int DEG = KP == 64 ? 1 : KP == 112 ? 2 : KP == 192 ? 3 : 0;
      if constexpr (DEG > 0) {
        if (c.g.d == DEG) {
          if (c.g.glm) tile_launch<KP, true, DEG>(c, w, flag, prob, st, list, plist);
          else tile_launch<KP, false, DEG>(c, w, flag, prob, st, list, plist);
          if (screened) *screened = plist != nullptr;
          return;
        }
      }
    }
  }
  const Geom& g = c.g;
  const size_t sm = (size_t)HID * (KP + 8) * 2 + (size_t)HID * (HID + 8) * 2 + (size_t)4 * 32 * (KP + 8) * 2 +
                    (3 * HID + 1) * sizeof(float) + 128;
  raise_smem(k_mlp_infer<T, KP>, sm);
  // persistent grid: a few blocks per SM (the weights are staged once per block)
  const int64_t tiles = (g.ncell + 127) / 128;
  const unsigned nb = (unsigned)std::min<int64_t>(tiles, (int64_t)c.nsm * 4);
  k_mlp_infer<T, KP><<<nb, 128, sm, st>>>(g, c.mlp, (const T*)w, wmean, (const __nv_bfloat16*)c.mlp_w1,
                                           (const __nv_bfloat16*)c.mlp_w2, c.mlp_bias, c.mlp_thresh, flag, prob,
                                           list, c.sc, amr_feat(c));
}

int mlp_infer_launch(Ctx& c, const void* w, const double* wmean, uint8_t* flag, float* prob, cudaStream_t st,
                     int32_t* list, int32_t* pos_list, bool* screened) {
  if (screened) *screened = false;
  if (!c.mlp_w1) return -1;
  const bool f32 = c.p.precision == DG_PREC_FP32MIX;
  // FP32 form: features read the float mirror of the FP64 means (exact copies)
  switch (c.mlp_kp) {
#define KPCASE(K)                                                                 \
  case K:                                                                         \
    if (f32) infer_launch<float, K>(c, w, nullptr, flag, prob, st, list, pos_list, screened); \
    else infer_launch<double, K>(c, w, nullptr, flag, prob, st, list, nullptr, nullptr);      \
    break;
    KPCASE(64)
    KPCASE(80)
    KPCASE(112)
    KPCASE(192)
#undef KPCASE
    default:
      return -7;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace dgmhd
