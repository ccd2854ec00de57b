// FP64 operator on uniform 2D meshes (GLM and Powell, degrees 1-3): the sizes
// fixed at compile time and the work spread for small meshes, where a step is
// latency: the accuracy runs take 32^2 cells. On such a mesh the generic kernels
// walked run-time loops of dependent loads (45 us per cell pass, 37 us per face
// pass at 32^2, degree 2, Powell), one warp per cell with 9 of 32 lanes busy at
// the volume points.
// * k2_face: one thread per face point, lanes over cells (every load of the two
//   cells' rows is independent and coalesced), one warp per block so that 192
//   warps reach 152 SMs; HLLD of dg_sf.cuh.
// * k2_cell: 4 cells per block; volume points, face terms and rows of the 4 cells
//   are each one flat index range over the block's 192 threads (180 rows at
//   degree 2, Powell), and a row's sum runs in one chain per axis and face.
//   (Fetching tables, rows and fluxes together at the start gained nothing.)
// * k2_jump, k2_dt: the timestep in two launches instead of four; the last block
//   forms the step's scalars.
// Bound by latency up to about 64^2 cells, by the FP64 pipe beyond. GB300, Powell,
// degree 2, per step of three stages, generic kernels and these: 32^2 cells 289 and
// 125 us, 128^2 1.83 and 0.81 ms, 512^2 26.9 and 11.7 ms (GLM 15.6 and 11.1 ms).
// FP32 runs stay on the generic kernels: their FP64 means show another rounding of
// the FP32 fluxes at 1e-9.
#include <cuda_runtime.h>

#include <algorithm>

#include "dg_dt.cuh"
#include "dg_kernels.cuh"
#include "dg_phys.cuh"
#include "dg_sf.cuh"

namespace dgmhd {

namespace {

using sf::V;

template <int DEG, bool GLM>
struct D2 {
  static constexpr int NQ = DEG + 1, QV = NQ * NQ, N = (DEG + 1) * (DEG + 2) / 2;
  static constexpr int NDIV = GLM ? 0 : 2 * N - DEG * (DEG + 1) / 2;  // Table A1, D = 2
  static constexpr int NV = GLM ? 9 : 8, NLEG = GLM ? 9 : 6;         // Legendre variables (Powell: B_z among them)
  static constexpr int NR = NLEG * N + NDIV, NF = GLM ? 9 : 10;
  static constexpr int CB = 4, NT = 192;
  // Legendre variable k: its variable and its first row
  static constexpr __device__ int var(int k) { return GLM || k < 5 ? k : 7; }
  static constexpr __device__ int row0(int k) { return GLM || k < 5 ? k * N : 5 * N + NDIV; }
};
// index of mode (i, j): total degree, then i descending
constexpr __device__ int mode2d(int i, int j) { return (i + j) * (i + j + 1) / 2 + j; }

__device__ __forceinline__ int64_t nbr2(const Geom& g, int64_t c, int a, int dir) {
  const unsigned cc = (unsigned)c, nx = (unsigned)g.nx;
  int iy = (int)(cc / nx), ix = (int)(cc - iy * nx);
  int& k = a == 0 ? ix : iy;
  const int n = a == 0 ? g.nx : g.ny;
  k += dir;
  k = k < 0 ? k + n : (k >= n ? k - n : k);
  return (int64_t)iy * g.nx + ix;
}

// F[axis][point][slot][cell]: the flux of the nine variables (GLM), or of the
// eight, then B^n_F minus the left and the right cell's own normal trace
template <int DEG, bool GLM>
__global__ void __launch_bounds__(32) k2_face(Geom g, const double* __restrict__ Lf, const V* __restrict__ w,
                                              V* __restrict__ F, const DevScalars* __restrict__ sc, V eps) {
  using D = D2<DEG, GLM>;
  constexpr int N = D::N, NQ = D::NQ, NDIV = D::NDIV;
  const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x;
  if (c >= g.ncell) return;
  const int ap = blockIdx.y, a = ap / NQ, p = ap - a * NQ;
  const int64_t cl = nbr2(g, c, a, -1);
  const int64_t S = g.stride;
  const V y = sf::Rule<DEG>::node(0) * (p == 0 ? 1.0 : p == NQ - 1 ? -1.0
              : DEG == 2 ? 0.0 : (p == 1 ? 1.0 : -1.0) * (sf::Rule<3>::x(1) / sf::Rule<3>::x(0)));
  const V l[4] = {1.0, y, 1.5 * y * y - 0.5, (2.5 * y * y - 1.5) * y};
  V u[2][9];
#pragma unroll
  for (int s = 0; s < 2; ++s) {  // 0: the left cell on its +a face, 1: the own cell on its -a face
    const V* pw = w + (s ? c : cl);
    const V sg = s ? -1.0 : 1.0;
#pragma unroll
    for (int k = 0; k < D::NLEG; ++k) {
      V m[N];
#pragma unroll
      for (int q = 0; q < N; ++q) m[q] = pw[(int64_t)(D::row0(k) + q) * S];
      V val = 0.0;
#pragma unroll
      for (int j = 0; j <= DEG; ++j) {  // tangential mode; the normal modes summed with their sign
        V even = 0.0, odd = 0.0;
#pragma unroll
        for (int i = 0; i + j <= DEG; ++i) {
          const V x = a == 0 ? m[mode2d(i, j)] : m[mode2d(j, i)];
          if (i & 1) odd += x;
          else even += x;
        }
        val = __fma_rn(l[j], __fma_rn(sg, odd, even), val);
      }
      u[s][D::var(k)] = val;
    }
    if constexpr (!GLM) {
      V bx = 0.0, by = 0.0;
      const double* T = Lf + (int64_t)(s ? 2 * a : 2 * a + 1) * NDIV * 2 * NQ + p;
#pragma unroll
      for (int j = 0; j < NDIV; ++j) {
        const V x = pw[(int64_t)(5 * N + j) * S];
        bx = __fma_rn(x, __ldg(T + (j * 2 + 0) * NQ), bx);
        by = __fma_rn(x, __ldg(T + (j * 2 + 1) * NQ), by);
      }
      u[s][5] = bx;
      u[s][6] = by;
    }
  }
  // rotated frame: normal a, tangential (a + 1) % 3, (a + 2) % 3
  V uL[8], uR[8], Fo[8];
  auto rot = [&](const V* q, V* r) {
    r[0] = q[0];
    r[4] = q[4];
    r[1] = a == 0 ? q[1] : q[2];
    r[2] = a == 0 ? q[2] : q[3];
    r[3] = a == 0 ? q[3] : q[1];
    r[5] = a == 0 ? q[5] : q[6];
    r[6] = a == 0 ? q[6] : q[7];
    r[7] = a == 0 ? q[7] : q[5];
  };
  rot(u[0], uL);
  rot(u[1], uR);
  const V bn = sf::hlld(uL, uR, g.gamma, eps, Fo);
  V out[10];
  if constexpr (GLM) {  // interface values of Sec. 4.1.5
    const V ch = sc->ch;
    Fo[5] = __fma_rn(0.5, u[0][8] + u[1][8], -(0.5 * ch * (uR[5] - uL[5])));
    out[8] = ch * ch * __fma_rn(0.5, uL[5] + uR[5], -((u[1][8] - u[0][8]) / (2.0 * ch)));
  } else {
    out[8] = bn - uL[5];
    out[9] = bn - uR[5];
  }
  out[0] = Fo[0];
  out[4] = Fo[4];
  out[1] = a == 0 ? Fo[1] : Fo[3];
  out[2] = a == 0 ? Fo[2] : Fo[1];
  out[3] = a == 0 ? Fo[3] : Fo[2];
  out[5] = a == 0 ? Fo[5] : Fo[7];
  out[6] = a == 0 ? Fo[6] : Fo[5];
  out[7] = a == 0 ? Fo[7] : Fo[6];
  V* o = F + (int64_t)ap * D::NF * S + c;
#pragma unroll
  for (int k = 0; k < D::NF; ++k) o[k * S] = out[k];
}

// Cell update: volume integral, surface terms, Powell's face term or the GLM
// damping, SSP combination (cmode 0: plain rhs, 1: ca == 0, 2: ca != 0)
template <int DEG, bool GLM>
__global__ void __launch_bounds__(192) k2_cell(Geom g, Tables<double> tb, const V* __restrict__ w,
                                               const V* __restrict__ F, V* out, const V* w0, double ca, double cb,
                                               int cmode, const DevScalars* __restrict__ sc) {
  // out may alias w0: each element is read, then written, by one thread.
  using D = D2<DEG, GLM>;
  constexpr int N = D::N, NQ = D::NQ, QV = D::QV, NDIV = D::NDIV, NV = D::NV, NR = D::NR, CB = D::CB, NT = D::NT;
  __shared__ V W[NR][CB], G[2][NV][QV][CB], FS[4][NV][NQ][CB], Q[8][CB];
  const int t = threadIdx.x;
  const int64_t c0 = (int64_t)blockIdx.x * CB, S = g.stride;
  auto cell = [&](int i) { return min(c0 + i, g.ncell - 1); };  // absent cells repeat the last one
  for (int k = t; k < NR * CB; k += NT) W[k / CB][k % CB] = w[(int64_t)(k / CB) * S + cell(k % CB)];
  __syncthreads();
  const V ch = GLM ? sc->ch : 0.0;
  // weighted fluxes at the volume points
  for (int k = t; k < QV * CB; k += NT) {
    const int q = k / CB, i = k % CB;
    V u[9], f[9];
    u[8] = 0.0;
#pragma unroll
    for (int b = 0; b < D::NLEG; ++b) {
      V s = 0.0;
#pragma unroll
      for (int l = 0; l < N; ++l) s = __fma_rn(W[D::row0(b) + l][i], __ldg(tb.Pv + l * QV + q), s);
      u[D::var(b)] = s;
    }
    if constexpr (!GLM) {
      u[5] = u[6] = 0.0;
#pragma unroll
      for (int j = 0; j < NDIV; ++j)
#pragma unroll
        for (int cc = 0; cc < 2; ++cc)
          u[5 + cc] = __fma_rn(W[5 * N + j][i], __ldg(tb.Lv + (j * 2 + cc) * QV + q), u[5 + cc]);
    }
    const V wq = __ldg(tb.wv + q);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      flux_dir(u, a, (V)g.gamma, GLM, ch * ch, f);
#pragma unroll
      for (int v = 0; v < NV; ++v) G[a][v][q][i] = wq * f[v];
    }
  }
  // Powell: q(<u>_K) = (0, B, v.B, v) from the cell means (Sec. 4.1.3)
  if (!GLM && t < CB) {
    const V ir = 1.0 / W[0][t];
    const V vx = W[N][t] * ir, vy = W[2 * N][t] * ir, vz = W[3 * N][t] * ir;
    V b[3] = {0.0, 0.0, W[D::row0(5)][t]};
#pragma unroll
    for (int j = 0; j < 2; ++j)  // the degree-0 LDF rows come first
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) b[cc] = __fma_rn(W[5 * N + j][t], __ldg(tb.L0 + j * 2 + cc), b[cc]);
    Q[0][t] = 0.0;
    Q[1][t] = b[0];
    Q[2][t] = b[1];
    Q[3][t] = b[2];
    Q[4][t] = vx * b[0] + vy * b[1] + vz * b[2];
    Q[5][t] = vx;
    Q[6][t] = vy;
    Q[7][t] = vz;
  }
  __syncthreads();
  // outward face terms, weighted: face f = 2 axis + side
  for (int k = t; k < 4 * NV * NQ * CB; k += NT) {
    const int i = k % CB, p = k / CB % NQ, v = k / (CB * NQ) % NV, f = k / (CB * NQ * NV), a = f >> 1, side = f & 1;
    const int64_t c = cell(i);
    const V* q = F + (int64_t)(a * NQ + p) * D::NF * S + (side ? nbr2(g, c, a, 1) : c);
    V x = q[v * S];
    if (!GLM && v > 0) x = __fma_rn(Q[v][i], q[(side ? 8 : 9) * S], x);  // the +a face's left cell is this one
    FS[f][v][p][i] = (side ? 1.0 : -1.0) * __ldg(tb.wf + p) * x;
  }
  __syncthreads();
  const double dt = sc->dt, metric = 2.0 / g.dx;
  for (int k = t; k < NR * CB; k += NT) {
    const int r = k / CB, i = k % CB;
    if (c0 + i >= g.ncell) continue;
    V acc[2] = {0.0, 0.0}, fac[4] = {0.0, 0.0, 0.0, 0.0};
    const bool ldf = !GLM && r >= 5 * N && r < 5 * N + NDIV;
    if (!ldf) {
      const bool bz = !GLM && r >= 5 * N + NDIV;
      const int v = bz ? 7 : r / N, l = bz ? r - 5 * N - NDIV : r % N;
#pragma unroll
      for (int q = 0; q < QV; ++q)
#pragma unroll
        for (int a = 0; a < 2; ++a) acc[a] = __fma_rn(G[a][v][q][i], __ldg(tb.dPv + (a * N + l) * QV + q), acc[a]);
#pragma unroll
      for (int p = 0; p < NQ; ++p)
#pragma unroll
        for (int f = 0; f < 4; ++f) fac[f] = __fma_rn(FS[f][v][p][i], __ldg(tb.Pf + (f * N + l) * NQ + p), fac[f]);
    } else {
      const int j = r - 5 * N;
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
#pragma unroll
        for (int q = 0; q < QV; ++q)
#pragma unroll
          for (int a = 0; a < 2; ++a)
            acc[a] = __fma_rn(G[a][5 + cc][q][i], __ldg(tb.dLv + ((a * NDIV + j) * 2 + cc) * QV + q), acc[a]);
#pragma unroll
        for (int p = 0; p < NQ; ++p)
#pragma unroll
          for (int f = 0; f < 4; ++f)
            fac[f] = __fma_rn(FS[f][5 + cc][p][i], __ldg(tb.Lf + ((f * NDIV + j) * 2 + cc) * NQ + p), fac[f]);
      }
    }
    V rhs = metric * __ldg(tb.minv + r) * ((acc[0] + acc[1]) - ((fac[0] + fac[1]) + (fac[2] + fac[3])));
    if (GLM && r >= 8 * N) rhs = __fma_rn(-sc->kappa, W[r][i], rhs);
    const int64_t o = (int64_t)r * S + c0 + i;
    if (cmode != 0) {
      const V s = cb * __fma_rn(dt, rhs, W[r][i]);
      rhs = cmode == 2 ? __fma_rn(ca, w0[o], s) : s;
    }
    out[o] = rhs;
  }
}

// Powell timestep's face jumps, one thread per face point (lanes over cells):
// w_p |B^n_F - B^n_L| and w_p |B^n_F - B^n_R| at J[axis][point][side][cell]. Also
// resets the timestep's minimum for k2_dt behind it.
template <int DEG>
__global__ void __launch_bounds__(32) k2_jump(Geom g, Tables<double> tb, const V* __restrict__ w, V* __restrict__ J,
                                              DevScalars* __restrict__ sc) {
  using D = D2<DEG, false>;
  constexpr int N = D::N, NQ = D::NQ, NDIV = D::NDIV;
  const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x;
  if (c == 0 && blockIdx.y == 0) dt_init(sc);
  if (c >= g.ncell) return;
  const int ap = blockIdx.y, a = ap / NQ, p = ap - a * NQ;
  const int64_t cl = nbr2(g, c, a, -1), S = g.stride;
  V r[2], b[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int f = s ? 2 * a : 2 * a + 1;
    const V* pw = w + (s ? c : cl);
    V x[N], z[NDIV], rs = 0.0, bs = 0.0;
#pragma unroll
    for (int l = 0; l < N; ++l) x[l] = pw[(int64_t)l * S];
#pragma unroll
    for (int j = 0; j < NDIV; ++j) z[j] = pw[(int64_t)(5 * N + j) * S];
#pragma unroll
    for (int l = 0; l < N; ++l) rs = __fma_rn(x[l], __ldg(tb.Pf + (f * N + l) * NQ + p), rs);
#pragma unroll
    for (int j = 0; j < NDIV; ++j) bs = __fma_rn(z[j], __ldg(tb.Lf + ((f * NDIV + j) * 2 + a) * NQ + p), bs);
    r[s] = rs;
    b[s] = bs;
  }
  const V bF = bn_face(r[0], r[1], b[0], b[1]), wp = __ldg(tb.wf + p);
  V* o = J + (int64_t)ap * 2 * S + c;
  o[0] = wp * fabs(bF - b[0]);
  o[S] = wp * fabs(bF - b[1]);
}

// eq. cfl (and eq. powell_dt) of every cell, its minimum, and the step's scalars
// by the last block to finish
template <int DEG, bool GLM>
__global__ void __launch_bounds__(32) k2_dt(Geom g, Tables<double> tb, const V* __restrict__ w,
                                            const V* __restrict__ J, dg_mhd_params prm, DevScalars* sc,
                                            double* dt_out) {
  using D = D2<DEG, GLM>;
  constexpr int N = D::N, NQ = D::NQ;
  const int64_t S = g.stride;
  double dt = DBL_MAX, smax = 0.0;
  for (int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x; c < g.ncell; c += (int64_t)gridDim.x * 32) {
    if (g.owned && !g.owned[c]) continue;
    V m[8], jump[4 * NQ];
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = w[(int64_t)(GLM || k < 5 ? k * N : k == 7 ? D::row0(5) : 5 * N + k - 5) * S + c];
    if constexpr (!GLM) {
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const int64_t cp = nbr2(g, c, a, 1);
#pragma unroll
        for (int p = 0; p < NQ; ++p) {
          const V* q = J + (int64_t)(a * NQ + p) * 2 * S;
          jump[(2 * a) * NQ + p] = q[S + c];  // minus face: its right side
          jump[(2 * a + 1) * NQ + p] = q[cp];  // plus face: its left side
        }
      }
    }
    const V ir = 1.0 / m[0], vx = m[1] * ir, vy = m[2] * ir, vz = m[3] * ir;
    V bx = m[5], by = m[6];
    if constexpr (!GLM) {
      bx = m[5] * __ldg(tb.L0) + m[6] * __ldg(tb.L0 + 2);
      by = m[5] * __ldg(tb.L0 + 1) + m[6] * __ldg(tb.L0 + 3);
    }
    const V b2 = bx * bx + by * by + m[7] * m[7];
    const V pr = (g.gamma - 1.0) * (m[4] - 0.5 * m[0] * (vx * vx + vy * vy + vz * vz) - 0.5 * b2);
    const V sum = fabs(vx) + fabs(vy) + 2.0 * sqrt((g.gamma * pr + b2) * ir);
    V dtc = prm.cfl * g.dx / ((2.0 * DEG + 1.0) * sum);
    smax = fmax(smax, 0.5 * sum);
    if constexpr (!GLM) {
      V acc = 0.0;
#pragma unroll
      for (int k = 0; k < 4 * NQ; ++k) acc += jump[k];
      // (1/V_K) oint |B^n_F - B^n_K| dS: the face measure dx / 2 over the volume dx^2
      const V rate = 0.5 * acc * fabs(vx * bx + vy * by + vz * m[7]);
      if (rate > 0.0) dtc = fmin(dtc, prm.eta_powell * g.dx * m[4] / rate);
    }
    if (!(dtc > 0.0) || !isfinite(dtc)) {
      atomicOr(&sc->status, 1);
      dtc = DBL_MAX;
    }
    dt = fmin(dt, dtc);
  }
  dt = warp_min(dt);
  smax = -warp_min(-smax);
  if (threadIdx.x == 0) {
    atomicMin(&sc->dt_bits, dbits(dt));
    atomicMax(&sc->smax_bits, dbits(smax));
    __threadfence();
    if (atomicInc(&sc->dt_done, gridDim.x - 1) == gridDim.x - 1) {  // the counter is back at zero
      __threadfence();
      dt_finalize(g, prm, sc, nullptr, dt_out);
    }
  }
}

template <int DEG, bool GLM>
void run(const Geom& g, const Tables<double>& tb, const double* w, double* F, double* out, const double* w0, double ca,
         double cb, int cmode, const DevScalars* sc, double eps, bool face, cudaStream_t st) {
  using D = D2<DEG, GLM>;
  if (face) k2_face<DEG, GLM><<<dim3((unsigned)((g.ncell + 31) / 32), 2 * D::NQ), 32, 0, st>>>(g, tb.Lf, w, F, sc, eps);
  else
    k2_cell<DEG, GLM><<<(unsigned)((g.ncell + D::CB - 1) / D::CB), D::NT, 0, st>>>(g, tb, w, F, out, w0, ca, cb, cmode,
                                                                                  sc);
}

template <int DEG>
void by_scheme(const Geom& g, const Tables<double>& tb, const double* w, double* F, double* out, const double* w0,
               double ca, double cb, int cmode, const DevScalars* sc, double eps, bool face, cudaStream_t st) {
  if (g.glm) run<DEG, true>(g, tb, w, F, out, w0, ca, cb, cmode, sc, eps, face, st);
  else run<DEG, false>(g, tb, w, F, out, w0, ca, cb, cmode, sc, eps, face, st);
}

template <int DEG, bool GLM>
bool sizes_ok(const Geom& g) {
  using D = D2<DEG, GLM>;
  return g.n == D::N && g.ndiv == D::NDIV && g.nrows == D::NR && g.Qv == D::QV && g.Qf == D::NQ &&
         (GLM || (g.ldf0 == 5 * D::N && g.bz2d == 5 * D::N + D::NDIV && g.DB == 2));
}

}  // namespace

bool op2d_ok(const Geom& g) {
  if (g.D != 2) return false;
  switch (g.d) {
    case 1: return g.glm ? sizes_ok<1, true>(g) : sizes_ok<1, false>(g);
    case 2: return g.glm ? sizes_ok<2, true>(g) : sizes_ok<2, false>(g);
    case 3: return g.glm ? sizes_ok<3, true>(g) : sizes_ok<3, false>(g);
  }
  return false;
}

namespace {

template <int DEG>
void dt_by_scheme(const Geom& g, const Tables<double>& tb, const double* w, double* J, const dg_mhd_params& p,
                  DevScalars* sc, double* dt_out, int nsm, cudaStream_t st) {
  const unsigned nb = (unsigned)std::min<int64_t>((g.ncell + 31) / 32, (int64_t)nsm * 16);
  if (g.glm) {
    launch_dt_init(sc, st);
    k2_dt<DEG, true><<<nb, 32, 0, st>>>(g, tb, w, J, p, sc, dt_out);
  } else {
    k2_jump<DEG><<<dim3((unsigned)((g.ncell + 31) / 32), 2 * D2<DEG, false>::NQ), 32, 0, st>>>(g, tb, w, J, sc);
    k2_dt<DEG, false><<<nb, 32, 0, st>>>(g, tb, w, J, p, sc, dt_out);
  }
}

}  // namespace

void launch_dt_2d(const Geom& g, const Tables<double>& tb, const double* w, double* J, const dg_mhd_params& p,
                  DevScalars* sc, double* dt_out, int nsm, cudaStream_t st) {
  if (g.d == 1) dt_by_scheme<1>(g, tb, w, J, p, sc, dt_out, nsm, st);
  else if (g.d == 2) dt_by_scheme<2>(g, tb, w, J, p, sc, dt_out, nsm, st);
  else dt_by_scheme<3>(g, tb, w, J, p, sc, dt_out, nsm, st);
}

static void launch_2d(const Geom& g, const Tables<double>& tb, const double* w, double* F, double* out,
                      const double* w0, double ca, double cb, int cmode, const DevScalars* sc, double eps, bool face,
                      cudaStream_t st) {
  switch (g.d) {
    case 1: by_scheme<1>(g, tb, w, F, out, w0, ca, cb, cmode, sc, eps, face, st); break;
    case 2: by_scheme<2>(g, tb, w, F, out, w0, ca, cb, cmode, sc, eps, face, st); break;
    case 3: by_scheme<3>(g, tb, w, F, out, w0, ca, cb, cmode, sc, eps, face, st); break;
  }
}

void launch_face_2d(const Geom& g, const Tables<double>& tb, const double* w, double* F, const DevScalars* sc,
                    double eps, cudaStream_t st) {
  launch_2d(g, tb, w, F, nullptr, nullptr, 0.0, 0.0, 0, sc, eps, true, st);
}

void launch_cell_2d(const Geom& g, const Tables<double>& tb, const double* w, double* F, double* out, const double* w0,
                    double ca, double cb, int combine, const DevScalars* sc, cudaStream_t st) {
  launch_2d(g, tb, w, F, out, w0, ca, cb, combine ? (ca != 0.0 ? 2 : 1) : 0, sc, 0.0, false, st);
}

}  // namespace dgmhd
