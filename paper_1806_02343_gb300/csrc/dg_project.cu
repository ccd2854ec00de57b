// L2 projection of point values onto the basis (Sec. 3.1, eq. u-exp inverted) in
// 3D, one axis at a time (dg_sf.cuh): one thread per (variable, cell) reduces
// the npts values along z, then y, then x to the moments of total degree <= d.
// 79 FP64 operations per variable at degree 2 and 3 points per axis instead of
// the 270 products of the dense form (and their weights); the point values are
// read once, coalesced along the cells, instead of once per row by one warp per
// cell. Powell: the LDF rows from B's Legendre moments through the sparse map
// (the LDF functions are polynomials of total degree <= d). Bound by the FP64
// pipe. Measured on GB300, 96^3 cells, GLM, degree 2, 3 points: 11.3 ms dense,
// 1.6 ms now.
#include <cuda_runtime.h>

#include "dg_kernels.cuh"
#include "dg_ldf.cuh"
#include "dg_sf.cuh"

namespace dgmhd {

namespace {

using sf::V;
constexpr int NTJ = 9 * 32;

// ldf: the map A[j][3][n], then 1 / mass of the LDF rows (Powell)
template <typename T, int DEG, int NP, bool GLM>
__global__ void __launch_bounds__(NTJ) k_project_sf(Geom g, const double* __restrict__ nodal,
                                                    const double* __restrict__ ldf, T* __restrict__ w,
                                                    double* __restrict__ wmean) {
  constexpr int RN = NP - 1;  // rule index: NP points
  constexpr int N = LdfPattern<DEG>::N, NDIV = LdfPattern<DEG>::NDIV, M2 = sf::n_modes2(DEG);
  __shared__ double RL[GLM ? 1 : 3 * N][32];
  const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;
  const int64_t S = g.stride;
  const int64_t cb = (int64_t)blockIdx.x * 32 + lane;
  const bool live = cb < g.ncell;
  const int64_t c = live ? cb : g.ncell - 1;
  V R[N];
  if (GLM || v < 8) {
    const double* f = nodal + (int64_t)v * (NP * NP * NP) * S + c;
    V mx[M2][NP];  // [(k2, k3)][x point]
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      V my[DEG + 1][NP];  // [k3][y point]
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        V u[NP], m[DEG + 1];
#pragma unroll
        for (int k = 0; k < NP; ++k) u[k] = f[(int64_t)((i * NP + j) * NP + k) * S];
        sf::reduce1<RN, DEG + 1>(u, m);
#pragma unroll
        for (int k = 0; k <= DEG; ++k) my[k][j] = m[k];
      }
      sf::each<0, DEG + 1>([&](auto K3) {
        constexpr int k3 = decltype(K3)::value;
        V m[DEG + 1 - k3];
        sf::reduce1<RN, DEG + 1 - k3>(my[k3], m);
#pragma unroll
        for (int k2 = 0; k2 + k3 <= DEG; ++k2) mx[sf::mode2_idx<DEG>(k2, k3)][i] = m[k2];
      });
    }
    sf::each<0, DEG + 1>([&](auto K2) {
      constexpr int k2 = decltype(K2)::value;
      sf::each<0, DEG + 1 - k2>([&](auto K3) {
        constexpr int k3 = decltype(K3)::value;
        V m[DEG + 1 - k2 - k3];
        sf::reduce1<RN, DEG + 1 - k2 - k3>(mx[sf::mode2_idx<DEG>(k2, k3)], m);
#pragma unroll
        for (int k1 = 0; k1 + k2 + k3 <= DEG; ++k1)
          R[sf::mode_idx(k1, k2, k3)] = m[k1];
      });
    });
  }
  // the moments' scale (sf::reduce1)
  auto scale = [](int i, int j, int k) { return sf::sig<RN>(i) * sf::sig<RN>(j) * sf::sig<RN>(k); };
  auto put = [&](int row, int mean, V x) {
    if (!live) return;
    w[(int64_t)row * S + c] = (T)x;
    if (sizeof(T) == 4 && mean >= 0) wmean[(int64_t)mean * S + c] = x;
  };
  const bool leg = GLM || v < 5;
#pragma unroll
  for (int i = 0; i <= DEG; ++i)
#pragma unroll
    for (int j = 0; i + j <= DEG; ++j)
#pragma unroll
      for (int k = 0; i + j + k <= DEG; ++k) {
        const int l = sf::mode_idx(i, j, k);
        if (leg) put(v * N + l, l == 0 ? v : -1, R[l] * (scale(i, j, k) * sf::mode_minv(i, j, k)));
        else if (v < 8) RL[(v - 5) * N + l][lane] = R[l] * scale(i, j, k);
      }
  if constexpr (!GLM) {
    __syncthreads();
    sf::each<0, NDIV>([&](auto J) {
      constexpr int j = decltype(J)::value;
      if (j % 9 == v) {
        V s = 0.0;
        sf::each<0, 3 * N>([&](auto I) {
          constexpr int cc = decltype(I)::value / N, l = decltype(I)::value % N;
          if constexpr (ldf_has<DEG>(j, cc, l)) s = __fma_rn(RL[cc * N + l][lane], __ldg(ldf + (j * 3 + cc) * N + l), s);
        });
        // 1 / mass in the working precision, as in the operator's tables (and the dense projection)
        put(5 * N + j, j < 3 ? 5 + j : -1, s * (double)(T)__ldg(ldf + NDIV * 3 * N + j));
      }
    });
  }
}

template <typename T, int DEG, int NP>
void run(const Geom& g, const double* nodal, const double* ldf, T* w, double* wmean, cudaStream_t st) {
  const unsigned nb = (unsigned)((g.ncell + 31) / 32);
  if (g.glm) k_project_sf<T, DEG, NP, true><<<nb, NTJ, 0, st>>>(g, nodal, ldf, w, wmean);
  else k_project_sf<T, DEG, NP, false><<<nb, NTJ, 0, st>>>(g, nodal, ldf, w, wmean);
}

}  // namespace

// 3D, degrees 1-3, with d + 1 up to d + 3 points per axis (Solver.project_ic's
// default), the counts initial states are given with, and degree 3 with 3; any
// other count runs the dense kernel.
bool project_sf_ok(const Geom& g, int npts) {
  return g.D == 3 && g.d >= 1 && g.d <= 3 && npts >= (g.d == 3 ? 3 : g.d + 1) && npts <= g.d + 3;
}

bool ldf_pattern_ok(int degree, const double* A) {
  auto check = [&](auto P, auto has) {
    for (int j = 0; j < decltype(P)::NDIV; ++j)
      for (int cc = 0; cc < 3; ++cc)
        for (int l = 0; l < decltype(P)::N; ++l)
          if (A[(j * 3 + cc) * decltype(P)::N + l] != 0.0 && !has(j, cc, l)) return false;
    return true;
  };
  if (degree == 1) return check(LdfPattern<1>{}, [](int j, int c, int l) { return ldf_has<1>(j, c, l); });
  if (degree == 2) return check(LdfPattern<2>{}, [](int j, int c, int l) { return ldf_has<2>(j, c, l); });
  return degree == 3 && check(LdfPattern<3>{}, [](int j, int c, int l) { return ldf_has<3>(j, c, l); });
}

template <typename T>
void launch_project_sf(const Geom& g, int npts, const double* nodal, const double* ldf, T* w, double* wmean,
                       cudaStream_t st) {
  switch (10 * g.d + npts) {
    case 12: run<T, 1, 2>(g, nodal, ldf, w, wmean, st); break;
    case 13: run<T, 1, 3>(g, nodal, ldf, w, wmean, st); break;
    case 14: run<T, 1, 4>(g, nodal, ldf, w, wmean, st); break;
    case 23: run<T, 2, 3>(g, nodal, ldf, w, wmean, st); break;
    case 24: run<T, 2, 4>(g, nodal, ldf, w, wmean, st); break;
    case 25: run<T, 2, 5>(g, nodal, ldf, w, wmean, st); break;
    case 33: run<T, 3, 3>(g, nodal, ldf, w, wmean, st); break;
    case 34: run<T, 3, 4>(g, nodal, ldf, w, wmean, st); break;
    case 35: run<T, 3, 5>(g, nodal, ldf, w, wmean, st); break;
    case 36: run<T, 3, 6>(g, nodal, ldf, w, wmean, st); break;
  }
}
template void launch_project_sf<float>(const Geom&, int, const double*, const double*, float*, double*, cudaStream_t);
template void launch_project_sf<double>(const Geom&, int, const double*, const double*, double*, double*, cudaStream_t);

}  // namespace dgmhd
