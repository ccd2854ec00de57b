// L2 projection of point values onto the basis (Sec. 3.1, eq. u-exp inverted) in
// 3D. FP32 form: one axis at a time (dg_sf.cuh); one thread per (variable, cell)
// reduces the npts values along z, then y, then x to the moments of total degree <= d.
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
template <int DEG, int NP, bool GLM>
__global__ void __launch_bounds__(NTJ) k_project_sf(Geom g, const double* __restrict__ nodal,
                                                    const double* __restrict__ ldf, float* __restrict__ w,
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
    w[(int64_t)row * S + c] = (float)x;
    if (mean >= 0) wmean[(int64_t)mean * S + c] = x;
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
        put(5 * N + j, j < 3 ? 5 + j : -1, s * (double)(float)__ldg(ldf + NDIV * 3 * N + j));
      }
    });
  }
}

template <int DEG, int NP>
void run(const Geom& g, const double* nodal, const double* ldf, float* w, double* wmean, cudaStream_t st) {
  const unsigned nb = (unsigned)((g.ncell + 31) / 32);
  if (g.glm) k_project_sf<DEG, NP, true><<<nb, NTJ, 0, st>>>(g, nodal, ldf, w, wmean);
  else k_project_sf<DEG, NP, false><<<nb, NTJ, 0, st>>>(g, nodal, ldf, w, wmean);
}

// The dense projection with lanes over cells: a warp holds the rows of one
// Legendre variable, or 9 LDF rows, and takes the points in order; the weighted
// value of a point is formed once per warp instead of once per row, the loads are
// coalesced and the table's entries warp-uniform. Every row's sum is that of
// k_project, product by product (LDF: without the components that vanish), so
// FP64 states keep its bits: the TVB procedure takes square roots of differences
// that vanish where the transverse field does (a^2 - c_s^2 in alpha_f), so on
// such states the last bits of the initial means appear at 1e-8 after one step.
// Bound by the FP64 pipe. GB300, 96^3 cells, GLM, degree 2, 3 points: 8.2 ms the
// generic kernel, 4.0 ms this one (Powell: 21.5 and 4.1 ms).
template <typename T, int DEG, bool GLM>
__global__ void __launch_bounds__(128) k_project_rows(Geom g, int Qp, const double* __restrict__ tab,
                                                      const double* __restrict__ wq, const double* __restrict__ nodal,
                                                      const T* __restrict__ minv, T* __restrict__ w,
                                                      double* __restrict__ wmean) {
  constexpr int N = LdfPattern<DEG>::N, NDIV = LdfPattern<DEG>::NDIV, CH = 9;
  const int64_t S = g.stride;
  const int64_t c = (int64_t)blockIdx.x * 128 + threadIdx.x;
  const bool live = c < g.ncell;
  const double* f = nodal + (live ? c : 0);
  auto put = [&](int row, int mean, double acc) {
    acc *= (double)__ldg(minv + row);
    if (!live) return;
    w[(int64_t)row * S + c] = (T)acc;
    if (sizeof(T) == 4 && mean >= 0) wmean[(int64_t)mean * S + c] = acc;
  };
  const int unit = blockIdx.y;  // variable, then the chunks of LDF rows
  if (GLM || unit < 5) {
    double acc[N];
#pragma unroll
    for (int l = 0; l < N; ++l) acc[l] = 0.0;
    const double* t = tab + (size_t)unit * N * Qp * 3;
#pragma unroll 3
    for (int q = 0; q < Qp; ++q) {
      const double x = __ldg(wq + q) * f[(int64_t)(unit * Qp + q) * S];
#pragma unroll
      for (int l = 0; l < N; ++l) acc[l] = __fma_rn(x, __ldg(t + (size_t)(l * Qp + q) * 3), acc[l]);
    }
#pragma unroll
    for (int l = 0; l < N; ++l) put(unit * N + l, l == 0 ? unit : -1, acc[l]);
  } else if constexpr (!GLM) {
    sf::each<0, (NDIV + CH - 1) / CH>([&](auto K) {
      constexpr int j0 = decltype(K)::value * CH, n = NDIV - j0 < CH ? NDIV - j0 : CH;
      if (unit - 5 != decltype(K)::value) return;
      double acc[n];
#pragma unroll
      for (int i = 0; i < n; ++i) acc[i] = 0.0;
#pragma unroll 3
      for (int q = 0; q < Qp; ++q) {
        double x[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) x[k] = __ldg(wq + q) * f[(int64_t)((5 + k) * Qp + q) * S];
        sf::each<0, n>([&](auto I) {
          constexpr int i = decltype(I)::value;
          sf::each<0, 3>([&](auto CC) {
            constexpr int k = decltype(CC)::value;
            if constexpr (ldf_has<DEG>(j0 + i, k))
              acc[i] = __fma_rn(x[k], __ldg(tab + ((size_t)(5 * N + j0 + i) * Qp + q) * 3 + k), acc[i]);
          });
        });
      }
#pragma unroll
      for (int i = 0; i < n; ++i) put(5 * N + j0 + i, j0 + i < 3 ? 5 + j0 + i : -1, acc[i]);
    });
  }
}

template <typename T, int DEG>
void run_rows(const Geom& g, int Qp, const double* tab, const double* wq, const double* nodal, const T* minv, T* w,
              double* wmean, cudaStream_t st) {
  const unsigned nb = (unsigned)((g.ncell + 127) / 128);
  if (g.glm)
    k_project_rows<T, DEG, true><<<dim3(nb, 9), 128, 0, st>>>(g, Qp, tab, wq, nodal, minv, w, wmean);
  else
    k_project_rows<T, DEG, false><<<dim3(nb, 5 + (LdfPattern<DEG>::NDIV + 8) / 9), 128, 0, st>>>(
        g, Qp, tab, wq, nodal, minv, w, wmean);
}

}  // namespace

bool project_rows_ok(const Geom& g) { return g.D == 3 && g.d >= 1 && g.d <= 3; }

// FP32 form only: FP64 states keep the last bits of the dense sums
// (k_project_rows). With d + 1 up to d + 3 points per axis (Solver.project_ic's
// default), the counts initial states are given with, and degree 3 with 3; other
// counts run k_project_rows.
bool project_sf_ok(const Geom& g, int npts) {
  return project_rows_ok(g) && npts >= (g.d == 3 ? 3 : g.d + 1) && npts <= g.d + 3;
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

void launch_project_sf(const Geom& g, int npts, const double* nodal, const double* ldf, float* w, double* wmean,
                       cudaStream_t st) {
  switch (10 * g.d + npts) {
    case 12: run<1, 2>(g, nodal, ldf, w, wmean, st); break;
    case 13: run<1, 3>(g, nodal, ldf, w, wmean, st); break;
    case 14: run<1, 4>(g, nodal, ldf, w, wmean, st); break;
    case 23: run<2, 3>(g, nodal, ldf, w, wmean, st); break;
    case 24: run<2, 4>(g, nodal, ldf, w, wmean, st); break;
    case 25: run<2, 5>(g, nodal, ldf, w, wmean, st); break;
    case 33: run<3, 3>(g, nodal, ldf, w, wmean, st); break;
    case 34: run<3, 4>(g, nodal, ldf, w, wmean, st); break;
    case 35: run<3, 5>(g, nodal, ldf, w, wmean, st); break;
    case 36: run<3, 6>(g, nodal, ldf, w, wmean, st); break;
  }
}

// 3D, degrees 1-3 (Powell: with the LDF map's pattern); any number of points
template <typename T>
void launch_project_rows(const Geom& g, int npts, const double* tab, const double* wq, const double* nodal,
                         const T* minv, T* w, double* wmean, cudaStream_t st) {
  const int Qp = npts * npts * npts;
  if (g.d == 1) run_rows<T, 1>(g, Qp, tab, wq, nodal, minv, w, wmean, st);
  else if (g.d == 2) run_rows<T, 2>(g, Qp, tab, wq, nodal, minv, w, wmean, st);
  else run_rows<T, 3>(g, Qp, tab, wq, nodal, minv, w, wmean, st);
}
template void launch_project_rows<float>(const Geom&, int, const double*, const double*, const double*, const float*,
                                         float*, double*, cudaStream_t);
template void launch_project_rows<double>(const Geom&, int, const double*, const double*, const double*,
                                          const double*, double*, double*, cudaStream_t);

}  // namespace dgmhd
