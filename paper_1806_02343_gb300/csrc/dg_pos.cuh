// FP32 positivity screen (Sec. 4.3), shared by the screen kernel of the
// limiter and the tiled learned indicator, which holds every row of its cells in
// registers already.
#pragma once
#include "dg_ctx.h"
#include "dg_ldf.cuh"
#include "dg_sf.cuh"

namespace dgmhd {

// row of the k-th mean (Legendre mode 0 of rho, m, E, psi; degree-0 LDF rows
// for B in the Powell form; the B_z mode 0 row in 2D)
__host__ __device__ __forceinline__ int screen_mean_row(const Geom& g, int k) {
  if (g.glm || k < 5) return k * g.n;
  if (g.D == 3) return g.ldf0 + (k - 5);
  return k < 7 ? g.ldf0 + (k - 5) : g.bz2d;
}

// Whether the FP32 tests below can be trusted with a cell of this density and
// energy: their products of two conserved variables (rho E, m^2, B^2) lose up to
// 1.2e-38 where they leave FP32's normal numbers, and with both above 1e-30, and
// their product, that stays below a hundredth of the tests' margins (1e-4 of the
// energy, times at least a hundredth of the density). Below it -- FP64 states in
// small units, or rows near the end of FP32's range -- every product may be zero
// whatever the pressure: such cells take the FP64 procedure.
__device__ __forceinline__ bool pos_range(float rho, float E) {
  constexpr float tiny = 1e-30f;
  return rho > tiny && E > tiny && rho * E > tiny;
}

// The end of pos_screen_rows: means mt and deviation bounds dv of the 8 variables
__device__ __forceinline__ bool pos_screen_bound(const PosScreen& ps, const float* mt, float* dv) {
  const float mg = 1e-4f;
#pragma unroll
  for (int v = 0; v < 8; ++v) dv[v] = dv[v] * (1.f + mg) + mg * fabsf(mt[v]);
  const float rlo = mt[0] - dv[0];
  if (rlo > ps.eps_rho * 2.f && pos_range(rlo, mt[4])) {
    float kin = 0.f, mag = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float mu = fabsf(mt[1 + i]) + dv[1 + i];
      const float bu = fabsf(mt[5 + i]) + dv[5 + i];
      kin += mu * mu;
      mag += bu * bu;
    }
    const float plo = ps.gm1 * (mt[4] - dv[4] - 0.5f * kin / rlo - 0.5f * mag);
    if (plo > ps.eps_p * 2.f + mg * fabsf(mt[4])) return true;
  }
  return false;
}

// Rigorous screen in FP32 from the float mirror of the means: |P_l| <= 1 and
// |phi_j,c| <= maxabs on the cell bound |u_v(x) - mean_v| by dev_v at every
// point; a relative margin 1e-4 covers the rounding of the bound itself. True:
// rho and p clear twice their floors everywhere and the cell needs no work.
// row(r) returns the cell's coefficient of row r.
template <typename Row>
__device__ __forceinline__ bool pos_screen_rows(const Geom& g, const PosScreen& ps, Row row) {
  float mt[8];
#pragma unroll
  for (int k = 0; k < 5; ++k) mt[k] = row(screen_mean_row(g, k));
  if (g.glm) {
#pragma unroll
    for (int k = 5; k < 8; ++k) mt[k] = row(screen_mean_row(g, k));
  } else {
    mt[5] = mt[6] = mt[7] = 0.f;
    for (int j = 0; j < g.D; ++j)
      for (int cc = 0; cc < g.D; ++cc) mt[5 + cc] += row(g.ldf0 + j) * ps.ldf_mean0[j * 3 + cc];
    if (g.bz2d >= 0) mt[7] = row(g.bz2d);
  }
  float dv[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  const int nlg = g.glm ? 8 : 5;
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    if (v >= nlg) continue;
    for (int l = 1; l < g.n; ++l) dv[v] += fabsf(row(v * g.n + l));
  }
  if (!g.glm) {
    for (int j = g.D; j < g.ndiv; ++j) {
      const float aj = fabsf(row(g.ldf0 + j));
#pragma unroll
      for (int cc = 0; cc < 3; ++cc)
        if (cc < g.D) dv[5 + cc] += aj * ps.ldf_maxabs[j * 3 + cc];
    }
    if (g.bz2d >= 0)
      for (int l = 1; l < g.n; ++l) dv[7] += fabsf(row(g.bz2d + l));
  }
  return pos_screen_bound(ps, mt, dv);
}

// Point-wise screen in FP32, 3D degrees 1 and 2: the state at every volume and
// face point of the cell, one axis at a time (planes of z, rows of y, points of
// x; on a plane or row through the cell's faces only the points that exist).
// True: the density clears its floor and the pressure of every point and of the
// mean clears its floor by more than the rounding, so the positivity procedure
// leaves the cell as it is. With S_v = |mean_v| + dev_v (dev: sum of
// |coefficients| x basis bound) every value carries at most about 30 roundings,
// 2e-6 S_v; a point is cleared with rho >= 0.1 S_rho and
//   rho (E - B^2/2 - eps_p/(g-1) - t (S_E + S_B^2/2)) >= m^2/2 + t S_m^2/2,
// t = 1e-4: at least four times what those roundings can move either side
// (pos_range: and what products near the end of FP32's range lose).
// A non-finite value clears nothing. coef(v, l): Legendre coefficient l of
// variable v (v < 8).
template <int DEG, typename Coef>
__device__ __forceinline__ bool pos_points_clear(Coef coef, const float (&mt)[8], const float (&dv)[8], float eps_rho,
                                                 float eps_p, float gm1) {
  constexpr int NQ = DEG + 1, NX = NQ + 2, M2 = sf::n_modes2(DEG);
  constexpr float t = 1e-4f;
  float S[8];
#pragma unroll
  for (int v = 0; v < 8; ++v) S[v] = fabsf(mt[v]) + dv[v];
  const float c1 = eps_p / gm1 + t * (S[4] + 0.5f * (S[5] * S[5] + S[6] * S[6] + S[7] * S[7]));
  const float c2 = 0.5f * t * (S[1] * S[1] + S[2] * S[2] + S[3] * S[3]);
  const float r0 = fmaxf(eps_rho + t * S[0], 0.1f * S[0]);
  bool ok = pos_range(S[0], S[4]);
  auto test = [&](const float (&u)[8]) {
    const float b2 = u[5] * u[5] + u[6] * u[6] + u[7] * u[7], m2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
    const float e = u[4] - 0.5f * b2 - c1;
    ok = ok && u[0] >= r0 && u[0] * e - 0.5f * m2 >= c2;
  };
  test(mt);
  auto node = [](int i) {  // -1, the Gauss points, +1
    constexpr float a = (float)sf::Rule<DEG>::x(0);
    return i == 0 ? -1.f : i == NX - 1 ? 1.f : i == 1 ? -a : i == NX - 2 ? a : 0.f;
  };
#pragma unroll 1
  for (int iz = 0; iz < NX; ++iz) {
    const float z = node(iz), z2 = 1.5f * z * z - 0.5f;
    const bool zin = iz > 0 && iz < NX - 1;
    float g[8][M2];
    sf::each<0, 8>([&](auto VI) {
      constexpr int v = decltype(VI)::value;
#pragma unroll
      for (int i = 0; i <= DEG; ++i)
#pragma unroll
        for (int j = 0; i + j <= DEG; ++j) {
          float x = coef(VI, i, j, 0);
          if (i + j + 1 <= DEG) x = fmaf(coef(VI, i, j, 1), z, x);
          if (i + j + 2 <= DEG) x = fmaf(coef(VI, i, j, 2), z2, x);
          g[v][sf::mode2_idx<DEG>(i, j)] = x;
        }
    });
#pragma unroll 1
    for (int iy = zin ? 0 : 1; iy < (zin ? NX : NX - 1); ++iy) {
      const float yy = node(iy), y2 = 1.5f * yy * yy - 0.5f;
      const bool in = zin && iy > 0 && iy < NX - 1;
      float h[8][DEG + 1];
#pragma unroll
      for (int v = 0; v < 8; ++v)
#pragma unroll
        for (int i = 0; i <= DEG; ++i) {
          float x = g[v][sf::mode2_idx<DEG>(i, 0)];
          if (i + 1 <= DEG) x = fmaf(g[v][sf::mode2_idx<DEG>(i, 1)], yy, x);
          if (i + 2 <= DEG) x = fmaf(g[v][sf::mode2_idx<DEG>(i, 2)], y2, x);
          h[v][i] = x;
        }
      auto point = [&](float x) {
        const float x2 = 1.5f * x * x - 0.5f;
        float u[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          u[v] = fmaf(h[v][1], x, h[v][0]);
          if (DEG >= 2) u[v] = fmaf(h[v][DEG >= 2 ? 2 : 0], x2, u[v]);
        }
        test(u);
      };
#pragma unroll
      for (int ix = 1; ix < NX - 1; ++ix) point(node(ix));
      if (in) {
        point(-1.f);
        point(1.f);
      }
    }
  }
  return ok;
}

// pos_points_clear from a cell's rows (LDF B through the sparse map)
template <int DEG, int GLMF, typename Row>
__device__ __forceinline__ bool pos_points_rows(Row row, const LdfLeg& ll, float eps_rho, float eps_p,
                                                const PosScreen& ps, float (&devt)[8]) {
  constexpr int N = LdfPattern<DEG>::N, NDIV = LdfPattern<DEG>::NDIV;
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    devt[v] = 0.f;
    if (GLMF || v < 5)
      for (int l = 1; l < N; ++l) devt[v] += fabsf(row(v * N + l));
  }
  if (!GLMF)
    for (int j = 3; j < NDIV; ++j) {
      const float aj = fabsf(row(5 * N + j));
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) devt[5 + cc] += aj * ps.ldf_maxabs[j * 3 + cc];
    }
  auto coef = [&](auto VI, int i, int j, int k) -> float {
    constexpr int v = decltype(VI)::value;
    const int l = sf::mode_idx(i, j, k);
    if constexpr (GLMF || v < 5) {
      return row(v * N + l);
    } else {
      float x = 0.f;
#pragma unroll
      for (int q = 0; q < NDIV; ++q)
        if (ldf_has<DEG>(q, v - 5, l)) x = fmaf(row(5 * N + q), ll.A[(q * 3 + v - 5) * N + l], x);
      return x;
    }
  };
  float mt[8];
  sf::each<0, 8>([&](auto VI) { mt[decltype(VI)::value] = coef(VI, 0, 0, 0); });
  return pos_points_clear<DEG>(coef, mt, devt, eps_rho, eps_p, ps.gm1);
}

// ballot compaction of a warp's cells into list[0 .. *count)
__device__ __forceinline__ void append_cells(bool mine, int64_t c, int32_t* __restrict__ list, unsigned* count) {
  const int lane = threadIdx.x & 31;
  const unsigned bal = __ballot_sync(0xffffffffu, mine);
  unsigned at = 0;
  if (lane == 0 && bal) at = atomicAdd(count, (unsigned)__popc(bal));
  at = __shfl_sync(0xffffffffu, at, 0);
  if (mine) list[at + __popc(bal & ((1u << lane) - 1u))] = (int32_t)c;
}

}  // namespace dgmhd
