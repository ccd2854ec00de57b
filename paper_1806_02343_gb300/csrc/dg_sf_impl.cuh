// FP64 operator on uniform 3D meshes, sum-factorised (dg_sf.cuh), for the GLM
// scheme (degrees 1-3) and the Powell scheme with the LDF basis (degrees 1, 2):
// one thread per (variable, cell), 32 consecutive cells per block, nine warps,
// one variable each, so that every branch on the variable is warp-uniform and
// global loads and stores are coalesced along the cells. Powell has eight
// variables: B is carried in the Legendre form of its components through the
// sparse map of dg_ldf.cuh; the ninth warp works on points only.
// Both kernels are bound by the FP64 pipe (2 operations per clock and SM).
// Measured on GB300, smooth GLM state, 45 x 40 x 36 cells, degree 2, per
// evaluation: face + cell 2.22 + 1.66 ms with dense contractions, 1.23 + 0.56
// now; Powell blast, 48^3 cells: 3.88 + 3.27 ms, 1.98 + 0.93 now.
#include <type_traits>

#include "dg_fast.cuh"
#include "dg_ldf.cuh"
#include "dg_sf.cuh"

#if !defined(DG_SF_DEG)
#error "include from a dg_sf_d<degree>.cu unit that defines DG_SF_DEG"
#endif

namespace dgmhd {

namespace {

using sf::V;
constexpr int NTS = 9 * 32;  // threads per block

template <int DEG>
struct SfDims {
  static constexpr int N = FastDims<DEG>::N, QF = FastDims<DEG>::QF, NQ = DEG + 1, QP = NQ * NQ;
  static constexpr int M2 = sf::n_modes2(DEG);  // moments of a face's flux
  static constexpr size_t face_smem = (size_t)2 * QF * 9 * 32 * sizeof(V);
  // cell kernel: planes of volume points per pass, slots per point
  static constexpr int PPP = DEG == 1 ? 2 : 1, NPASS = NQ / PPP, PQ = PPP * QP, NS = 22;
  // two buffers where two blocks still fit on an SM: the next plane's values need no barrier of their own
  static constexpr int NBUF = DEG == 2 ? 2 : 1;
  static constexpr size_t cell_smem = (size_t)NBUF * PQ * NS * 32 * sizeof(V);
};

// The values of the sparse LDF -> Legendre map and 1 / mass of the LDF rows
// (constant bank; the same for every context of this degree)
template <int DEG>
struct LdfTab {
  double A[LdfPattern<DEG>::NDIV][3][LdfPattern<DEG>::N];
  double minv[LdfPattern<DEG>::NDIV];
};
#if DG_SF_DEG <= 2
__constant__ LdfTab<DG_SF_DEG> c_ldf;
#endif

// Legendre coefficients of variable v of cell c: its own rows, or (Powell, v >=
// 5) component v - 5 of B from the LDF rows that contain it
template <int DEG, bool GLM>
__device__ __forceinline__ void sf_coefs(const V* __restrict__ w, int64_t S, int64_t c, int v,
                                         V (&x)[FastDims<DEG>::N]) {
  constexpr int N = FastDims<DEG>::N;
  if (GLM || v < 5) {
    const V* p = w + (int64_t)(v * N) * S + c;
#pragma unroll
    for (int l = 0; l < N; ++l, p += S) x[l] = *p;
  } else {
#if DG_SF_DEG <= 2
    const V* p = w + (int64_t)(5 * N) * S + c;
    auto comp = [&](auto CC) {
      constexpr int cc = decltype(CC)::value;
#pragma unroll
      for (int l = 0; l < N; ++l) x[l] = 0.0;
      sf::each<0, LdfPattern<DEG>::NDIV>([&](auto J) {
        constexpr int j = decltype(J)::value;
        if constexpr (ldf_has<DEG>(j, cc)) {
          const V wj = p[j * S];
          sf::each<0, N>([&](auto L) {
            constexpr int l = decltype(L)::value;
            if constexpr (ldf_has<DEG>(j, cc, l)) x[l] = __fma_rn(wj, c_ldf.A[j][cc][l], x[l]);
          });
        }
      });
    };
    if (v == 5) comp(std::integral_constant<int, 0>{});
    else if (v == 6) comp(std::integral_constant<int, 1>{});
    else if (v == 7) comp(std::integral_constant<int, 2>{});
#endif
  }
}

// cell coordinates and periodic neighbours (cell counts stay below 2^31)
struct Coord {
  int ix, iy, iz;
};
__device__ __forceinline__ Coord coord_of(const FastGeom& g, int64_t c) {
  const unsigned cc = (unsigned)c, nx = (unsigned)g.nx, ny = (unsigned)g.ny;
  const unsigned r = cc / nx;
  return Coord{(int)(cc - r * nx), (int)(r % ny), (int)(r / ny)};
}
__device__ __forceinline__ int64_t nbr(const FastGeom& g, Coord k, int a, int dir) {
  int& x = a == 0 ? k.ix : a == 1 ? k.iy : k.iz;
  const int n = a == 0 ? g.nx : a == 1 ? g.ny : g.nz;
  x += dir;
  x = x < 0 ? x + n : (x >= n ? x - n : x);
  return ((int64_t)k.iz * g.ny + k.iy) * g.nx + k.ix;
}

template <int DEG>
__device__ __forceinline__ void sf_trace(int A, bool plus, const V* c, V* tr) {
  constexpr int QF = FastDims<DEG>::QF;
  V g[sf::n_modes2(DEG)], u[QF];
  if (A == 0) sf::face_coefs<DEG, 0>(c, plus, g);
  else if (A == 1) sf::face_coefs<DEG, 1>(c, plus, g);
  else sf::face_coefs<DEG, 2>(c, plus, g);
  sf::expand2<DEG>(g, u);
#pragma unroll
  for (int p = 0; p < QF; ++p) tr[p * NTS] = u[p];
}

// Face fluxes, the three axes one after the other: traces of the left and the
// own cell (variable threads), HLLD and the GLM interface values (one face
// point per thread; one copy of the code, the axis rotates the shared-memory
// slots), then the flux's 2D moments of total degree <= d over the face
// (variable threads), which both neighbouring cells read: the surface
// contraction is done once per face instead of once per side.
// F[axis][moment][slot][cell], moments normalised as in sf::reduce1; slots:
// the nine variables (GLM), or the eight variables, then B^n_F minus the left
// and the right cell's own normal trace (Powell: the face term's jumps).
template <int DEG, bool GLM>
__global__ void __launch_bounds__(NTS, 2) k_sf_face(const FastGeom g, const V* __restrict__ w, V* __restrict__ F,
                                                    const DevScalars* __restrict__ sc, V eps) {
  using D = SfDims<DEG>;
  constexpr int N = D::N, QF = D::QF, M2 = D::M2, NV = GLM ? 9 : 8, NF = GLM ? 9 : 10;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* TR = reinterpret_cast<V*>(smraw);  // [2][QF][9][32]
  const int t = threadIdx.x, lane = t & 31, v = t >> 5;
  const int64_t S = g.stride;
  const int64_t cb = (int64_t)blockIdx.x * 32 + lane;
  const bool live = cb < g.ncell;
  const int64_t c = live ? cb : g.ncell - 1;  // dead lanes repeat the last cell and store nothing
  const Coord q = coord_of(g, c);
  const V ch = GLM ? sc->ch : 0.0;
  const V ich = GLM ? 1.0 / (2.0 * ch) : 0.0;
#pragma unroll 1
  for (int A = 0; A < 3; ++A) {
    if (v < NV) {
      V x[N];
      sf_coefs<DEG, GLM>(w, S, nbr(g, q, A, -1), v, x);
      sf_trace<DEG>(A, true, x, TR + t);
      sf_coefs<DEG, GLM>(w, S, c, v, x);
      sf_trace<DEG>(A, false, x, TR + QF * NTS + t);
    }
    __syncthreads();
    const int t1 = A == 2 ? 0 : A + 1, t2 = A == 0 ? 2 : A - 1;
    for (int p = v; p < QF; p += 9) {
      V* L = TR + p * NTS + lane;
      V* R = L + QF * NTS;
      const int sl[8] = {0, (1 + A) * 32, (1 + t1) * 32, (1 + t2) * 32, 4 * 32, (5 + A) * 32, (5 + t1) * 32, (5 + t2) * 32};
      V uL[8], uR[8], Fo[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        uL[k] = L[sl[k]];
        uR[k] = R[sl[k]];
      }
      const V bn = sf::hlld(uL, uR, g.gamma, eps, Fo);
      if constexpr (GLM) {  // interface values of Sec. 4.1.5
        const V pL = L[8 * 32], pR = R[8 * 32];
        Fo[5] = __fma_rn(0.5, pL + pR, -(0.5 * ch * (uR[5] - uL[5])));
        L[8 * 32] = ch * ch * __fma_rn(0.5, uL[5] + uR[5], -((pR - pL) * ich));
      } else {
        L[8 * 32] = bn - uL[5];
        R[8 * 32] = bn - uR[5];
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) L[sl[k]] = Fo[k];
    }
    __syncthreads();
    for (int s = v; s < NF; s += 9) {
      V f[QF], m[M2];
      const V* T = TR + (s == 9 ? QF * NTS + 8 * 32 : s * 32) + lane;
#pragma unroll
      for (int p = 0; p < QF; ++p) f[p] = T[p * NTS];
      sf::reduce2<DEG, DEG>(f, m);
      V* o = F + (int64_t)(A * M2 * NF + s) * S + c;
#pragma unroll
      for (int k = 0; k < M2; ++k, o += NF * S)
        if (live) *o = m[k];
    }
    __syncthreads();
  }
}

// slots of a volume point: 0 T_xx, 1-3 m, 4 E-flux x, 5-7 B, 8 psi (or zero),
// 9-13 T_xy T_xz T_yy T_yz T_zz, 14-15 E-flux y z, 16-18 A_xy A_xz A_yz,
// 19-21 their negatives; T = rho v v - B B + p_T, A_ij = B_i v_j - v_i B_j
enum { PS_TXX = 0, PS_M = 1, PS_EX = 4, PS_B = 5, PS_PSI = 8, PS_TXY = 9, PS_TXZ, PS_TYY, PS_TYZ, PS_TZZ, PS_EY,
       PS_EZ, PS_AXY, PS_AXZ, PS_AYZ, PS_NXY, PS_NXZ, PS_NYZ };
// where variable v finds its flux along x, y, z
__device__ __forceinline__ void flux_slots(int v, int& x, int& y, int& z) {
  switch (v) {
    case 0: x = PS_M; y = PS_M + 1; z = PS_M + 2; break;
    case 1: x = PS_TXX; y = PS_TXY; z = PS_TXZ; break;
    case 2: x = PS_TXY; y = PS_TYY; z = PS_TYZ; break;
    case 3: x = PS_TXZ; y = PS_TYZ; z = PS_TZZ; break;
    case 4: x = PS_EX; y = PS_EY; z = PS_EZ; break;
    case 5: x = PS_PSI; y = PS_AXY; z = PS_AXZ; break;
    case 6: x = PS_NXY; y = PS_PSI; z = PS_AYZ; break;
    case 7: x = PS_NXZ; y = PS_NYZ; z = PS_PSI; break;
    default: x = PS_B; y = PS_B + 1; z = PS_B + 2; break;  // psi: c_h^2 B_a, the factor at the end
  }
}

// fluxes of one volume point from its conserved values, in place: every flux
// component once per point (22 values for the nine variables)
template <bool GLM>
__device__ __forceinline__ void point_flux(V* pr, V gamma) {
  auto s = [&](int k) -> V& { return pr[k * 32]; };
  const V mx = s(1), my = s(2), mz = s(3), E = s(4), bx = s(5), by = s(6), bz = s(7);
  const V ir = 1.0 / s(0);
  const V vx = mx * ir, vy = my * ir, vz = mz * ir;
  const V b2 = __fma_rn(bx, bx, __fma_rn(by, by, bz * bz));
  const V ke2 = __fma_rn(mx, vx, __fma_rn(my, vy, mz * vz));
  const V p = (gamma - 1.0) * __fma_rn(-0.5, b2, __fma_rn(-0.5, ke2, E));
  const V pT = __fma_rn(0.5, b2, p);
  const V H = E + pT, vb = __fma_rn(vx, bx, __fma_rn(vy, by, vz * bz));
  s(PS_TXX) = __fma_rn(mx, vx, __fma_rn(-bx, bx, pT));
  s(PS_TXY) = __fma_rn(mx, vy, -bx * by);
  s(PS_TXZ) = __fma_rn(mx, vz, -bx * bz);
  s(PS_TYY) = __fma_rn(my, vy, __fma_rn(-by, by, pT));
  s(PS_TYZ) = __fma_rn(my, vz, -by * bz);
  s(PS_TZZ) = __fma_rn(mz, vz, __fma_rn(-bz, bz, pT));
  s(PS_EX) = __fma_rn(H, vx, -vb * bx);
  s(PS_EY) = __fma_rn(H, vy, -vb * by);
  s(PS_EZ) = __fma_rn(H, vz, -vb * bz);
  const V axy = __fma_rn(bx, vy, -by * vx), axz = __fma_rn(bx, vz, -bz * vx), ayz = __fma_rn(by, vz, -bz * vy);
  s(PS_AXY) = axy;
  s(PS_AXZ) = axz;
  s(PS_AYZ) = ayz;
  s(PS_NXY) = -axy;
  s(PS_NXZ) = -axz;
  s(PS_NYZ) = -ayz;
  if (!GLM) s(PS_PSI) = 0.0;
}

// Scale of mode (i, j, k)'s accumulated residual: the factor of the first
// term of its volume integral (see plane_moments); 1 for the mean.
template <int DEG>
constexpr __host__ __device__ double mode_scale(int i, int j, int k) {
  using sf::sig;
  return i > 0 ? (2 * i - 1) * sig<DEG>(i - 1) * sig<DEG>(j) * sig<DEG>(k)
       : j > 0 ? (2 * j - 1) * sig<DEG>(i) * sig<DEG>(j - 1) * sig<DEG>(k)
       : k > 0 ? (2 * k - 1) * sig<DEG>(i) * sig<DEG>(j) * sig<DEG>(k - 1)
               : 1.0;
}

// f(i, j, k, l) for the modes (l: their index) of total degree <= DEG
template <int DEG, typename F>
__device__ __forceinline__ void each_mode(F&& f) {
#pragma unroll
  for (int i = 0; i <= DEG; ++i)
#pragma unroll
    for (int j = 0; i + j <= DEG; ++j)
#pragma unroll
      for (int k = 0; i + j + k <= DEG; ++k) f(i, j, k, sf::mode_idx(i, j, k));
}

// one plane xi_z = node(Q) of the volume integral: fx, fy, fz = the plane's
// values of the variable's flux along each axis (point index x * NQ + y); racc
// in units of mode_scale. l_n' = sum of (2 m + 1) l_m over m = n-1, n-3, ...,
// so along x and y the moments below the mode's own degree enter, along z l_k'(z).
template <int DEG, int Q>
__device__ __forceinline__ void plane_moments(const V* fx, const V* fy, const V* fz, V* racc) {
  using sf::sig;
  constexpr int MD = DEG - 1;
  constexpr double z = sf::Rule<DEG>::node(Q), wz = sf::Rule<DEG>::w0() * sf::Rule<DEG>::wrel(Q);
  V m[sf::n_modes2(MD)];
  sf::reduce2<DEG, MD>(fx, m);
  each_mode<DEG>([&](int i, int j, int k, int l) {
#pragma unroll
    for (int n = i - 1; n >= 0; n -= 2)
      sf::axpy(racc[l], (2 * n + 1) * sig<DEG>(n) * sig<DEG>(j) * wz * sf::leg(k, z) / mode_scale<DEG>(i, j, k),
               m[sf::mode2_idx<MD>(n, j)]);
  });
  sf::reduce2<DEG, MD>(fy, m);
  each_mode<DEG>([&](int i, int j, int k, int l) {
#pragma unroll
    for (int n = j - 1; n >= 0; n -= 2)
      sf::axpy(racc[l], (2 * n + 1) * sig<DEG>(i) * sig<DEG>(n) * wz * sf::leg(k, z) / mode_scale<DEG>(i, j, k),
               m[sf::mode2_idx<MD>(i, n)]);
  });
  sf::reduce2<DEG, MD>(fz, m);
  each_mode<DEG>([&](int i, int j, int k, int l) {
    if (k > 0)
      sf::axpy(racc[l], sig<DEG>(i) * sig<DEG>(j) * wz * sf::dleg(k, z) / mode_scale<DEG>(i, j, k),
               m[sf::mode2_idx<MD>(i, j)]);
  });
}

// values on the plane xi_z = node(Q), u[x * NQ + y]
template <int DEG, int Q>
__device__ __forceinline__ void plane_values(const V* c, V* u) {
  constexpr double z = sf::Rule<DEG>::node(Q);
  V g[sf::n_modes2(DEG)];
#pragma unroll
  for (int i = 0; i <= DEG; ++i)
#pragma unroll
    for (int j = 0; i + j <= DEG; ++j) {
      V a = c[sf::mode_idx(i, j, 0)];
#pragma unroll
      for (int k = 1; i + j + k <= DEG; ++k) sf::axpy(a, sf::leg(k, z), c[sf::mode_idx(i, j, k)]);
      g[sf::mode2_idx<DEG>(i, j)] = a;
    }
  sf::expand2<DEG>(g, u);
}

// Volume integral of the thread's variable, plane by plane: values (variable
// threads), fluxes (one point per thread), moments (variable threads),
// exchanged through PR [NBUF][PQ][NS][32].
template <int DEG, bool GLM>
__device__ __forceinline__ void sf_volume(const V* wl, V* PR, V gamma, V* racc) {
  using D = SfDims<DEG>;
  constexpr int QP = D::QP, NS = D::NS, NV = GLM ? 9 : 8;
  const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;
  int sx, sy, sz;
  flux_slots(v, sx, sy, sz);
  sf::each<0, D::NPASS>([&](auto PASS) {
    constexpr int pass = decltype(PASS)::value;
    V* B = PR + (pass % D::NBUF) * D::PQ * NS * 32 + lane;
    if (D::NBUF == 1 && pass > 0) __syncthreads();
    if (v < NV) {
      sf::each<0, D::PPP>([&](auto I) {
        constexpr int q = decltype(I)::value;
        V u[QP];
        plane_values<DEG, pass * D::PPP + q>(wl, u);
#pragma unroll
        for (int p = 0; p < QP; ++p) B[((q * QP + p) * NS + v) * 32] = u[p];
      });
    }
    __syncthreads();
    for (int p = v; p < D::PQ; p += 9) point_flux<GLM>(B + p * NS * 32, gamma);
    __syncthreads();
    if (v < NV) {
      sf::each<0, D::PPP>([&](auto I) {
        constexpr int q = decltype(I)::value;
        V fx[QP], fy[QP], fz[QP];
#pragma unroll
        for (int p = 0; p < QP; ++p) fx[p] = B[((q * QP + p) * NS + sx) * 32];
#pragma unroll
        for (int p = 0; p < QP; ++p) fy[p] = B[((q * QP + p) * NS + sy) * 32];
#pragma unroll
        for (int p = 0; p < QP; ++p) fz[p] = B[((q * QP + p) * NS + sz) * 32];
        plane_moments<DEG, pass * D::PPP + q>(fx, fy, fz, racc);
      });
    }
  });
}

// adds the faces normal to axis A: m / p the moments of the -A and the +A face
template <int DEG, int A>
__device__ __forceinline__ void surface_axis(const V* m, const V* p, V* racc) {
  using sf::sig;
#pragma unroll
  for (int j = 0; j <= DEG; ++j)
#pragma unroll
    for (int k = 0; j + k <= DEG; ++k) {
      const int i2 = sf::mode2_idx<DEG>(j, k);
      const V even = m[i2] - p[i2], odd = m[i2] + p[i2];
#pragma unroll
      for (int n = 0; n + j + k <= DEG; ++n) {
        const int l = A == 0 ? sf::mode_idx(n, j, k) : A == 1 ? sf::mode_idx(j, n, k) : sf::mode_idx(j, k, n);
        if (l == 0) continue;  // the mean row is summed on its own
        const double sc = A == 0 ? mode_scale<DEG>(n, j, k) : A == 1 ? mode_scale<DEG>(j, n, k) : mode_scale<DEG>(j, k, n);
        const double f = sig<DEG>(j) * sig<DEG>(k) / sc;
        sf::axpy(racc[l], (n & 1) ? -f : f, (n & 1) ? odd : even);
      }
    }
}

// Cell update: volume integral, surface terms from the face moments, Powell's
// face term or the GLM damping, SSP combination (cmode 0: plain rhs, 1: ca ==
// 0, 2: ca != 0). The two cells of a face add the same stored moment with
// opposite signs, so their contributions to the means cancel exactly.
template <int DEG, bool GLM>
__global__ void __launch_bounds__(NTS, 2) k_sf_cell(const FastGeom g, const V* __restrict__ w,
                                                    const V* __restrict__ F, V* out, const V* w0, double ca,
                                                    double cb, int cmode, const DevScalars* __restrict__ sc) {
  // out may alias w0: each element is read, then written, by one thread.
  using D = SfDims<DEG>;
  constexpr int N = D::N, M2 = D::M2, NV = GLM ? 9 : 8, NF = GLM ? 9 : 10;
  constexpr double s00 = sf::sig<DEG>(0) * sf::sig<DEG>(0);
  extern __shared__ __align__(16) unsigned char smraw[];
  V* PR = reinterpret_cast<V*>(smraw);
  const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;  // warp-uniform variable
  const int64_t S = g.stride;
  const int64_t cbk = (int64_t)blockIdx.x * 32 + lane;
  const bool live = cbk < g.ncell;
  const int64_t c = live ? cbk : g.ncell - 1;  // dead lanes repeat the last cell and store nothing
  const Coord q = coord_of(g, c);
  const double dt = sc->dt;
  V wl[N], racc[N];
  if (v < NV) sf_coefs<DEG, GLM>(w, S, c, v, wl);
#pragma unroll
  for (int l = 0; l < N; ++l) racc[l] = 0.0;
  sf_volume<DEG, GLM>(wl, PR, g.gamma, racc);
  V qv = 0.0;  // Powell: q(<u>_K) = (0, B, v.B, v) of this variable from the cell means (Sec. 4.1.3)
  if (!GLM) {
    V* QM = PR;  // [8][32] the means
    __syncthreads();
    if (v < NV) QM[v * 32 + lane] = wl[0];
    __syncthreads();
    auto m = [&](int k) { return QM[k * 32 + lane]; };
    if (v >= 1 && v <= 3) qv = m(4 + v);
    else if (v == 4) qv = (m(1) * m(5) + m(2) * m(6) + m(3) * m(7)) / m(0);
    else if (v >= 5 && v < 8) qv = m(v - 4) / m(0);
  } else if (v == 8) {
    const V ch2 = sc->ch * sc->ch;
#pragma unroll
    for (int l = 1; l < N; ++l) racc[l] *= ch2;
  }
  V mean = 0.0;
  if (v < NV) {
    V fs[6];
    sf::each<0, 3>([&](auto AX) {
      constexpr int A = decltype(AX)::value;
      const int64_t cp = nbr(g, q, A, +1);
      V m[M2], p[M2];
      const V* f = F + (int64_t)(A * M2 * NF) * S;
#pragma unroll
      for (int k = 0; k < M2; ++k, f += NF * S) {
        m[k] = f[v * S + c];
        p[k] = f[v * S + cp];
        if (!GLM && v > 0) {  // this cell is the right one of its -A face, the left one of its +A face
          m[k] = __fma_rn(qv, f[9 * S + c], m[k]);
          p[k] = __fma_rn(qv, f[8 * S + cp], p[k]);
        }
      }
      surface_axis<DEG, A>(m, p, racc);
      fs[2 * A] = m[0];
      fs[2 * A + 1] = -p[0];
    });
    mean = (fs[0] + fs[1]) + (fs[2] + fs[3]) + (fs[4] + fs[5]);
  }
  const double tm = g.metric;
  // row r of the state (its stage input x) with residual rhs
  auto put = [&](int64_t r, V x, V rhs) {
    const int64_t i = r * S + c;
    if (!live) return;
    if (cmode != 0) {
      const V u = cb * __fma_rn(dt, rhs, x);
      rhs = cmode == 2 ? __fma_rn(ca, w0[i], u) : u;
    }
    out[i] = rhs;
  };
  if (GLM || v < 5) {
    const double kap = GLM && v == 8 ? sc->kappa : 0.0;
    put(v * N, wl[0], __fma_rn(-kap, wl[0], g.kmean * s00 * mean));
    each_mode<DEG>([&](int i, int j, int k, int l) {
      if (l > 0)
        put(v * N + l, wl[l],
            __fma_rn(-kap, wl[l], tm * (sf::mode_minv(i, j, k) * mode_scale<DEG>(i, j, k)) * racc[l]));
    });
  }
#if DG_SF_DEG <= 2
  if constexpr (!GLM) {
    // B: the residuals in Legendre form back to the LDF rows (the LDF functions
    // are the same polynomials: R_j = sum A[j][c][l] R[c][l]), rows spread over the warps
    V* RL = PR + 8 * 32;  // [3][N][32]
    if (v >= 5 && v < 8) {
      each_mode<DEG>([&](int i, int j, int k, int l) {
        RL[((v - 5) * N + l) * 32 + lane] = l == 0 ? s00 * mean : mode_scale<DEG>(i, j, k) * racc[l];
      });
    }
    __syncthreads();
    sf::each<0, LdfPattern<DEG>::NDIV>([&](auto J) {
      constexpr int j = decltype(J)::value;
      if (j % 9 == v) {
        V R = 0.0;
        sf::each<0, 3 * N>([&](auto I) {
          constexpr int cc = decltype(I)::value / N, l = decltype(I)::value % N;
          if constexpr (ldf_has<DEG>(j, cc, l)) R = __fma_rn(RL[(cc * N + l) * 32 + lane], c_ldf.A[j][cc][l], R);
        });
        put(5 * N + j, w[(int64_t)(5 * N + j) * S + c], tm * c_ldf.minv[j] * R);
      }
    });
  }
#endif
}

}  // namespace

template <int DEG, bool GLM>
void launch_sf_face(const FastGeom& g, const double* w, double* F, const DevScalars* sc, double eps, cudaStream_t st) {
  using D = SfDims<DEG>;
  raise_smem(k_sf_face<DEG, GLM>, D::face_smem);
  k_sf_face<DEG, GLM><<<(unsigned)((g.ncell + 31) / 32), NTS, D::face_smem, st>>>(g, w, F, sc, eps);
}

template <int DEG, bool GLM>
void launch_sf_cell(const FastGeom& g, const double* w, const double* F, double* out, const double* w0, double ca,
                    double cb, int combine, const DevScalars* sc, cudaStream_t st) {
  using D = SfDims<DEG>;
  raise_smem(k_sf_cell<DEG, GLM>, D::cell_smem);
  const int cmode = combine ? (ca != 0.0 ? 2 : 1) : 0;
  k_sf_cell<DEG, GLM><<<(unsigned)((g.ncell + 31) / 32), NTS, D::cell_smem, st>>>(g, w, F, out, w0, ca, cb, cmode, sc);
}

#define DG_SF_INST(GLM)                                                                                          \
  template void launch_sf_face<DG_SF_DEG, GLM>(const FastGeom&, const double*, double*, const DevScalars*, double, \
                                               cudaStream_t);                                                     \
  template void launch_sf_cell<DG_SF_DEG, GLM>(const FastGeom&, const double*, const double*, double*,           \
                                               const double*, double, double, int, const DevScalars*, cudaStream_t);
DG_SF_INST(true)
#if DG_SF_DEG <= 2
DG_SF_INST(false)

// copies the map to the constant bank (synchronous; 0 or -3)
template <int DEG>
int sf_ldf_to_constant(const PowTabs<double, DEG>& pt) {
  LdfTab<DEG> t;
  for (int j = 0; j < LdfPattern<DEG>::NDIV; ++j) {
    for (int cc = 0; cc < 3; ++cc)
      for (int l = 0; l < LdfPattern<DEG>::N; ++l) t.A[j][cc][l] = pt.Af[cc][j][l];
    t.minv[j] = pt.minvL[j];
  }
  return cudaMemcpyToSymbol(c_ldf, &t, sizeof(t)) == cudaSuccess ? 0 : -3;
}
template int sf_ldf_to_constant<DG_SF_DEG>(const PowTabs<double, DG_SF_DEG>&);
#endif

}  // namespace dgmhd
