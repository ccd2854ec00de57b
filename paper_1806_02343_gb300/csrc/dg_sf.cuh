// Sum-factorised pieces of the FP64 DG kernels (dg_sf_impl.cuh): the 1D
// Legendre <-> Gauss-point transforms they apply along one axis at a time (Sec.
// 3.1, 3.5) and the face flux (Sec. 4.1.2).
//
// Why: FP64 is bound by the number of its operations (GB300 does 2 FP64
// operations per clock and SM, 1/64 of FP32). A dense modal -> nodal
// contraction costs N multiply-adds per point (10 at degree 2). The basis is a
// product of 1D Legendre polynomials and the Gauss points are symmetric, so one
// axis at a time, with the even and odd parts shared by the points +x and -x, a
// degree-2 cell needs 66 operations for its 27 volume points (270 dense) and 22
// per face trace of 9 points (90 dense); the volume integral needs moments of
// total degree <= d - 1 only (about 160 operations against 324), and the
// surface integral 6 moments per face instead of 9 points in 10 modes.
// (The FP32 form keeps its dense contractions: another order of its roundings
// would move the FP64 cell means that it carries by 5e-9.)
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

namespace dgmhd {
namespace sf {

using V = double;

// ------------------------------------------------------------------ 1D rule
// Gauss-Legendre points of the (d + 1)-point rule: the positive ones x(i), i <
// NP, and 0 where the number is odd; weights relative to w(0), so that the
// normalised sums below start with a plain addition.
template <int DEG>
struct Rule {
  static_assert(DEG >= 1 && DEG <= 5, "2 to 6 points");
  static constexpr int NQ = DEG + 1, NP = NQ / 2;
  static constexpr bool MID = NQ & 1;
  static constexpr __host__ __device__ double x(int i) {
    return DEG == 1 ? 0.57735026918962576451
         : DEG == 2 ? 0.77459666924148337704
         : DEG == 3 ? (i == 0 ? 0.86113631159405257522 : 0.33998104358485626480)
         : DEG == 4 ? (i == 0 ? 0.90617984593866399280 : 0.53846931010568309104)
                    : (i == 0 ? 0.93246951420315202781 : i == 1 ? 0.66120938646626451366 : 0.23861918608319690863);
  }
  static constexpr __host__ __device__ double w(int i) {  // weight of x(i)
    return DEG == 1 ? 1.0
         : DEG == 2 ? 5.0 / 9.0
         : DEG == 3 ? (i == 0 ? 0.34785484513745385737 : 0.65214515486254614263)
         : DEG == 4 ? (i == 0 ? 0.23692688505618908751 : 0.47862867049936646804)
                    : (i == 0 ? 0.17132449237917034504 : i == 1 ? 0.36076157304813860757 : 0.46791393457269104739);
  }
  static constexpr __host__ __device__ double w0() { return w(0); }
  static constexpr __host__ __device__ double wr(int i) { return w(i) / w(0); }
  static constexpr __host__ __device__ double wm() { return (DEG == 2 ? 8.0 / 9.0 : 0.56888888888888888889) / w(0); }  // of the point 0
  // node of point index q: -x(0) first ... +x(0) last
  static constexpr __host__ __device__ double node(int q) {
    return (MID && q == NP) ? 0.0 : (q < NP ? -x(q) : x(NQ - 1 - q));
  }
  static constexpr __host__ __device__ double wrel(int q) {
    return (MID && q == NP) ? wm() : (q < NP ? wr(q) : wr(NQ - 1 - q));
  }
};
constexpr __host__ __device__ double leg(int k, double x) {
  return k == 0 ? 1.0 : k == 1 ? x : k == 2 ? 1.5 * x * x - 0.5 : (2.5 * x * x - 1.5) * x;
}
// derivative of l_k
constexpr __host__ __device__ double dleg(int k, double x) {
  return k == 0 ? 0.0 : k == 1 ? 1.0 : k == 2 ? 3.0 * x : 7.5 * x * x - 1.5;
}
// the 1D moment of order k, sum_q w_q l_k(x_q) f_q, is sig(k) times the
// normalised one of `reduce1` (whose first point enters with factor 1)
template <int DEG>
constexpr __host__ __device__ double sig(int k) {
  return Rule<DEG>::w0() * leg(k, Rule<DEG>::x(0));
}
// index of the Legendre mode (i, j, k) in the basis order
constexpr __host__ __device__ int mode_idx(int i, int j, int k) {
  const int g = i + j + k, t = g - i;
  return g * (g + 1) * (g + 2) / 6 + t * (t + 1) / 2 + k;
}
// 2D modes of total degree <= DEG in the order j along the first, k along the second tangential axis
template <int DEG>
constexpr __host__ __device__ int mode2_idx(int j, int k) {
  int n = 0;
  for (int a = 0; a < j; ++a) n += DEG + 1 - a;
  return n + k;
}
constexpr __host__ __device__ double mode_minv(int i, int j, int k) {  // 1 / mass of the Legendre mode
  return (2 * i + 1) * (2 * j + 1) * (2 * k + 1) / 8.0;
}
constexpr __host__ __device__ int n_modes2(int deg) { return (deg + 1) * (deg + 2) / 2; }
constexpr __host__ __device__ bool is_one(double x) { return x > 1.0 - 1e-13 && x < 1.0 + 1e-13; }
constexpr __host__ __device__ bool is_zero(double x) { return x > -1e-13 && x < 1e-13; }

// acc += f * x with f known at compile time (0, +-1 need no multiply)
__device__ __forceinline__ void axpy(V& acc, double f, V x) {
  if (is_zero(f)) return;
  if (is_one(f)) acc = acc + x;
  else if (is_one(-f)) acc = acc - x;
  else acc = __fma_rn(f, x, acc);
}

// values at the NQ points of sum_{k < K} c_k l_k
template <int DEG, int K>
__device__ __forceinline__ void expand1(const V* c, V* u) {
  using R = Rule<DEG>;
  if constexpr (K == 1) {
#pragma unroll
    for (int q = 0; q < R::NQ; ++q) u[q] = c[0];
  } else {
#pragma unroll
    for (int i = 0; i < R::NP; ++i) {
      const double x = R::x(i);
      V e = c[0];
      if constexpr (K > 2) e = __fma_rn(leg(2, x), c[2], e);
      if constexpr (K > 3) {
        V o = __fma_rn(leg(3, x), c[3], x * c[1]);
        u[i] = e - o;
        u[R::NQ - 1 - i] = e + o;
      } else {
        u[i] = __fma_rn(-x, c[1], e);
        u[R::NQ - 1 - i] = __fma_rn(x, c[1], e);
      }
    }
    if constexpr (R::MID) {
      u[R::NP] = c[0];
      if constexpr (K > 2) u[R::NP] = __fma_rn(leg(2, 0.0), c[2], c[0]);
    }
  }
}

// normalised moments m_k = sum_q w_q l_k(x_q) f_q / sig(k), k < K, of the values f[q]
template <int DEG, int K>
__device__ __forceinline__ void reduce1(const V* f, V* m) {
  using R = Rule<DEG>;
  V s[R::NP], d[R::NP];
#pragma unroll
  for (int i = 0; i < R::NP; ++i) {
    s[i] = f[R::NQ - 1 - i] + f[i];
    if constexpr (K > 1) d[i] = f[R::NQ - 1 - i] - f[i];
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    V a = (k & 1) ? d[0] : s[0];
#pragma unroll
    for (int i = 1; i < R::NP; ++i)
      axpy(a, R::wr(i) * leg(k, R::x(i)) / leg(k, R::x(0)), (k & 1) ? d[i] : s[i]);
    if constexpr (R::MID) {
      if (!(k & 1)) axpy(a, R::wm() * leg(k, 0.0) / leg(k, R::x(0)), f[R::NP]);
    }
    m[k] = a;
  }
}

// compile-time loop
template <int I, int N, typename F>
__device__ __forceinline__ void each(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    each<I + 1, N>(f);
  }
}

// 2D: coefficients g[mode2] of total degree <= DEG to the NQ x NQ points, u[i * NQ + j]
template <int DEG>
__device__ __forceinline__ void expand2(const V* g, V* u) {
  constexpr int NQ = DEG + 1;
  V h[NQ][DEG + 1];  // [first-axis point][second-axis mode]
  each<0, DEG + 1>([&](auto KK) {
    constexpr int k = decltype(KK)::value;
    V c[DEG + 1 - k], t[NQ];
#pragma unroll
    for (int j = 0; j + k <= DEG; ++j) c[j] = g[mode2_idx<DEG>(j, k)];
    expand1<DEG, DEG + 1 - k>(c, t);
#pragma unroll
    for (int i = 0; i < NQ; ++i) h[i][k] = t[i];
  });
#pragma unroll
  for (int i = 0; i < NQ; ++i) expand1<DEG, DEG + 1>(h[i], u + i * NQ);
}

// 2D normalised moments of total degree <= MD of the values f[(i * NQ + j)] into m (order mode2_idx<MD>)
template <int DEG, int MD>
__device__ __forceinline__ void reduce2(const V* f, V* m) {
  constexpr int NQ = DEG + 1;
  V r[MD + 1][NQ];  // [second-axis moment][first-axis point]
#pragma unroll
  for (int i = 0; i < NQ; ++i) {
    V t[MD + 1];
    reduce1<DEG, MD + 1>(f + i * NQ, t);
#pragma unroll
    for (int k = 0; k <= MD; ++k) r[k][i] = t[k];
  }
  each<0, MD + 1>([&](auto KK) {
    constexpr int k = decltype(KK)::value;
    V t[MD + 1 - k];
    reduce1<DEG, MD + 1 - k>(r[k], t);
#pragma unroll
    for (int j = 0; j + k <= MD; ++j) m[mode2_idx<MD>(j, k)] = t[j];
  });
}

// 2D coefficients, on the face xi_A = side (+-1), of a cell's Legendre field
template <int DEG, int A>
__device__ __forceinline__ void face_coefs(const V* c, bool plus, V* g) {
#pragma unroll
  for (int j = 0; j <= DEG; ++j)
#pragma unroll
    for (int k = 0; j + k <= DEG; ++k) {
      auto at = [&](int i) {
        return A == 0 ? c[mode_idx(i, j, k)] : A == 1 ? c[mode_idx(j, i, k)] : c[mode_idx(j, k, i)];
      };
      V e = at(0);
#pragma unroll
      for (int i = 2; i + j + k <= DEG; i += 2) e = e + at(i);
      if (1 + j + k <= DEG) {
        V o = at(1);
#pragma unroll
        for (int i = 3; i + j + k <= DEG; i += 2) o = o + at(i);
        e = plus ? e + o : e - o;
      }
      g[mode2_idx<DEG>(j, k)] = e;
    }
}

// ------------------------------------------------------------------ face flux
// HLLD flux of the rotated conserved traces u = (rho, m_n, m_t1, m_t2, E, B_n,
// B_t1, B_t2) (Miyoshi & Kusano 2005; the solver of Sec. 4.1.2), the scheme of
// dg_phys.cuh's `face_flux` with fewer FP64 operations (about 340 per point
// against 490; every division and square root costs about nine):
// * one division for 1 / rho of both sides and one for the four star-state
//   denominators (products of the operands: they stay in range for densities
//   and speeds whose fourth powers do), one square root for the larger fast speed;
// * each side's energy with B_n = B^n_F is its own plus (B^n_F^2 - B_n^2) / 2
//   (its pressure is kept), and the fast-speed discriminant is
//   (a^2 - b^2)^2 + 4 a^2 b_t^2, a sum of squares;
// * the upwind side of the contact is selected before the flux is assembled;
//   the two jump terms carry the wave speeds clipped at zero. In a supersonic
//   state the star terms are dropped by selection (they may be anything), and
//   the outer wave speeds alone select the side: without pressure and field
//   S_L = S_R, and S_M is 0 / 0 or noise.
// Writes the rotated flux (F[5] = 0) and returns B^n_F.
__device__ __forceinline__ V vmin(V a, V b) { return a < b ? a : b; }
__device__ __forceinline__ V vmax(V a, V b) { return a > b ? a : b; }
// x > 0 (and not NaN) from the upper word, off the FP64 pipe; false for subnormal x
__device__ __forceinline__ bool positive(V x) { return (unsigned)(__double2hiint(x) - 1) < 0x7ff00000u; }

__device__ __forceinline__ V hlld(const V* uL, const V* uR, V gamma, V eps, V* F) {
  const V rL = uL[0], rR = uR[0];
  const V ir = 1.0 / (rL * rR);
  // B^n_F of eq. bxface-average
  const V sL = rsqrt(rL), sR = rsqrt(rR);
  const V bn = __fma_rn(uL[5], sL, uR[5] * sR) / (sL + sR);
  const V bn2 = bn * bn;
  struct Side {
    V u, v, w, E, pT, cf2;
  } l, r;
  auto side = [&](const V* q, V ir1, Side& s) {
    s.u = q[1] * ir1;
    s.v = q[2] * ir1;
    s.w = q[3] * ir1;
    const V ke2 = __fma_rn(q[3], s.w, __fma_rn(q[2], s.v, q[1] * s.u));
    const V bt2 = __fma_rn(q[7], q[7], q[6] * q[6]);
    const V bo2 = q[5] * q[5];
    const V p = (gamma - 1.0) * __fma_rn(-0.5, bt2 + bo2, __fma_rn(-0.5, ke2, q[4]));
    const V b2 = bt2 + bn2;
    s.E = __fma_rn(0.5, bn2 - bo2, q[4]);
    s.pT = __fma_rn(0.5, b2, p);
    const V a2 = gamma * p * ir1, bb = b2 * ir1;
    const V df = a2 - bb;
    const V disc = vmax(__fma_rn(4.0 * a2, bt2 * ir1, df * df), 0.0);
    s.cf2 = 0.5 * (a2 + bb + sqrt(disc));
  };
  side(uL, ir * rR, l);
  side(uR, ir * rL, r);
  const V cm = sqrt(vmax(l.cf2, r.cf2));
  const V SL = vmin(l.u, r.u) - cm, SR = vmax(l.u, r.u) + cm;
  const V dL = SL - l.u, dR = SR - r.u;
  const V mL = rL * dL, mR = rR * dR;
  const V iden = 1.0 / (mR - mL);
  const V SM = __fma_rn(-mL, l.u, __fma_rn(mR, r.u, l.pT - r.pT)) * iden;
  const V pTs = __fma_rn(-mL, r.pT, __fma_rn(mL * mR, r.u - l.u, mR * l.pT)) * iden;
  const V eL = SL - SM, eR = SR - SM;
  const V qL = mL * eL, qR = mR * eR;
  V ddL = qL - bn2, ddR = qR - bn2;
  const bool gL = fabs(ddL) < eps * (fabs(qL) + bn2), gR = fabs(ddR) < eps * (fabs(qR) + bn2);
  // 1 / (eL eR ddL ddR) once; a degenerate side's denominator is replaced by 1
  ddL = gL ? 1.0 : ddL;
  ddR = gR ? 1.0 : ddR;
  const V e = eL * eR, d = ddL * ddR;
  const V t = 1.0 / (e * d), td = t * d, te = t * e;
  const V ieL = td * eR, ieR = td * eL, iL = te * ddR, iR = te * ddL;
  const V rsL = mL * ieL, rsR = mR * ieR;
  const V fvL = gL ? 0.0 : bn * (l.u - SM) * iL, fbL = gL ? 1.0 : __fma_rn(mL, dL, -bn2) * iL;
  const V fvR = gR ? 0.0 : bn * (r.u - SM) * iR, fbR = gR ? 1.0 : __fma_rn(mR, dR, -bn2) * iR;
  const V vL = __fma_rn(uL[6], fvL, l.v), wL = __fma_rn(uL[7], fvL, l.w), yL = uL[6] * fbL, zL = uL[7] * fbL;
  const V vR = __fma_rn(uR[6], fvR, r.v), wR = __fma_rn(uR[7], fvR, r.w), yR = uR[6] * fbR, zR = uR[7] * fbR;
  const V iqL = rsqrt(rsL), iqR = rsqrt(rsR);
  const V sqL = rsL * iqL, sqR = rsR * iqR;
  const V abn = fabs(bn);
  const V SsL = __fma_rn(-abn, iqL, SM), SsR = __fma_rn(abn, iqR, SM);
  // the double-starred tangential state (common to both sides of the contact)
  const V sgn = bn >= 0.0 ? 1.0 : -1.0;
  const V inv = 1.0 / (sqL + sqR);
  const V qs = sqL * sqR * sgn;
  const V vss = __fma_rn(sqL, vL, __fma_rn(sqR, vR, (yR - yL) * sgn)) * inv;
  const V wss = __fma_rn(sqL, wL, __fma_rn(sqR, wR, (zR - zL) * sgn)) * inv;
  const V yss = __fma_rn(sqL, yR, __fma_rn(sqR, yL, (vR - vL) * qs)) * inv;
  const V zss = __fma_rn(sqL, zR, __fma_rn(sqR, zL, (wR - wL) * qs)) * inv;
  const bool superL = positive(SL), superR = positive(-SR);
  const bool left = superL | (!superR & (SM >= 0.0));  // (short-circuit operators: 3% slower passes)
  auto pick = [&](V a, V b) { return left ? a : b; };
  const V xr = pick(rL, rR), xu = pick(l.u, r.u), xv = pick(l.v, r.v), xw = pick(l.w, r.w);
  const V xy = pick(uL[6], uR[6]), xz = pick(uL[7], uR[7]), xE = pick(l.E, r.E), xp = pick(l.pT, r.pT);
  const V xm = pick(uL[1], uR[1]), xm2 = pick(uL[2], uR[2]), xm3 = pick(uL[3], uR[3]);
  const V xd = pick(dL, dR), xi = pick(ieL, ieR), xrs = pick(rsL, rsR);
  const V xvs = pick(vL, vR), xws = pick(wL, wR), xys = pick(yL, yR), xzs = pick(zL, zR);
  const V xq = pick(sqL, -sqR);
  const bool super = left ? superL : superR;
  // clipped at zero: the outer speed of a side that is not supersonic has its sign already
  const V S1 = pick(SL, SR), Ss = pick(SsL, SsR);
  const V S2 = (__double2hiint(Ss) < 0) == left ? Ss : 0.0;
  const V vb = __fma_rn(xu, bn, __fma_rn(xv, xy, xw * xz));
  const V vbs = __fma_rn(SM, bn, __fma_rn(xvs, xys, xws * xzs));
  const V vbss = __fma_rn(SM, bn, __fma_rn(vss, yss, wss * zss));
  // (d E - pT u + pT* S_M + B_n (vb - vb*)) / (S - S_M)
  const V Es = __fma_rn(bn, vb - vbs, __fma_rn(pTs, SM, __fma_rn(xd, xE, -(xp * xu)))) * xi;
  const V dEs = xq * (vbss - vbs) * sgn;  // E** - E*
  auto add = [&](V f, V j1, V j2) { return super ? f : __fma_rn(S2, j2, __fma_rn(S1, j1, f)); };
  auto add1 = [&](V f, V j1) { return super ? f : __fma_rn(S1, j1, f); };
  F[0] = add1(xm, xrs - xr);
  F[1] = add1(__fma_rn(xm, xu, xp - bn2), __fma_rn(xrs, SM, -xm));
  F[2] = add(__fma_rn(xm, xv, -(bn * xy)), __fma_rn(xrs, xvs, -xm2), xrs * (vss - xvs));
  F[3] = add(__fma_rn(xm, xw, -(bn * xz)), __fma_rn(xrs, xws, -xm3), xrs * (wss - xws));
  F[4] = add(__fma_rn(xE + xp, xu, -(bn * vb)), Es - xE, dEs);
  F[5] = 0.0;
  F[6] = add(__fma_rn(xy, xu, -(bn * xv)), xys - xy, yss - xys);
  F[7] = add(__fma_rn(xz, xu, -(bn * xw)), xzs - xz, zss - xzs);
  return bn;
}

}  // namespace sf
}  // namespace dgmhd
