// Conservative detector in front of the TVB procedure (Sec. 4.2): whether the
// procedure can change a slope of the cell, in FP32 and with a margin, so that
// the procedure itself (dg_limit.cu `tvb_cell`, unchanged) runs only on the few
// cells this cannot exclude, in full warps. 3D degrees 1 and 2.
#pragma once
#include "dg_ctx.h"
#include "dg_sf.cuh"

namespace dgmhd {

// The procedure changes a slope of axis a only where a characteristic amplitude
// c of the slope exceeds thr and minmod(c, beta c+, beta c-) differs from c. The
// amplitudes here and there are the same expressions of the same means and
// slopes, rounded differently. Two errors are allowed for (TvbAmp::e): of the
// eigenvector weights, kTvbWeight times the terms of the amplitude with the
// weights bounded by 1 -- alpha_f,s = sqrt((a^2 - c_s^2) / (c_f^2 - c_s^2)) has
// a radicand with an absolute error of about 1.3e-4 at the limits of `fine`
// (speeds 5% apart, pressure 3% of the energy), so 1.2e-2 --, and of the
// primitive increments, kTvbRound (some 100 roundings) times the absolute values
// of the terms they are the differences of. Nearer to a degeneracy (c_f ~ c_s,
// or a transverse field near zero) only the direction-free bounds b are used.
// Where c_f ~ c_s (gap c_f^2 - c_s^2 below kTvbGap c_f^2), b allows for weights
// above 1 as well: the procedure takes any gap above rel c_f^2, and near a = c_A
// without a transverse field the gap is what the rounding of its radicand leaves,
// so that alpha^2 = (1 +- (a^2 - b^2) / gap) / 2 reaches (1 + 4 sqrt(eps) / rel) / 2:
// weights up to 22 in FP32 (eps = 6e-8, rel = 1e-6; 11 seen), 150 in FP64 (1.1e-16,
// 1e-12). At kTvbGap they are 1 to 0.2%.
constexpr float kTvbWeight = 2e-2f, kTvbRound = 1e-5f, kTvbGap = 2e-2f;
template <typename T>
constexpr float kTvbWide = sizeof(T) == 4 ? 32.f : 256.f;

template <int GLMF>
struct TvbAmp {
  float c[9];              // amplitudes
  float b[9], e[9];        // upper bounds for any direction of the transverse field, errors
};

// The error terms hold while increments down to the FP64 rounding of the means
// (1e-16 of them) are normal FP32 numbers: FP64 states whose density or energy is
// outside 1e-15 .. 1e15 leave every cell to the procedure.
template <typename T>
__device__ __forceinline__ bool tvb_range(const float (&m)[9]) {
  constexpr float lo = 1e-15f, hi = 1e15f;
  return sizeof(T) == 4 || (m[0] > lo && m[0] < hi && m[4] > lo && m[4] < hi);
}

__device__ __forceinline__ float tvb_sqrt(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float tvb_rcp(float x) { return __fdividef(1.f, x); }

template <int GLMF>
struct TvbEig {
  float rho, ir, isr, a2i, v[3], B[3], gm1, ich;
  float cf, cs, af, as, by, bz, sgn, isra;
  float wmax;       // bound of the weights
  bool sane, fine;  // the pressure keeps its leading digits; away from the degeneracies
};

template <int A, int GLMF>
__device__ __forceinline__ void tvb_eig(const float (&m)[9], float gamma, float ch, float wide, TvbEig<GLMF>& e) {
  constexpr int T1 = (A + 1) % 3, T2 = (A + 2) % 3;
  e.rho = m[0];
  e.ir = tvb_rcp(m[0]);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    e.v[i] = m[1 + i] * e.ir;
    e.B[i] = m[5 + i];
  }
  e.gm1 = gamma - 1.f;
  e.ich = GLMF ? tvb_rcp(ch) : 0.f;
  const float bt2 = e.B[T1] * e.B[T1] + e.B[T2] * e.B[T2], bn2 = e.B[A] * e.B[A];
  const float p = e.gm1 * (m[4] - 0.5f * m[0] * (e.v[0] * e.v[0] + e.v[1] * e.v[1] + e.v[2] * e.v[2]) - 0.5f * (bt2 + bn2));
  const float a2 = gamma * p * e.ir, b2 = (bt2 + bn2) * e.ir;
  const float disc = tvb_sqrt(fmaxf((a2 + b2) * (a2 + b2) - 4.f * a2 * bn2 * e.ir, 0.f));
  const float cf2 = 0.5f * (a2 + b2 + disc), cs2 = fmaxf(0.5f * (a2 + b2 - disc), 0.f);
  e.a2i = tvb_rcp(a2);
  e.isr = rsqrtf(m[0]);
  e.isra = e.isr * rsqrtf(a2);
  e.cf = tvb_sqrt(cf2);
  e.cs = tvb_sqrt(cs2);
  const float bt = tvb_sqrt(bt2), id = tvb_rcp(cf2 - cs2), ibt = tvb_rcp(bt);
  e.wmax = cf2 - cs2 > kTvbGap * cf2 ? 1.f : wide;
  e.sane = p > 1e-4f * m[4];
  e.fine = cf2 - cs2 > 0.05f * cf2 && bt > 1e-3f * tvb_sqrt(m[0] * cf2) && p > 0.03f * m[4];
  e.af = tvb_sqrt(fmaxf(a2 - cs2, 0.f) * id);
  e.as = tvb_sqrt(fmaxf(cf2 - a2, 0.f) * id);
  e.by = e.B[T1] * ibt;
  e.bz = e.B[T2] * ibt;
  e.sgn = e.B[A] >= 0.f ? 1.f : -1.f;
}

// amplitudes of a conserved increment with their bounds and errors. CAST: the
// increment is a difference of means m rounded to FP32 beforehand (FP64 states),
// off by up to 1.2e-7 |m| more. (FP64 differences rounded afterwards need no such
// term, but their FP64 operations made a pass 13.6 -> 19.0 us on 21^3 cells; with
// the term 16.0 us.)
template <int A, bool CAST, int GLMF>
__device__ __forceinline__ void tvb_amp(const TvbEig<GLMF>& e, const float (&d)[9], const float (&m)[9],
                                        TvbAmp<GLMF>& o) {
  constexpr int T1 = (A + 1) % 3, T2 = (A + 2) % 3;
  // the magnitudes that kTvbRound applies to
  auto s = [&](int k) { return CAST ? fmaf(1.5e-7f / kTvbRound, fabsf(m[k]), fabsf(d[k])) : fabsf(d[k]); };
  const float dr = d[0], du = (d[1 + A] - e.v[A] * dr) * e.ir, dv = (d[1 + T1] - e.v[T1] * dr) * e.ir,
              dw = (d[1 + T2] - e.v[T2] * dr) * e.ir;
  const float ke = 0.5f * (e.v[0] * e.v[0] + e.v[1] * e.v[1] + e.v[2] * e.v[2]);
  float dp = ke * dr + d[4], sp = ke * s(0) + s(4);
  float su = (s(1 + A) + fabsf(e.v[A]) * s(0)) * e.ir, st = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    dp -= e.v[i] * d[1 + i] + e.B[i] * d[5 + i];
    sp += fabsf(e.v[i]) * s(1 + i) + fabsf(e.B[i]) * s(5 + i);
    if (i != A) st += (s(1 + i) + fabsf(e.v[i]) * s(0)) * e.ir;
  }
  dp *= e.gm1;
  sp *= e.gm1;
  const float dby = d[5 + T1], dbz = d[5 + T2];
  const float vpar = e.by * dv + e.bz * dw, bpar = e.by * dby + e.bz * dbz;
  const float vperp = e.by * dw - e.bz * dv, bperp = e.by * dbz - e.bz * dby;
  const float h = 0.5f * e.a2i, pr = 0.5f * dp * e.ir * e.a2i, br = 0.5f * bpar * e.isra;
  const float f1 = h * (e.af * e.cf * du - e.as * e.cs * e.sgn * vpar), f2 = e.af * pr + e.as * br;
  const float s1 = h * (e.as * e.cs * du + e.af * e.cf * e.sgn * vpar), s2 = e.as * pr - e.af * br;
  o.c[0] = f2 - f1;
  o.c[6] = f2 + f1;
  o.c[2] = s2 - s1;
  o.c[4] = s2 + s1;
  o.c[1] = 0.5f * (vperp + e.sgn * bperp * e.isr);
  o.c[5] = 0.5f * (vperp - e.sgn * bperp * e.isr);
  o.c[3] = dr - dp * e.a2i;
  const float nv = fabsf(dv) + fabsf(dw), nb = fabsf(dby) + fabsf(dbz), sb = s(5 + T1) + s(5 + T2);
  const float wf = h * e.cf * (fabsf(du) + nv) + 0.5f * (fabsf(dp) * e.ir * e.a2i + nb * e.isra);
  const float rf = h * e.cf * (su + st) + 0.5f * (sp * e.ir * e.a2i + sb * e.isra);
  const float ef = kTvbWeight * wf + kTvbRound * rf;
#pragma unroll
  for (int k = 0; k < 7; k += 2) {
    o.b[k] = e.wmax * wf + ef;
    o.e[k] = ef;
  }
  const float wa = 0.5f * (nv + nb * e.isr), ea = kTvbWeight * wa + kTvbRound * 0.5f * (CAST ? st + sb * e.isr : st);
  o.b[1] = o.b[5] = wa + ea;
  o.e[1] = o.e[5] = ea;
  // the entropy wave has no weights: rounding, and a^2's own error (3e-3 at the limit of `sane`)
  o.e[3] = kTvbRound * (s(0) + sp * e.a2i) + 5e-3f * fabsf(dp) * e.a2i;
  o.b[3] = fabsf(o.c[3]) + o.e[3];
  if constexpr (GLMF) {
    o.c[7] = 0.5f * (d[5 + A] - d[8] * e.ich);
    o.c[8] = 0.5f * (d[5 + A] + d[8] * e.ich);
    o.e[7] = o.e[8] = kTvbRound * (s(5 + A) + s(8) * fabsf(e.ich));
    o.b[7] = fabsf(o.c[7]) + o.e[7];
    o.b[8] = fabsf(o.c[8]) + o.e[8];
  } else {
    o.c[7] = d[5 + A];
    o.e[7] = kTvbRound * s(5 + A);
    o.b[7] = fabsf(o.c[7]) + o.e[7];
  }
}

// Axis A cannot trigger: every amplitude of the slopes `sl` stays below thr, or
// both neighbour differences (dp, dm: loaded by `diffs` where needed) clear it.
// T: the procedure's precision.
template <typename T, int A, int GLMF, typename Diffs>
__device__ __forceinline__ bool tvb_axis_clear(const float (&m)[9], const float (&sl)[9], float gamma, float ch,
                                               float thr, float beta, Diffs diffs) {
  TvbEig<GLMF> e;
  tvb_eig<A>(m, gamma, ch, kTvbWide<T>, e);
  if (!e.sane) return false;
  TvbAmp<GLMF> x;
  tvb_amp<A, false>(e, sl, m, x);
  constexpr int V = GLMF ? 9 : 8;
  bool below = true;
#pragma unroll
  for (int k = 0; k < V; ++k) below = below && x.b[k] < thr;
  if (below) return true;
  if (!e.fine) return false;
  below = true;
#pragma unroll
  for (int k = 0; k < V; ++k) below = below && fabsf(x.c[k]) + x.e[k] < thr;
  if (below) return true;
  float dpl[9], dmi[9];
  diffs(dpl, dmi);
  TvbAmp<GLMF> p, q;
  tvb_amp<A, sizeof(T) == 8>(e, dpl, m, p);
  tvb_amp<A, sizeof(T) == 8>(e, dmi, m, q);
  bool ok = true;
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const float a = fabsf(x.c[k]) + x.e[k];
    const float sg = x.c[k] < 0.f ? -1.f : 1.f;
    ok = ok && (a < thr || (beta * (sg * p.c[k] - p.e[k]) >= a && beta * (sg * q.c[k] - q.e[k]) >= a));
  }
  return ok;
}

}  // namespace dgmhd
