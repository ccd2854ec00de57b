// Sparsity of the 3D LDF -> Legendre map (dg_fast.cuh PowTabs): which Legendre
// coefficients (component c, mode l) the LDF function j has, bit c * N + l of
// kLdf.m[j]. The curls of Legendre-product potentials touch few modes: 14 of
// 132 entries at degree 1, 38 of 780 at degree 2, 112 of 3000 at degree 3, so the kernels' forward and
// back maps skip the others at compile time. The tables are checked against
// this pattern when they are built (a basis with any other entry falls back to
// the generic kernels).
#pragma once
#include <cstdint>

namespace dgmhd {

template <int DEG>
struct LdfPattern;
template <>
struct LdfPattern<1> {
  static constexpr int N = 4, NDIV = 11;
  static constexpr uint32_t m(int j) {
    constexpr uint32_t t[NDIV] = {0x100, 0x10, 0x1, 0x200, 0x20, 0x400, 0x840, 0x80, 0x842, 0x4, 0x8};
    return t[j];
  }
};
template <>
struct LdfPattern<2> {
  static constexpr int N = 10, NDIV = 26;
  static constexpr uint32_t m(int j) {
    constexpr uint32_t t[NDIV] = {0x100000,   0x400,      0x1,     0x200000,  0x800,      0x400000,   0x801000,
                                  0x2000,     0x801002,   0x4,     0x8,       0x1000000,  0x4000,     0x2000000,
                                  0x4008000,  0x10000,    0x8000000, 0x10020000, 0x20040000, 0x80000, 0x4008010,
                                  0x10020020, 0x20040040, 0x80,    0x100,     0x200};
    return t[j];
  }
};
template <>
struct LdfPattern<3> {
  static constexpr int N = 20, NDIV = 50;
  static constexpr uint64_t m(int j) {
    constexpr uint64_t t[NDIV] = {
        0x10000000000,    0x100000,         0x1,              0x20000000000,    0x200000,         0x40000000000,
        0x80000400000,    0x800000,         0x80000400002,    0x4,              0x8,              0x100000000000,
        0x1000000,        0x200000000000,   0x400002000000,   0x4000000,        0x800000000000,   0x1000008000000,
        0x2000010000000,  0x20000000,       0x400002000010,   0x1000008000020,  0x2000010000040,  0x80,
        0x100,            0x200,            0x4000000000000,  0x40000000,       0x8000000000000,  0x10000080000000,
        0x100000000,      0x20000000000000, 0x40000200000000, 0x80000400000000, 0x800000000,      0x100000000000000,
        0x200081000400002, 0x400002000000000, 0xa00085000400002, 0x8000000000,  0xa10085080400402, 0x40000200000800,
        0x80000400001000, 0xa10085080402402, 0x400002000004000, 0xa1008508040a402, 0x10000,       0x20000,
        0x40000,          0x80000};
    return t[j];
  }
};
template <int DEG>
constexpr bool ldf_has(int j, int c, int l) {
  return (LdfPattern<DEG>::m(j) >> (c * LdfPattern<DEG>::N + l)) & 1u;
}
// functions with the coefficient (c, l)
template <int DEG>
constexpr int ldf_terms(int c, int l) {
  int n = 0;
  for (int j = 0; j < LdfPattern<DEG>::NDIV; ++j) n += ldf_has<DEG>(j, c, l) ? 1 : 0;
  return n;
}
// component c of function j is not identically zero
template <int DEG>
constexpr bool ldf_has(int j, int c) {
  return (LdfPattern<DEG>::m(j) >> (c * LdfPattern<DEG>::N)) & ((1u << LdfPattern<DEG>::N) - 1u);
}

}  // namespace dgmhd
