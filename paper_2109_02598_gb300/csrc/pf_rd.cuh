// The reaction and the Euler update of N coupled species on four sites, shared by the 2D and
// 3D kernels (so that both give the same bits for the same neighbour sums). Per site, in a fixed
// order: for each field acc = (D_i h^-2) * (neighbour sum - 2d u_i); for each monomial m
// (ascending) its value prod_j u_j^e by repeated multiplication (j ascending), then
// acc_i += K[i][m] * value (fma); finally u_i + dt acc_i (fma).
//
// The exponents are data, the same for every site. Loops over a monomial's factors with a
// choice of species in each cost three times the arithmetic (160 instructions a site for three
// species and seven monomials, most of them selects, loop control and instruction-cache misses).
// Instead the monomials of degree three or less, 35 in four species, are written out, each a
// product straight from the registers; the host gives a monomial's place among them
// (rd_places), a warp-uniform jump. One of higher degree has a loop per species. The monomials'
// loop is not unrolled, so the code is short. (Written out in the caller's order behind bit tests
// instead, with the rates in the constant bank: the same time in 3D, 2 % slower in 2D.) The 2D
// kernel, three species and seven monomials: 4096^2 190 -> 213 GLUPS, 2048^2 179 -> 195.
#pragma once

#include "pf_internal.h"

namespace pf {

// Places of a pair a <= b (of PF_MAX_FIELDS species) and a triple a <= b <= c among those of
// their degree.
constexpr int rd_pair(int a, int b) {
  int n = 0;
  for (int i = 0; i < a; ++i) n += PF_MAX_FIELDS - i;
  return n + b - a;
}
constexpr int rd_triple(int a, int b, int c) {
  int n = 0;
  for (int i = 0; i < a; ++i) n += (PF_MAX_FIELDS - i) * (PF_MAX_FIELDS - i + 1) / 2;
  for (int i = a; i < b; ++i) n += PF_MAX_FIELDS - i;
  return n + c - b;
}
static_assert(rd_pair(3, 3) == 9 && rd_triple(3, 3, 3) == 19, "10 pairs, 20 triples");

// u[f]: the state, ls[f]: the Laplacians' neighbour sums (before the factor), res[f]: the new
// state.
template <int NF>
__device__ __forceinline__ void rd_sites4(float4 (&u)[NF], const float4 (&ls)[NF],
                                          const RdParams& p, float4 (&res)[NF]) {
  float4 acc[NF];
#pragma unroll
  for (int i = 0; i < NF; ++i) acc[i] = mul4(p.D[i], ls[i]);
#pragma unroll 1
  for (int m = 0; m < p.nmono; ++m) {
    float4 v = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
    // (no code: else the compiler forms all the products before the loop, in 60 registers)
#pragma unroll
    for (int i = 0; i < NF; ++i)
      asm volatile("" : "+f"(u[i].x), "+f"(u[i].y), "+f"(u[i].z), "+f"(u[i].w));
    // cases of species past NF - 1 are never taken (their code repeats the last species')
#define PF_U(a) u[a < NF ? a : NF - 1]
#define PF_RD1(a) \
  case 1 + a: v = PF_U(a); break;
#define PF_RD2(a, b) \
  case 1 + PF_MAX_FIELDS + rd_pair(a, b): v = mul4(PF_U(a), PF_U(b)); break;
#define PF_RD3(a, b, c) \
  case 15 + rd_triple(a, b, c): v = mul4(mul4(PF_U(a), PF_U(b)), PF_U(c)); break;
    switch (p.place[m]) {
      case 0: break;
      PF_RD1(0) PF_RD1(1) PF_RD1(2) PF_RD1(3) PF_RD2(0, 0) PF_RD2(0, 1) PF_RD2(0, 2) PF_RD2(0, 3)
      PF_RD2(1, 1) PF_RD2(1, 2) PF_RD2(1, 3) PF_RD2(2, 2) PF_RD2(2, 3) PF_RD2(3, 3) PF_RD3(0, 0, 0)
      PF_RD3(0, 0, 1) PF_RD3(0, 0, 2) PF_RD3(0, 0, 3) PF_RD3(0, 1, 1) PF_RD3(0, 1, 2)
      PF_RD3(0, 1, 3) PF_RD3(0, 2, 2) PF_RD3(0, 2, 3) PF_RD3(0, 3, 3) PF_RD3(1, 1, 1)
      PF_RD3(1, 1, 2) PF_RD3(1, 1, 3) PF_RD3(1, 2, 2) PF_RD3(1, 2, 3) PF_RD3(1, 3, 3)
      PF_RD3(2, 2, 2) PF_RD3(2, 2, 3) PF_RD3(2, 3, 3) PF_RD3(3, 3, 3)
      default:
#pragma unroll
        for (int j = 0; j < NF; ++j)
#pragma unroll 1
          for (int e = (p.E[m] >> (2 * j)) & 3; e > 0; --e) v = mul4(v, u[j]);
    }
#undef PF_U
#undef PF_RD1
#undef PF_RD2
#undef PF_RD3
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      const float k = p.K[i][m];
      acc[i].x = __fmaf_rn(k, v.x, acc[i].x);
      acc[i].y = __fmaf_rn(k, v.y, acc[i].y);
      acc[i].z = __fmaf_rn(k, v.z, acc[i].z);
      acc[i].w = __fmaf_rn(k, v.w, acc[i].w);
    }
  }
#pragma unroll
  for (int i = 0; i < NF; ++i) res[i] = fma4(p.dt, acc[i], u[i]);
}

}  // namespace pf
