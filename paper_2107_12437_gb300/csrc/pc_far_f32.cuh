// The field of a dipole far from it, to first order in the charges' separation: what the difference
// form of pc_lw_f32.cuh (dipole_pair) becomes when the separation s is so small against the distance
// R, and the charges so slow, that the terms it drops lie below float32 rounding.
//
// The net field q [F(x+) - F(x-)] of two charges at R_j + sigma s p / 2 (sigma = +-1) is odd in sigma
// for equal masses: s d' d'' enter linearly and then cubed.  The linear part is evaluated at one
// retarded time, the centre's, on the samples of (X, V, A) = (d/(qL), d'/(qc), d'' dt/(qc)) there,
//   E   = (rho.p) (3 X/R^5 + 3 V/R^4 + A/R^3) rho - (X/R^3 + V/R^2 + A/R) p
//   B   = (V/R^3 + A/R^2) (p x rho)        phi = (rho.p) (X/R^3 + V/R^2)       A = (V/R) p
// (units of dipole_pair; the Coulomb field of E and B has the X and V terms, the radiation field the
// A terms).  The relative size of the dropped terms, measured against both charges in extended
// precision over all directions and phases, is at most 1.0 (X/R)^2 + 2.5 V^2 of the sum of the
// terms' magnitudes.  With kFarX = X/R and kFarV = V at their largest that is 4e-8 + 3.6e-8, about
// one rounding of float32 (6e-8).  Unequal masses leave even terms, of relative size
// |mu+ - mu-| max(X/R, V), which have to stay below kFarAsym.
#pragma once
#include "pc_lw_f32x2.cuh"

namespace pc {

constexpr float kFarX = 2e-4f;
constexpr float kFarV = 1.2e-4f;
constexpr float kFarAsym = 2e-8f;

// The smallest distance (c dt) at which a dipole whose moments stay within |X| <= xmax, |V| <= vmax is
// far; infinite where no distance is.  Written so that a NaN gives infinity.
__device__ __forceinline__ float far_limit(float xmax, float vmax, float mup, float mum) {
  const float asym = fabsf(mup - mum);
  const float x = fmaxf(xmax * (1.f / kFarX), asym * xmax * (1.f / kFarAsym));
  return (vmax <= kFarV && asym * vmax <= kFarAsym && x < 1e30f) ? x : __int_as_float(0x7f800000);
}

__device__ __forceinline__ float rsqrt_fast(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_fast(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// floor by rounding down onto the integers (|x| < 2^22): the integer in the low mantissa bits
constexpr float kFloorMagic = 12582912.f;  // 1.5 * 2^23
constexpr int kFloorBits = 0x4B400000;
__device__ __forceinline__ V2 floor_bits2(V2 x) { return V2(__fadd2_rd(x.v, make_float2(kFloorMagic, kFloorMagic))); }

}  // namespace pc
