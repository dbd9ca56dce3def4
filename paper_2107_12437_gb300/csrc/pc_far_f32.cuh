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

namespace pc {

// ------------------------------------------------------------------------------------------------
// The terms that the first-order form drops, for a float64 evaluation split in two: the linear part in
// float64, the rest, smaller by (X/R)^2 and V^2, in float32.
//
// Expansion of one charge's field coefficients in its offset eps X along the axis (eps = mu+ or -mu-),
// lengths in units of R, on the history segment of the centre's retarded time (X, V, A linear there with
// slopes X', V', A'), through third order: the charge's distance 1 + d follows from
//   (1 + d)^2 = 1 - 2 mu y + y^2,  y = eps (X - d X'),  mu = rho.p / R,
// its velocity and acceleration are w = eps (V - d V'), g = eps (A - d A') (times R, R^2), and with
// h = mu - y, R_u = 1 + d - w h, G = 1 - w^2 + g h the coefficients of E = C_a rho + D p and B = C_b (rho x p),
// phi and A are those of dipole_pair.  For equal masses the even terms cancel between the charges and the
// third-order one counts 1 - 3 mu+ mu- = 1/4.
// Checked in extended precision against both charges (all directions and phases, 200 THz): with the cubic
// terms the field is within 5e-12 (X/R = 2e-3), 6e-13 (1e-3), 9e-14 (5e-4), 1.5e-14 (2e-4) of the sum of
// the terms' magnitudes, fifth-order truncation included, where the first-order form has (X/R)^2.  The sum
// of the two charges' fields in float64 rounds at 1e-16 R/X of it.
// ------------------------------------------------------------------------------------------------
struct Cubic {
  float Ca, D, Cb, phi, A;
};
// mu = cos(rho, p); x = X/R, v = V, al = A R and the slopes per sample dX, dV R, dA R^2
__device__ __forceinline__ Cubic cubic_terms(float mu, float x, float v, float al, float dX, float dV, float dA) {
  const float d1 = -mu * x;
  const float xx = x * x, xp = x * dX, mm = mu * mu;
  const float d2 = 0.5f * xx * (1.f - mm) - mm * xp;
  const float d3 = mu * (dX * d2 + x * (xp + d2));
  const float y2 = -d1 * dX, y3 = -d2 * dX;
  const float w2 = -d1 * dV, w3 = -d2 * dV;
  const float g2 = -d1 * dA, g3 = -d2 * dA;
  const float u1 = fmaf(-v, mu, d1), u2 = d2 - fmaf(w2, mu, -v * x), u3 = d3 - fmaf(w3, mu, -fmaf(v, y2, w2 * x));
  const float i1 = -u1, i2 = fmaf(u1, u1, -u2), i3 = fmaf(u1, fmaf(2.f, u2, -u1 * u1), -u3);
  const float J1 = 2.f * i1, J2 = fmaf(i1, i1, 2.f * i2);
  const float K1 = 3.f * i1, K2 = 3.f * fmaf(i1, i1, i2), K3 = fmaf(3.f, i3, i1 * fmaf(6.f, i2, i1 * i1));
  const float G1 = al * mu, G2 = fmaf(g2, mu, -fmaf(al, x, v * v)),
              G3 = fmaf(g3, mu, -fmaf(2.f * v, w2, fmaf(al, y2, g2 * x)));
  const float GK1 = G1 + K1, GK2 = fmaf(G1, K1, G2 + K2), GK3 = fmaf(G2, K1, fmaf(G1, K2, G3 + K3));
  const float Cb1 = -(v + al), Cb2 = -fmaf(v, GK1, fmaf(al, J1, w2 + g2)),
              Cb3 = -fmaf(v, GK2, fmaf(w2, GK1, fmaf(al, J2, fmaf(g2, J1, w3 + g3))));
  Cubic o;
  o.Ca = GK3;
  o.D = fmaf(d1, Cb2, fmaf(d2, Cb1, Cb3)) - fmaf(x, GK2, fmaf(y2, GK1, y3));
  o.Cb = Cb3;
  o.phi = i3;
  o.A = fmaf(v, i2, fmaf(w2, i1, w3));
  return o;
}

// The distance from which the split form serves a float64 driving field.  With X/R <= kSplitX the cubic
// terms' float32 rounding is 1e-14 of the pair's field, against the 1e-16 R/X (3e-13) at which the sum of
// the two charges rounds there (less only where they do not cancel: on a ring of 256 with moments along its
// axis E_d was within 2.5e-16 of binary128; 6.5e-4 here made that 8e-16).  V <= kSplitV keeps the fifth order
// in V below 1e-14.  Equal masses only: the second order of unequal ones, in float32, would be 1e-11.
constexpr double kSplitX = 4e-4, kSplitV = 2e-4;

}  // namespace pc
