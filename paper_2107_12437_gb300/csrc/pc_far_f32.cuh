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

// Reverse of cubic_terms for a loss that depends on Ca and D (the driving field): their adjoints in, those of
// mu, x, v, al and of the three slopes out.  Checked against central differences of cubic_terms.
struct CubicIn {
  float mu, x, v, al, dX, dV, dA;
};
__device__ __forceinline__ CubicIn cubic_terms_rev(float mu, float x, float v, float al, float p, float q, float r, float Cab,
                                                   float Db, Cubic &val) {
  const float d1 = -mu * x, xx = x * x, xp = x * p, mm = mu * mu;
  const float d2 = 0.5f * xx * (1.f - mm) - mm * xp, e3 = p * d2 + x * (xp + d2), d3 = mu * e3;
  const float y2 = -d1 * p, y3 = -d2 * p, w2 = -d1 * q, w3 = -d2 * q, g2 = -d1 * r, g3 = -d2 * r;
  const float u1 = d1 - v * mu, u2 = d2 - w2 * mu + v * x, u3 = d3 - w3 * mu + v * y2 + w2 * x;
  const float i1 = -u1, i2 = u1 * u1 - u2, i3 = u1 * (2.f * u2 - u1 * u1) - u3;
  const float J1 = 2.f * i1, J2 = i1 * i1 + 2.f * i2;
  const float K1 = 3.f * i1, K2 = 3.f * (i1 * i1 + i2), K3 = 3.f * i3 + i1 * (6.f * i2 + i1 * i1);
  const float G1 = al * mu, G2 = g2 * mu - al * x - v * v, G3 = g3 * mu - 2.f * v * w2 - al * y2 - g2 * x;
  const float GK1 = G1 + K1, GK2 = G1 * K1 + G2 + K2;
  const float Cb1 = -(v + al), Cb2 = -(v * GK1 + al * J1 + w2 + g2),
              Cb3 = -(v * GK2 + w2 * GK1 + al * J2 + g2 * J1 + w3 + g3);
  val.Ca = G2 * K1 + G1 * K2 + G3 + K3;
  val.D = d1 * Cb2 + d2 * Cb1 + Cb3 - x * GK2 - y2 * GK1 - y3;
  float d1b = Db * Cb2, d2b = Db * Cb1;
  const float m = -Db * d1, Cb1b = Db * d2, n = -Db;
  float xb = -Db * GK2, y2b = -Db * GK1;
  const float y3b = -Db;
  float GK2b = -Db * x + n * v, GK1b = -Db * y2 + n * w2 + m * v;
  float vb = n * GK2 + m * GK1 - Cb1b, alb = n * J2 + m * J1 - Cb1b;
  float w2b = n * GK1 + m, g2b = n * J1 + m, w3b = n, g3b = n;
  const float J2b = n * al, J1b = n * g2 + m * al;
  const float G2b = Cab * K1 + GK2b, K1b = Cab * G2 + GK2b * G1 + GK1b, G1b = Cab * K2 + GK2b * K1 + GK1b;
  const float K2b = Cab * G1 + GK2b, G3b = Cab, K3b = Cab;
  g3b += G3b * mu;
  float mub = G3b * g3 + G2b * g2 + G1b * al;
  vb -= 2.f * (G3b * w2 + G2b * v);
  w2b -= 2.f * G3b * v;
  alb += G1b * mu - G3b * y2 - G2b * x;
  y2b -= G3b * al;
  g2b += G2b * mu - G3b * x;
  xb -= G3b * g2 + G2b * al;
  const float i3b = 3.f * K3b;
  const float i1b = K3b * (6.f * i2 + 3.f * i1 * i1) + 6.f * K2b * i1 + 3.f * K1b + 2.f * (J2b * i1 + J1b);
  const float i2b = 6.f * K3b * i1 + 3.f * K2b + 2.f * J2b;
  const float u3b = -i3b, u1b = i3b * (2.f * u2 - 3.f * u1 * u1) + 2.f * i2b * u1 - i1b, u2b = 2.f * i3b * u1 - i2b;
  w3b -= u3b * mu;
  mub -= u3b * w3 + u2b * w2 + u1b * v;
  vb += u3b * y2 + u2b * x - u1b * mu;
  y2b += u3b * v;
  w2b += u3b * x - u2b * mu;
  xb += u3b * w2 + u2b * v;
  d2b += u2b - (g3b * r + w3b * q + y3b * p);
  d1b += u1b - (g2b * r + w2b * q + y2b * p);
  CubicIn o;
  o.dA = -(g3b * d2 + g2b * d1);
  o.dV = -(w3b * d2 + w2b * d1);
  float pb = -(y3b * d2 + y2b * d1);
  mub += u3b * e3;
  const float t = u3b * mu;
  pb += t * d2;
  d2b += t * (p + x);
  xb += t * (xp + d2);
  const float xpb = t * x - d2b * mm, xxb = 0.5f * d2b * (1.f - mm), mmb = -d2b * (0.5f * xx + xp);
  o.dX = pb + xpb * x;
  o.x = xb + xpb * p + 2.f * x * xxb - d1b * mu;
  o.mu = mub + 2.f * mu * mmb - d1b * x;
  o.v = vb;
  o.al = alb;
  return o;
}

// The second-order terms, which the two charges of equal masses share: their derivative along a change of
// (x, v, al) at fixed slopes enters where only one of the charges sees that change.
__device__ __forceinline__ Cubic quad_terms(float mu, float x, float v, float al, float dX, float dV, float dA) {
  const float d1 = -mu * x;
  const float d2 = 0.5f * x * x * (1.f - mu * mu) - mu * mu * x * dX;
  const float y2 = -d1 * dX, w2 = -d1 * dV, g2 = -d1 * dA;
  const float u1 = fmaf(-v, mu, d1), u2 = d2 - fmaf(w2, mu, -v * x);
  const float i1 = -u1, i2 = fmaf(u1, u1, -u2);
  const float J1 = 2.f * i1, K1 = 3.f * i1, K2 = 3.f * fmaf(i1, i1, i2);
  const float G1 = al * mu, G2 = fmaf(g2, mu, -fmaf(al, x, v * v));
  const float GK1 = G1 + K1;
  Cubic o;
  o.Ca = fmaf(G1, K1, G2 + K2);
  o.Cb = -fmaf(v, GK1, fmaf(al, J1, w2 + g2));
  o.D = fmaf(d1, -(v + al), o.Cb) - fmaf(x, GK1, y2);
  o.phi = i2;
  o.A = fmaf(v, i1, w2);
  return o;
}
// that derivative along (ex, ev, ea), exact for a quadratic form: half the difference at +-t times it, t
// making the step as large as the point
__device__ __forceinline__ void add_quad_slope(Cubic &c, float sign, float mu, float x, float v, float al, float dX, float dV,
                                               float dA, float ex, float ev, float ea) {
  const float t = __fdividef(fabsf(x) + fabsf(v) + fabsf(al), fabsf(ex) + fabsf(ev) + fabsf(ea) + 1e-30f);
  const Cubic a = quad_terms(mu, fmaf(t, ex, x), fmaf(t, ev, v), fmaf(t, ea, al), dX, dV, dA);
  const Cubic b = quad_terms(mu, fmaf(-t, ex, x), fmaf(-t, ev, v), fmaf(-t, ea, al), dX, dV, dA);
  const float w = t > 0.f ? __fdividef(0.5f * sign, t) : 0.f;
  c.Ca = fmaf(w, a.Ca - b.Ca, c.Ca);
  c.D = fmaf(w, a.D - b.D, c.D);
  c.Cb = fmaf(w, a.Cb - b.Cb, c.Cb);
  c.phi = fmaf(w, a.phi - b.phi, c.phi);
  c.A = fmaf(w, a.A - b.A, c.A);
}

// The distance from which the split form serves a float64 driving field.  With X/R <= kSplitX the cubic
// terms' float32 rounding is 1e-14 of the pair's field, against the 1e-16 R/X (3e-13) at which the sum of
// the two charges rounds there (less only where they do not cancel: on a ring of 256 with moments along its
// axis E_d was within 2.5e-16 of binary128; 6.5e-4 here made that 8e-16).  V <= kSplitV keeps the fifth order
// in V below 1e-14.  Equal masses only: the second order of unequal ones, in float32, would be 1e-11.
constexpr double kSplitX = 4e-4, kSplitV = 2e-4;


// The split form continues the centre's history segment to both charges and adds, for one that has left it,
// its overshoot times the second difference of the samples at that end: exact on piecewise linear histories
// only while at most one charge is off the segment, and less than a segment off it.  Seen from any point the
// charges' retarded samples lie up to |X| (1 + kSplitV) apart, so |X| has to stay below one sample.  (With 2
// samples the field was 5e-9 off, with 6.7 1e-8; and a charge that far from its centre can be past the end of
// the history or within an exclusion radius where the centre is not.)
constexpr float kSplitSamples = 0.95f;

// One dipole's field at a point in the split form, for the float64 field sum and for near fields that
// cancel in float32: r the separation from its centre (c dt), p its axis, qs = q / e, u the time in samples,
// d / dd / ddd its float64 history with the scales (1/(qL), 1/(qc), dt/(qc)) and H the float32 mirror.
// Adds the linear part to lin[10] (float64) and the cubic terms to cub[10] (float32), both as (E, B, phi, A)
// in the units of dipole_pair.  False, adding nothing, where the two-charge form has to decide: off the
// interior of the history, within rmin of the centre, X, X/R or V beyond the limits at the samples, or
// samples that are not those of a smooth motion.  Equal masses only (the caller's condition).
// 1/R comes from float32's by one third-order step y (1 + e/2 + 3 e^2/8), e = 1 - R^2 y^2 (its error 5 e^3/16
// is below 1e-19), the sample index by adding 1.5 * 2^52 with rounding down: about 66 instructions on the
// float64 unit a pair, where the two charges' roots and difference form take 280.
struct SplitLimits {
  float x, v, rmin;
};
template <int KIND>
__device__ __forceinline__ bool split_dipole(double rx, double ry, double rz, double px, double py, double pz, double qs,
                                             double u, const double *d, const double *dd, const double *ddd, double sx,
                                             double sv, double sa, const float4 *H, int S, const SplitLimits lim,
                                             double (&lin)[10], float (&cub)[10]) {
  const double R2 = fma(rz, rz, fma(ry, ry, rx * rx));
  const float fx = (float)rx, fy = (float)ry, fz = (float)rz;
  const float R2f = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
  const float iRf = rsqrt_fast(R2f), Rf = R2f * iRf;
  // (the radiation field's cubic terms are a difference from the Coulomb field's, which outweighs it close by)
  if (!(Rf > (KIND == PC_RADIATION ? fmaxf(lim.rmin, 300.f) : lim.rmin) && Rf < 1e9f)) return false;
  const double y = (double)iRf;
  const double e = fma(-(R2 * y), y, 1.0);
  const double i = fma(y * e, fma(e, 0.375, 0.5), y);
  const double R = R2 * i;
  const double x = u - R;
  if (!(x > 2.0 && x < (double)(S - 3))) return false;
  const double magic = 6755399441055744.0;  // 1.5 * 2^52
  const double m = __dadd_rd(x, magic);
  const int k = __double2loint(m);
  const double th = (u - (m - magic)) - R;  // (u less a whole number of samples is exact)
  const float4 h0 = __ldg(H + k), h1 = __ldg(H + k + 1);
  // (the slope of X enters as a speed does; samples of d need not follow those of d')
  // (each by itself: a maximum would pass over a NaN, which the two-charge form refuses in d)
  const float xl = fminf(lim.x * Rf, kSplitSamples);
  if (!(fabsf(h0.x) <= xl && fabsf(h1.x) <= xl && fabsf(h0.y) <= lim.v && fabsf(h1.y) <= lim.v &&
        fabsf(h1.x - h0.x) <= lim.v))
    return false;
  const double d0 = d[k], v0 = dd[k], a0 = ddd[k];
  const double Dd = d[k + 1] - d0, Dv = dd[k + 1] - v0, Da = ddd[k + 1] - a0;
  double X = fma(th, Dd, d0), V = fma(th, Dv, v0), A = fma(th, Da, a0);
  const float qf = (float)qs, pxf = (float)px, pyf = (float)py, pzf = (float)pz, thf = (float)th;
  const float mu = fmaf(fz, pzf, fmaf(fy, pyf, fx * pxf)) * iRf;
  // (the slopes from the float64 samples: a difference of float32 ones is good to 5e-5 only, which put
  // 1e-14 instead of 1e-15 into the fields of 10 pm dipoles)
  const float dX = (float)(Dd * sx), dV = (float)(Dv * sv), dA = (float)(Da * sa);
  const float Xf = fmaf(thf, dX, h0.x);
  if (KIND == PC_RADIATION) {
    // the radiation field's cubic terms are a difference from the Coulomb field's, in float32: where the slow motion
    // of a charge or a zero of A leaves little of the former, that rounding (1e-7 of (X/R + V)^3) is all of it
    const float c = fabsf(Xf) * iRf + fmaxf(fabsf(h0.y), fabsf(h1.y));
    if (!(c * c * c <= 1e-5f * fabsf(fmaf(thf, dA, h0.z)) * Rf)) return false;
  }
  // a charge whose own retarded time lies off the centre's segment: its state differs from the segment's
  // extension by the overshoot times the second difference of the samples.  The charges' delays are off the
  // centre's by -+ X mu / 2 + (X^2 (1 - mu^2) / 2 - mu^2 X X') / 4 R: the overshoots from those in float64
  // (float32 ones, good to 1e-7 of a sample, put 1e-13 into the potentials at such points)
  const float s1 = 0.5f * Xf * mu, s2 = 0.25f * Xf * iRf * fmaf(0.5f * Xf, fmaf(-mu, mu, 1.f), -mu * mu * Rf * dX);
  float ex = 0.f, ev = 0.f, ea = 0.f, sign = 0.f;
  if (fabsf(thf - 0.5f) + fabsf(s1) + fabsf(s2) > 0.499999f) {
    const double tp = th + (double)(s1 - s2), tm = th - (double)(s1 + s2);  // the charges' fractions
    const double lp = fmax(-tp, 0.0), lm = fmax(-tm, 0.0), hp = fmax(tp - 1.0, 0.0), hm = fmax(tm - 1.0, 0.0);
    const double lo = lp + lm, hi = hp + hm;
    if (lo > 0.0 || hi > 0.0) {
      const int n = lo > 0.0 ? k : k + 1;
      const double o = lo > 0.0 ? lo : hi;
      const double eX = o * ((d[n + 1] - d[n]) - (d[n] - d[n - 1])), eV = o * ((dd[n + 1] - dd[n]) - (dd[n] - dd[n - 1])),
                   eA = o * ((ddd[n + 1] - ddd[n]) - (ddd[n] - ddd[n - 1]));
      X = fma(0.5, eX, X);
      V = fma(0.5, eV, V);
      A = fma(0.5, eA, A);
      // the next order, of opposite sign for the two charges
      sign = (lo > 0.0 ? lp > lm : hp > hm) ? 1.f : -1.f;
      ex = (float)(eX * sx) * iRf;
      ev = (float)(eV * sv);
      ea = (float)(eA * sa) * Rf;
      // what is left out, of the order of the change e times the change of X's slope there or the square of
      // (X/R, V), stays below 1e-11 of the pair's field for every history that its samples resolve (140 a
      // period); others (noise, jumps) take the two charges here
      const float of = (float)o;
      if (!(fmaf(fabsf(ex), Rf, 3e-8f * of) * (fabsf(ex) + fabsf(ev) + fabsf(ea)) <=
            1e-11f * of * (fabsf(Xf) * iRf + fabsf(h0.y) + fabsf(h0.z) * Rf)))
        return false;
    }
  }
  X *= sx;
  V *= sv;
  A *= sa;
  const double qx = qs * px, qy = qs * py, qz = qs * pz;
  const double i2 = i * i, rpi2 = fma(rz, qz, fma(ry, qy, rx * qx)) * i2;
  const double t1 = fma(i, X, V);
  double cE, cP, cB;
  if (KIND == PC_COULOMB) {
    cE = rpi2 * i2 * (3.0 * t1);
    cP = i2 * t1;
    cB = i2 * i * V;
  } else if (KIND == PC_RADIATION) {
    cE = rpi2 * i * A;
    cP = i * A;
    cB = i2 * A;
  } else {
    cE = rpi2 * i * fma(3.0 * i, t1, A);
    cP = i * fma(i, t1, A);
    cB = i2 * fma(i, V, A);
  }
  lin[0] = fma(-cP, qx, fma(cE, rx, lin[0]));
  lin[1] = fma(-cP, qy, fma(cE, ry, lin[1]));
  lin[2] = fma(-cP, qz, fma(cE, rz, lin[2]));
  lin[3] = fma(cB, fma(qy, rz, -(qz * ry)), lin[3]);
  lin[4] = fma(cB, fma(qz, rx, -(qx * rz)), lin[4]);
  lin[5] = fma(cB, fma(qx, ry, -(qy * rx)), lin[5]);
  lin[6] = fma(rpi2, t1, lin[6]);
  const double vi = V * i;
  lin[7] = fma(vi, qx, lin[7]);
  lin[8] = fma(vi, qy, lin[8]);
  lin[9] = fma(vi, qz, lin[9]);
  // the cubic terms (1 - 3 mu+ mu- = 1/4 for equal masses)
  const float xn = Xf * iRf, vf = fmaf(thf, dV, h0.y), al = fmaf(thf, dA, h0.z) * Rf;
  const float dVn = dV * Rf, dAn = dA * Rf * Rf;
  Cubic c = cubic_terms(mu, xn, vf, KIND == PC_COULOMB ? 0.f : al, dX, dVn, KIND == PC_COULOMB ? 0.f : dAn);
  if (sign != 0.f)
    add_quad_slope(c, sign, mu, xn, vf, KIND == PC_COULOMB ? 0.f : al, dX, dVn, KIND == PC_COULOMB ? 0.f : dAn, ex, ev,
                   KIND == PC_COULOMB ? 0.f : ea);
  float Ca = c.Ca, D = c.D, Cb = c.Cb;
  if (KIND == PC_RADIATION) {
    Cubic v = cubic_terms(mu, xn, vf, 0.f, dX, dVn, 0.f);
    if (sign != 0.f) add_quad_slope(v, sign, mu, xn, vf, 0.f, dX, dVn, 0.f, ex, ev, 0.f);
    Ca -= v.Ca;
    D -= v.D;
    Cb -= v.Cb;
  }
  const float q1 = 0.25f * qf * iRf, q2 = q1 * iRf;
  const float ca = q2 * Ca * iRf, cd = q2 * D, cb = q2 * Cb * iRf, cv = q1 * c.A;
  cub[0] += fmaf(ca, fx, cd * pxf);
  cub[1] += fmaf(ca, fy, cd * pyf);
  cub[2] += fmaf(ca, fz, cd * pzf);
  cub[3] = fmaf(cb, fy * pzf - fz * pyf, cub[3]);
  cub[4] = fmaf(cb, fz * pxf - fx * pzf, cub[4]);
  cub[5] = fmaf(cb, fx * pyf - fy * pxf, cub[5]);
  cub[6] = fmaf(q1, c.phi, cub[6]);
  cub[7] = fmaf(cv, pxf, cub[7]);
  cub[8] = fmaf(cv, pyf, cub[8]);
  cub[9] = fmaf(cv, pzf, cub[9]);
  return true;
}

// float64 field sum: errors against binary128 as the two-charge form's (300 points of the grid of 64 dipoles
// of 1, 10 and 20 pm: E rms 1.2-1.6e-12, B 4e-15, phi 2e-13, A 1.8e-15 in both; medians 1.2e-15)
constexpr float kSplitFieldX = 6e-5f, kSplitFieldV = 1e-4f;
// near fields of the mixed sum, kept to 1e-10 of the terms' magnitudes
constexpr float kSplitNearX = 1e-3f, kSplitNearV = 1e-3f;

}  // namespace pc
