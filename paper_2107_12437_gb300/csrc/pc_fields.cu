// Retarded Lienard-Wiechert field sum (arXiv 2107.12437, Sec. 2.1-2.2) on sm_103a.
//
// Two paths:
//   PC_F64   one thread per (point, time); every charge's retarded time is found by solving, on one
//            segment of its piecewise-linear history, the quadratic c^2 (t - t')^2 = |r - r_s(t')|^2
//            (Eq. ret_t with linear interpolation, Sec. 3.1), moving to the segment the root points
//            to until it lies inside; fields from Griffiths' form of Eqs. E, B, V, A in float64, a
//            dipole's two charges together in the difference form of the mixed path (below).
//   PC_MIXED a CTA owns a tile of points.  Per (tile, source) the float64 distance from the tile's
//            anchor point to the source reference gives the integer part of the retarded sample
//            index; per (point, source) everything else runs in float32 on offsets (lengths in
//            units of c*dt, so a delay in samples equals a distance).  The two charges of a dipole
//            are evaluated together in difference form: the net field q[E(x+) - E(x-)] is built
//            from differences of the scalar coefficients of the Lienard-Wiechert field that carry
//            no cancellation, so the s/R loss of the +-q pair (s = charge separation) does not
//            appear.  Contributions are summed in groups of 32 (the two-point kernel: 16) and the
//            group sums are added with Kahan compensation.
#include <stdio.h>

#include <algorithm>
#include <type_traits>

#include "pc_internal.cuh"
#include "pc_lw_f32.cuh"
#include "pc_lw_f32x2.cuh"
#include "pc_far_f32.cuh"
#include "pc_lw_f64.cuh"

namespace pc {

constexpr int kMaxT = 32;        // times per launch (the host splits longer lists)
constexpr int kMixThreads = 256; // points per CTA in the mixed path
constexpr int kChunk = 64;       // sources staged in shared memory at a time (the largest stage)
// per-chunk bit mask of the pairs that left the fast path: 32 or 64 sources per stage
template <int CH>
struct SlowMask {
  using T = typename std::conditional<(CH <= 32), unsigned, unsigned long long>::type;
  static __device__ __forceinline__ T bit(int j) { return (T)1 << j; }
  static __device__ __forceinline__ int first(T m) {
    if constexpr (CH <= 32) return __ffs((int)m) - 1;
    else return __ffsll((long long)m) - 1;
  }
};
// a dipole closer than kNearL c*dt to a point whose near field there cancels by more than kCancel
// (dipole_cancellation) is summed in float64 instead
constexpr float kNearL = 400.f;
constexpr float kCancel = 6.f;

struct Points {
  const double *list;  // [P][3] or null for a plane
  double o[3], eu[3], ev[3];
  int64_t nu, nv;
  int64_t P;
};

__device__ __forceinline__ void point_at(const Points &pd, int64_t p, double r[3]) {
  if (pd.list) {
    r[0] = pd.list[3 * p];
    r[1] = pd.list[3 * p + 1];
    r[2] = pd.list[3 * p + 2];
  } else {
    double iu = (double)(p / pd.nv), iv = (double)(p % pd.nv);
    r[0] = pd.o[0] + iu * pd.eu[0] + iv * pd.ev[0];
    r[1] = pd.o[1] + iu * pd.eu[1] + iv * pd.ev[1];
    r[2] = pd.o[2] + iu * pd.eu[2] + iv * pd.ev[2];
  }
}

struct Sources {
  // point charges
  int32_t M;
  int64_t S;
  double t0, dt;
  const double *q, *pos, *vel, *acc;
  int32_t static_before;
  // dipoles
  int32_t N;
  int64_t Sd;
  double t0d, dtd;
  const double *origin, *axis, *qd, *m1, *m2, *d, *dd, *ddd;
};

struct Outs {
  void *E, *B, *phi, *A;
  uint8_t *mask;
};

struct Launch {
  Points pts;
  Sources src;
  Outs out;
  int32_t T;            // times in this launch
  int64_t frame0;       // output frame of times[0]
  double times[kMaxT];
  double r_excl;
  int *status;
  // mixed path: float32 mirrors and per-charge references
  const float4 *Hd;     // [N][Sd] (d/(qL), d'/(qc), d'' dt/(qc), 0)
  const float4 *Hc;     // [M][S][3]: offset/L, v/c, a dt/c
  const double *cref;   // [M][3] reference position (sample 0)
  int32_t tile_shift;   // plane tiles of (256 >> tile_shift) rows x (1 << tile_shift) columns
  // mixed path, set on the host: each frame's time in dipole samples, 1/(c dt) of the dipole
  // history, and per dipole two float4 records (axis x, y, z, q/e), (m2/(m1+m2), m1/(m1+m2), 0, 0)
  double uf[kMaxT];
  float uf_hi[kMaxT], uf_lo[kMaxT];  // the same as float-float
  double iLd;
  float eu_L[3], ev_L[3];            // plane steps in units of c dt (dipole history)
  const float4 *srcf;
  float unit[4];                     // SI units of the float32 sums of E, B, phi, A
  // loop constants of the dipole sum, read from the parameter bank rather than held in registers:
  // r_excl in units of c dt, that plus 1.5 (the fast path's distance bound), and the number of
  // interior segments S - 3 (fast segments 1 <= j <= S - 3)
  float rex, rex_fast;
  unsigned jlim;
  // point charges: each frame's time in their samples, 1/(c dt) of their history, and the scales
  // of their float32 terms to the output unit (E, phi)
  double ufc[kMaxT];
  double iLc;
  float sE, sP;
  // the far form (pc_far_f32.cuh): per dipole the distance from which it applies, and the spread of a
  // tile's points about its anchor, both in c dt
  const float *rfar;
  float tile_r;
  // float64 sums of dipoles alone: of the kSplitAsk sampled pairs that split_count_kernel counts in status[1], the
  // number of near ones from which fields_f64_kernel runs and fields_split64_kernel does not (0: not asked)
  int near_min;
};

// the float32 outputs' units: E in k_e e / L^2, B in k_e e / (L^2 c), phi in k_e e / L,
// A in k_e e / (L c), L = c dt of the dipoles (of the point charges when there are no dipoles)
__host__ inline void set_units(Launch &L) {
  const double Lref = (L.src.N > 0) ? kC * L.src.dtd : kC * L.src.dt;
  if (L.src.N > 0) {
    L.rex = (float)(L.r_excl * L.iLd);
    L.rex_fast = L.rex + 1.5f;
    L.jlim = L.src.Sd > 3 ? (unsigned)(L.src.Sd - 3) : 0u;
  }
  const double kE2 = kKe * kE / (Lref * Lref), kP = kKe * kE / Lref;
  L.unit[0] = (float)kE2;
  L.unit[1] = (float)(kE2 / kC);
  L.unit[2] = (float)kP;
  L.unit[3] = (float)(kP / kC);
  if (L.src.M > 0) {
    const double Lch = kC * L.src.dt;
    L.iLc = 1.0 / Lch;
    L.sE = (float)((Lref / Lch) * (Lref / Lch));
    L.sP = (float)(Lref / Lch);
  }
}

// the frames of one launch: their times and, for the dipoles, the times in samples
__host__ inline void set_frames(Launch &L, const double *times, int32_t f0, int32_t n) {
  L.T = n;
  L.frame0 = f0;
  for (int i = 0; i < n; ++i) {
    L.times[i] = times[f0 + i];
    L.uf[i] = L.src.N > 0 ? (times[f0 + i] - L.src.t0d) / L.src.dtd : 0.0;
    L.ufc[i] = L.src.M > 0 ? (times[f0 + i] - L.src.t0) / L.src.dt : 0.0;
    L.uf_hi[i] = (float)L.uf[i];
    L.uf_lo[i] = (float)(L.uf[i] - (double)L.uf_hi[i]);
  }
}

// ================================================================================================
// float64 path
// ================================================================================================

// One dipole's two charges in float64 added to acc (units of dipole_pair): each charge's retarded time the
// exact root on its own history segment, the net field from differences of the coefficients.
template <int KIND>
__device__ __forceinline__ int dipole_f64(const Launch &L, int j, const double r[3], double u, double (&acc)[10],
                                          uint8_t &mask) {
  const Sources &s = L.src;
  const double iLd = L.iLd;
  const double q = s.qd[j], m1 = s.m1[j], m2 = s.m2[j];
  const double rx = (r[0] - s.origin[3 * j]) * iLd, ry = (r[1] - s.origin[3 * j + 1]) * iLd,
               rz = (r[2] - s.origin[3 * j + 2]) * iLd;
  const double rn = sqrt(rx * rx + ry * ry + rz * rz);
  const double px = s.axis[3 * j], py = s.axis[3 * j + 1], pz = s.axis[3 * j + 2];
  const double rp = rx * px + ry * py + rz * pz;
  const double x = u - rn;
  const double fl = floor(x);
  HistF64 H;
  H.d = s.d + (size_t)j * s.Sd;
  H.dd = s.dd + (size_t)j * s.Sd;
  H.ddd = s.ddd + (size_t)j * s.Sd;
  const double iq = 1.0 / q, imm = 1.0 / (m1 + m2);
  H.sx = iq * iLd;
  H.sv = iq * (1.0 / kC);
  H.sa = iq * (s.dtd / kC);
  double Xp, Vp, Ap, dp, Xm, Vm, Am, dm;
  const double mup = m2 * imm, mum = m1 * imm;
  const int err = dip_pair_exact<double, HistF64>(H, (int)s.Sd, (int)fl, x - fl, rn, rp, mup, mum, Xp, Vp, Ap, dp, Xm,
                                                  Vm, Am, dm, 1e-9);
  if (err) return err;
  dipole_pair<KIND, double>(rx, ry, rz, rn, px, py, pz, rp, mup, mum, q * (1.0 / kE), Xp, Vp, Ap, dp, Xm, Vm, Am, dm,
                            L.r_excl * iLd, acc, mask);
  return 0;
}
template <int KIND>
__device__ __noinline__ int dipole_f64_call(const Launch &L, int j, const double r[3], double u, double *acc, uint8_t *mask) {
  double a[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  const int e = dipole_f64<KIND>(L, j, r, u, a, *mask);
#pragma unroll
  for (int i = 0; i < 10; ++i) acc[i] = a[i];
  return e;
}
__device__ __forceinline__ void store_f64(const Launch &L, int f, int64_t p, const double E[3], const double B[3], double phi,
                                          const double A[3], uint8_t mask) {
  const int64_t o = (L.frame0 + f) * L.pts.P + p;
  if (L.out.E) {
    double *e = (double *)L.out.E + 3 * o;
    e[0] = E[0];
    e[1] = E[1];
    e[2] = E[2];
  }
  if (L.out.B) {
    double *b = (double *)L.out.B + 3 * o;
    b[0] = B[0];
    b[1] = B[1];
    b[2] = B[2];
  }
  if (L.out.phi) ((double *)L.out.phi)[o] = phi;
  if (L.out.A) {
    double *a = (double *)L.out.A + 3 * o;
    a[0] = A[0];
    a[1] = A[1];
    a[2] = A[2];
  }
  if (L.out.mask) L.out.mask[o] = mask;
}
// the sums in the units of the difference form to SI: E in k_e e / L^2, B in k_e e / (L^2 c), phi in
// k_e e / L, A in k_e e / (L c), L = c dt of the dipole history
__device__ __forceinline__ void scale_f64(double iLd, const double (&acc)[10], double E[3], double B[3], double &phi,
                                          double A[3]) {
  const double uP = kKe * kE * iLd, uE = uP * iLd;
  for (int i = 0; i < 3; ++i) {
    E[i] += uE * acc[i];
    B[i] += uE * (1.0 / kC) * acc[3 + i];
    A[i] += uP * (1.0 / kC) * acc[7 + i];
  }
  phi += uP * acc[6];
}

template <int KIND>
__global__ void __launch_bounds__(128) fields_f64_kernel(const Launch L) {
  if (L.status[1] < L.near_min) return;
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int f = blockIdx.y;
  if (p >= L.pts.P || f >= L.T) return;
  double r[3];
  point_at(L.pts, p, r);
  const double t = L.times[f];
  double E[3] = {0, 0, 0}, B[3] = {0, 0, 0}, A[3] = {0, 0, 0}, phi = 0.0;
  uint8_t mask = 0;
  int err = 0;
  const Sources &s = L.src;
  // ---- point charges ----
  if (s.M > 0) {
    const double u = (t - s.t0) / s.dt, cdt = kC * s.dt;
    for (int c = 0; c < s.M && !err; ++c) {
      TrajF64 tr;
      tr.dipole = false;
      tr.pos = s.pos + (size_t)c * s.S * 3;
      tr.vel = s.vel + (size_t)c * s.S * 3;
      tr.acc = s.acc + (size_t)c * s.S * 3;
      int64_t kr = (int64_t)floor(u);
      kr = kr < 0 ? 0 : (kr > s.S - 1 ? s.S - 1 : kr);
      double pr[3];
      tr.p(kr, pr);
      double dv[3] = {r[0] - pr[0], r[1] - pr[1], r[2] - pr[2]};
      double tau0 = sqrt(dot3(dv, dv)) * L.iLc;
      int64_t k;
      double th;
      err = solve_f64(tr, s.S, s.static_before, r, u, cdt, (int64_t)floor(u - tau0), &k, &th);
      if (err) break;
      double p0[3], v[3], a[3];
      if (k < 0) {
        tr.p(0, p0);
        v[0] = v[1] = v[2] = 0.0;
        a[0] = a[1] = a[2] = 0.0;
      } else {
        double p1[3], v1[3], a1[3];
        tr.p(k, p0);
        tr.p(k + 1, p1);
        tr.va(k, v, a);
        tr.va(k + 1, v1, a1);
        for (int i = 0; i < 3; ++i) {
          p0[i] += th * (p1[i] - p0[i]);
          v[i] += th * (v1[i] - v[i]);
          a[i] += th * (a1[i] - a[i]);
        }
      }
      double av[3] = {r[0] - p0[0], r[1] - p0[1], r[2] - p0[2]};
      lw_add_f64<KIND>(s.q[c], av, v, a, L.r_excl, E, B, &phi, A, &mask);
    }
  }
  // ---- dipoles: the two charges of each (Eqs. r_1, r_2) in difference form ----
  // Each charge's retarded time is the exact root on its own history segment (offsets from the
  // dipole centre in units of c dt, times in samples); the net field q [F(x+) - F(x-)] is formed
  // from differences of the Lienard-Wiechert coefficients (pc_lw_f32.cuh, dipole_pair), so the
  // R/s cancellation of the +-q pair costs no digits.
  if (s.N > 0 && !err) {
    const double u = (t - s.t0d) / s.dtd;
    double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int j = 0; j < s.N && !err; ++j) err = dipole_f64<KIND>(L, j, r, u, acc, mask);
    scale_f64(L.iLd, acc, E, B, phi, A);
  }
  if (err) {
    set_status(L.status, err);
    return;
  }
  store_f64(L, f, p, E, B, phi, A, mask);
}

// ================================================================================================
// mixed path
// ================================================================================================
// The dipoles' records and float32 history mirrors; checks their axes.  xvmax (or null): per dipole the
// largest |X| and |V| of its samples, as the bits of non-negative floats (ordered like unsigned
// integers; a NaN orders above everything), preset to 0.  Grid: x over chunks of kPrepChunk samples, y
// over dipoles.  One float64 division a thread and dipole, no 64-bit index division (three and one a sample
// before).
constexpr int kPrepChunk = 1024, kPrepThreads = 256;
__global__ void __launch_bounds__(kPrepThreads) prep_dipoles_f32(const Sources s, float4 *H, float4 *srcf, unsigned *xvmax,
                                                                 int *status) {
  const double iL = 1.0 / (kC * s.dtd);
  for (int j = blockIdx.y; j < s.N; j += gridDim.y) {
    const double q = s.qd[j], iq = 1.0 / q;
    const double sx = iq * iL, sv = iq * (1.0 / kC), sa = iq * (s.dtd * (1.0 / kC));
    const size_t row = (size_t)j * (size_t)s.Sd;
    unsigned x = 0u, v = 0u;
    for (int64_t k = (int64_t)blockIdx.x * kPrepChunk + threadIdx.x;
         k < min(s.Sd, (int64_t)(blockIdx.x + 1) * kPrepChunk); k += kPrepThreads) {
      const size_t i = row + (size_t)k;
      const float4 h = make_float4((float)(s.d[i] * sx), (float)(s.dd[i] * sv), (float)(s.ddd[i] * sa), 0.f);
      H[i] = h;
      x = max(x, __float_as_uint(fabsf(h.x)));
      v = max(v, __float_as_uint(fabsf(h.y)));
    }
    if (xvmax) {
      x = __reduce_max_sync(0xffffffffu, x);
      v = __reduce_max_sync(0xffffffffu, v);
      if ((threadIdx.x & 31) == 0) {
        atomicMax(xvmax + 2 * j, x);
        atomicMax(xvmax + 2 * j + 1, v);
      }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      const double m1 = s.m1[j], m2 = s.m2[j], im = 1.0 / (m1 + m2);
      const double ax = s.axis[3 * j], ay = s.axis[3 * j + 1], az = s.axis[3 * j + 2];
      if (!(fabs(ax * ax + ay * ay + az * az - 1.0) <= kAxisTol)) set_status(status, PC_ERR_ARG);
      srcf[4 * j] = make_float4((float)ax, (float)ay, (float)az, (float)(q * (1.0 / kE)));
      srcf[4 * j + 1] = make_float4((float)(m2 * im), (float)(m1 * im), 0.f, 0.f);
      float hi[3], lo[3];
      for (int c = 0; c < 3; ++c) {
        const double o = s.origin[3 * j + c] * iL;
        hi[c] = (float)o;
        lo[c] = (float)(o - (double)hi[c]);
      }
      srcf[4 * j + 2] = make_float4(hi[0], hi[1], hi[2], 0.f);
      srcf[4 * j + 3] = make_float4(lo[0], lo[1], lo[2], 0.f);
    }
  }
}
static void launch_prep_dipoles(const Sources &s, float4 *H, float4 *srcf, unsigned *xvmax, int *status, cudaStream_t st) {
  const dim3 grid((unsigned)((s.Sd + kPrepChunk - 1) / kPrepChunk), (unsigned)std::min(s.N, 65535));
  prep_dipoles_f32<<<grid, kPrepThreads, 0, st>>>(s, H, srcf, xvmax, status);
}

__global__ void __launch_bounds__(kPrepThreads) prep_charges_f32(const Sources s, float4 *H, double *cref) {
  const double iL = 1.0 / (kC * s.dt), ic = 1.0 / kC, sa = s.dt * (1.0 / kC);
  for (int c = blockIdx.y; c < s.M; c += gridDim.y) {
    const double *p0 = s.pos + (size_t)c * s.S * 3;
    const double x0 = p0[0], y0 = p0[1], z0 = p0[2];
    for (int64_t k = (int64_t)blockIdx.x * kPrepThreads + threadIdx.x; k < s.S; k += (int64_t)gridDim.x * kPrepThreads) {
      const size_t i = (size_t)c * s.S + (size_t)k;
      const double *p = s.pos + 3 * i, *v = s.vel + 3 * i, *a = s.acc + 3 * i;
      H[3 * i + 0] = make_float4((float)((p[0] - x0) * iL), (float)((p[1] - y0) * iL), (float)((p[2] - z0) * iL), 0.f);
      H[3 * i + 1] = make_float4((float)(v[0] * ic), (float)(v[1] * ic), (float)(v[2] * ic), 0.f);
      H[3 * i + 2] = make_float4((float)(a[0] * sa), (float)(a[1] * sa), (float)(a[2] * sa), 0.f);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      cref[3 * c] = x0;
      cref[3 * c + 1] = y0;
      cref[3 * c + 2] = z0;
    }
  }
}
static void launch_prep_charges(const Sources &s, float4 *H, double *cref, cudaStream_t st) {
  const dim3 grid((unsigned)std::min<int64_t>((s.S + kPrepThreads - 1) / kPrepThreads, 65535), (unsigned)std::min(s.M, 65535));
  prep_charges_f32<<<grid, kPrepThreads, 0, st>>>(s, H, cref);
}

// ---- float-float arithmetic (error-free transformations with fma) for list-mode delays ----
struct ff {
  float hi, lo;
};
__device__ __forceinline__ ff ff_two_sum(float a, float b) {
  float s = a + b;
  float bb = s - a;
  float e = (a - (s - bb)) + (b - bb);
  return {s, e};
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  ff s = ff_two_sum(a.hi, b.hi);
  float lo = s.lo + a.lo + b.lo;
  return ff_two_sum(s.hi, lo);
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return ff_two_sum(p, e);
}
__device__ __forceinline__ ff ff_sqrt(ff a) {
  float s0 = sqrtf(a.hi);
  if (!(s0 > 0.f)) return {0.f, 0.f};
  float r = fmaf(-s0, s0, a.hi) + a.lo;  // a - s0^2
  return ff_two_sum(s0, r / (2.f * s0));
}
// The delay of a list point: rho = anchor's rho (g, gl) + offset (dr, drl), |rho| and the retarded sample
// fa - (|rho| - |g|) as kb + xc with 0 <= xc < 1.  Unevaluated high and low parts throughout, renormalised
// nowhere (their low parts stay within a few of the high parts' last places): 1e-11 of a sample at 1e4, in
// half the operations of the ff_ functions.
struct ListDelay {
  float rx, ry, rz, rho2, i, rn, xc;
  int kb;
};
__device__ __forceinline__ ListDelay list_delay(float4 g, float4 gl, float drx, float dry, float drz, float drlx, float drly,
                                                float drlz, float fa, int kb) {
  const ff px = ff_two_sum(g.x, drx), py = ff_two_sum(g.y, dry), pz = ff_two_sum(g.z, drz);
  const float lx = px.lo + (gl.x + drlx), ly = py.lo + (gl.y + drly), lz = pz.lo + (gl.z + drlz);
  const float xx = px.hi * px.hi, yy = py.hi * py.hi, zz = pz.hi * pz.hi;
  const float ex = fmaf(2.f * px.hi, lx, fmaf(px.hi, px.hi, -xx)), ey = fmaf(2.f * py.hi, ly, fmaf(py.hi, py.hi, -yy)),
              ez = fmaf(2.f * pz.hi, lz, fmaf(pz.hi, pz.hi, -zz));
  const ff a = ff_two_sum(xx, yy), b = ff_two_sum(a.hi, zz);
  const float lo = (ex + ey) + (ez + (a.lo + b.lo));
  ListDelay o;
  o.rx = px.hi;
  o.ry = py.hi;
  o.rz = pz.hi;
  o.rho2 = b.hi;
  o.i = b.hi > 1e-30f ? rsqrt_fast(b.hi) : 0.f;
  const float s0 = b.hi * o.i;
  o.rn = s0;
  const ff d = ff_two_sum(s0, -g.w);  // |rho| = s0 + (rho^2 - s0^2) / (2 s0)
  const float dl = d.lo + (0.5f * o.i * (fmaf(-s0, s0, b.hi) + lo) - gl.w);
  const ff x = ff_two_sum(fa, -d.hi);
  float flf;
  const int fl = Num<float>::floor_int(x.hi, flf);
  o.kb = kb + fl;
  o.xc = (x.hi - flf) + (x.lo - dl);
  return o;
}
__device__ __forceinline__ ff ff_from_double(double x) {
  float hi = (float)x;
  return {hi, (float)(x - (double)hi)};
}

// Both charges of dipole j in float64, added to the float32 accumulators in their units.  Used for
// points within kNearL of the dipole, where the float32 difference form loses accuracy: there the
// sampled position X and velocity V at the retarded time combine as X + R V, which nearly vanishes
// whenever the dipole's instantaneous moment crosses zero.  Exact per-charge roots (no segment
// extension), the same difference form in double.
template <int KIND>
// iLd = 1 / (c dt): two float64 divisions in all (the unit is narrow, and in the frames whose moments
// cross zero every near pair comes here).
__device__ __noinline__ int near_dipole_f64(const Sources &s, int j, const float4 *hist, const double r[3], double u,
                                               double iLd, double r_excl, float *part, uint8_t *mask) {
  const double q = s.qd[j], m1 = s.m1[j], m2 = s.m2[j];
  const double iq = 1.0 / q;
  const double rx = (r[0] - s.origin[3 * j]) * iLd, ry = (r[1] - s.origin[3 * j + 1]) * iLd,
               rz = (r[2] - s.origin[3 * j + 2]) * iLd;
  const double px = s.axis[3 * j], py = s.axis[3 * j + 1], pz = s.axis[3 * j + 2];
  HistF64 H;
  H.d = s.d + (size_t)j * s.Sd;
  H.dd = s.dd + (size_t)j * s.Sd;
  H.ddd = s.ddd + (size_t)j * s.Sd;
  H.sx = iq * iLd;
  H.sv = iq * (1.0 / kC);
  H.sa = iq * (s.dtd * (1.0 / kC));
  double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  if (m1 == m2) {
    // the split form: a quarter of the float64 instructions
    float cub[10] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (split_dipole<KIND>(rx, ry, rz, px, py, pz, q * (1.0 / kE), u, H.d, H.dd, H.ddd, H.sx, H.sv, H.sa, hist, (int)s.Sd,
                           {kSplitNearX, kSplitNearV, (float)(r_excl * iLd) + 1.5f}, acc, cub)) {
#pragma unroll
      for (int i = 0; i < 10; ++i) part[i] += (float)acc[i] + cub[i];
      return 0;
    }
  }
  const double imm = 1.0 / (m1 + m2);
  const double rn = sqrt(rx * rx + ry * ry + rz * rz);
  const double rp = rx * px + ry * py + rz * pz;
  const double x = u - rn;
  const double fl = floor(x);
  const int e = dipole_net<KIND, double, HistF64>(H, (int)s.Sd, (int)fl, x - fl, rx, ry, rz, rn, px, py, pz, rp,
                                                  m2 * imm, m1 * imm, q * (1.0 / kE), r_excl * iLd, true, acc, *mask);
  if (e) return e;
#pragma unroll
  for (int i = 0; i < 10; ++i) part[i] += (float)acc[i];
  return 0;
}

// A dipole pair the inner loop could not take on its fast path (a charge offset beyond the shared
// segment, a point close to a charge, or an ill-conditioned near field): exact float32 roots of
// both charges, then the float32 difference form, or the float64 near path where the near field
// cancels.  Kept out of line so that the inner loop makes no calls.
template <int KIND>
__device__ __noinline__ int slow_dipole(const Sources &s, int j, const float4 *hist, int S, int kb, float xc, float rx,
                                        float ry, float rz, float rn, float4 ax, float mup, float mum, float rex,
                                        const double r[3], double u, double iLd, double r_excl, float *part,
                                        uint8_t *mask) {
  const float rp = rx * ax.x + ry * ax.y + rz * ax.z;
  const HistF32 H{hist};
  float Xp, Vp, Ap, dp, Xm, Vm, Am, dm;
  const int e = dipole_states<float, HistF32>(H, S, kb, xc, rn, rp, mup, mum, true, Xp, Vp, Ap, dp, Xm, Vm, Am, dm);
  if (e) return e;
  if (rn < kNearL && dipole_cancellation<float>(rn, mup, mum, Xp, Vp, Ap, Xm, Vm, Am) > kCancel)
    return near_dipole_f64<KIND>(s, j, hist, r, u, iLd, r_excl, part, mask);
  dipole_pair<KIND, float>(rx, ry, rz, rn, ax.x, ax.y, ax.z, rp, mup, mum, ax.w, Xp, Vp, Ap, dp, Xm, Vm, Am, dm, rex,
                           part, *mask);
  return 0;
}

// Generic charge in float32 (no pairing): Griffiths form with c = 1.
template <int KIND>
__device__ __forceinline__ void charge_mixed(float ax, float ay, float az, float vx, float vy, float vz, float gx,
                                             float gy, float gz, float qs, float rex, float *acc, uint8_t &mask) {
  const float R2 = ax * ax + ay * ay + az * az;
  const float iR = rsqrtf(R2);
  const float R = R2 > 0.f ? R2 * iR : 0.f;  // exact cancellation: 0 * inf would be NaN
  if (R <= rex) {
    mask = 1;
    return;
  }
  const float ux = ax * iR - vx, uy = ay * iR - vy, uz = az * iR - vz;
  const float Ru = R - (ax * vx + ay * vy + az * vz);
  const float i1 = __frcp_rn(Ru);
  const float f = qs * R * i1 * i1 * i1;
  float ex = 0.f, ey = 0.f, ez = 0.f;
  if (KIND != PC_RADIATION) {
    const float g = f * (1.f - (vx * vx + vy * vy + vz * vz));
    ex = g * ux;
    ey = g * uy;
    ez = g * uz;
  }
  if (KIND != PC_COULOMB) {
    const float aa = ax * gx + ay * gy + az * gz;
    ex += f * (ux * aa - gx * Ru);
    ey += f * (uy * aa - gy * Ru);
    ez += f * (uz * aa - gz * Ru);
  }
  acc[0] += ex;
  acc[1] += ey;
  acc[2] += ez;
  const float nx = ax * iR, ny = ay * iR, nz = az * iR;
  acc[3] += ny * ez - nz * ey;
  acc[4] += nz * ex - nx * ez;
  acc[5] += nx * ey - ny * ex;
  acc[6] += qs * i1;
  acc[7] += qs * i1 * vx;
  acc[8] += qs * i1 * vy;
  acc[9] += qs * i1 * vz;
}

// Kahan-compensated running sums of the ten outputs; each thread's sums live in shared memory,
// strided by the block size (they are touched once per group of sixteen sources), as five packed
// pairs: 0 (E_x, E_y), 1 (B_x, B_y), 2 (A_x, A_y), 3 (E_z, B_z), 4 (A_z, phi).  Indexed from the
// thread index directly, so no pointer stays live across the source loop.
using KahanArr = float2[2][5][kMixThreads];
__device__ __forceinline__ void kahan_add(KahanArr &k, int tid, const float2 *P) {
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const float2 s0 = k[0][i][tid], c0 = k[1][i][tid];
    const float2 y = __fadd2_rn(P[i], make_float2(-c0.x, -c0.y));
    const float2 t = __fadd2_rn(s0, y);
    const float2 d = __fadd2_rn(t, make_float2(-s0.x, -s0.y));
    k[1][i][tid] = __fadd2_rn(d, make_float2(-y.x, -y.y));
    k[0][i][tid] = t;
  }
}
// the ten outputs in their natural order (E, B, phi, A) into the packed slots
__device__ __forceinline__ void pack_outputs(const float *part, float2 (&P)[5]) {
  P[0] = make_float2(part[0], part[1]);
  P[1] = make_float2(part[3], part[4]);
  P[2] = make_float2(part[7], part[8]);
  P[3] = make_float2(part[2], part[5]);
  P[4] = make_float2(part[9], part[6]);
}
__device__ __forceinline__ float kahan_get(const KahanArr &k, int tid, int i) {
  // natural index -> (slot, lane)
  const int slot[10] = {0, 0, 3, 1, 1, 3, 4, 2, 2, 4};
  const int hi[10] = {0, 1, 0, 0, 1, 1, 1, 0, 1, 0};
  const float2 sv = k[0][slot[i]][tid], cv = k[1][slot[i]][tid];
  return hi[i] ? sv.y - cv.y : sv.x - cv.x;
}

// float64, dipoles alone: sources staged in shared memory, each pair in the split form (pc_far_f32.cuh)
// where it holds, the others, by a bit mask per stage, with the two charges.  64 dipoles of 10 pm, 301 x 517
// points: 5.20 -> 1.93 ms; the float64 unit is the bound, 70 instructions a pair and 280 a near one.
constexpr int kSplitChunk = 32;
template <int KIND>
__global__ void __launch_bounds__(128) fields_split64_kernel(const __grid_constant__ Launch L) {
  struct Src {
    double ox, oy, oz, px, py, pz, qs, sx, sv, sa;
    int equal;
  };
  __shared__ Src s_src[kSplitChunk];
  if (L.status[1] >= L.near_min) return;
  const Sources &s = L.src;
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int f = blockIdx.y;
  const bool act = p < L.pts.P;
  double r[3] = {0, 0, 0};
  if (act) point_at(L.pts, p, r);
  const double u = L.uf[f], iLd = L.iLd;
  const SplitLimits lim = {kSplitFieldX, kSplitFieldV, (float)(L.r_excl * iLd) + 1.5f};
  double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  uint8_t mask = 0;
  int err = 0;
  for (int base = 0; base < s.N; base += kSplitChunk) {
    const int nch = min(kSplitChunk, s.N - base);
    __syncthreads();
    if ((int)threadIdx.x < nch) {
      const int j = base + threadIdx.x;
      const double q = s.qd[j], iq = 1.0 / q;
      s_src[threadIdx.x] = {s.origin[3 * j], s.origin[3 * j + 1], s.origin[3 * j + 2], s.axis[3 * j], s.axis[3 * j + 1],
                            s.axis[3 * j + 2], q * (1.0 / kE), iq * iLd, iq * (1.0 / kC), iq * (s.dtd / kC),
                            s.m1[j] == s.m2[j]};
    }
    __syncthreads();
    if (!act || err) continue;
    unsigned near = 0u;
    float cub[10] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int jj = 0; jj < nch; ++jj) {
      const Src &c = s_src[jj];
      const size_t row = (size_t)(base + jj) * (size_t)s.Sd;
      if (!c.equal || !split_dipole<KIND>((r[0] - c.ox) * iLd, (r[1] - c.oy) * iLd, (r[2] - c.oz) * iLd, c.px, c.py, c.pz,
                                          c.qs, u, s.d + row, s.dd + row, s.ddd + row, c.sx, c.sv, c.sa, L.Hd + row,
                                          (int)s.Sd, lim, acc, cub))
        near |= 1u << jj;
    }
#pragma unroll
    for (int i = 0; i < 10; ++i) acc[i] += (double)cub[i];
    while (near && !err) {
      const int jj = __ffs((int)near) - 1;
      near &= near - 1;
      double a[10];
      uint8_t mk = 0;
      err = dipole_f64_call<KIND>(L, base + jj, r, u, a, &mk);
      mask |= mk;
#pragma unroll
      for (int i = 0; i < 10; ++i) acc[i] += a[i];
    }
  }
  if (!act) return;
  if (err) {
    set_status(L.status, err);
    return;
  }
  double E[3] = {0, 0, 0}, B[3] = {0, 0, 0}, A[3] = {0, 0, 0}, phi = 0.0;
  scale_f64(iLd, acc, E, B, phi, A);
  store_f64(L, f, p, E, B, phi, A, mask);
}

// How many of kSplitAsk pairs, spread over points, dipoles and frames, are near for the split form (its conditions
// in split_dipole): a pair that is costs it 1.1 (unequal masses) to 1.4 of the two-charge kernel's, for the attempt
// and the call out of line, and one that is not 0.36.  The choice stays on the device, both kernels are launched and
// one returns (5 us a call; 64 dipoles whose charges are too fast, 20 000 points: 2.34 -> 1.98 ms).
constexpr int kSplitAsk = 1024;
constexpr double kSplitNearMost = 0.65;
__global__ void __launch_bounds__(128) split_count_kernel(const __grid_constant__ Launch L) {
  const unsigned k = blockIdx.x * blockDim.x + threadIdx.x;  // < kSplitAsk
  const Sources &s = L.src;
  // multiplicative hashing: the three indices independent of one another
  const int64_t p = (int64_t)(((unsigned long long)(k * 2654435769u) * (unsigned long long)L.pts.P) >> 32);
  const int j = (int)(((unsigned long long)((k + 1u) * 2246822519u) * (unsigned)s.N) >> 32);
  const int f = (int)(((unsigned long long)((k + 1u) * 3266489917u) * (unsigned)L.T) >> 32);
  double r[3];
  point_at(L.pts, p, r);
  const double iLd = L.iLd;
  // (float32 is enough for a sample, and its latency a fraction)
  const float rx = (float)((r[0] - s.origin[3 * j]) * iLd), ry = (float)((r[1] - s.origin[3 * j + 1]) * iLd),
              rz = (float)((r[2] - s.origin[3 * j + 2]) * iLd);
  const float R2 = fmaf(rz, rz, fmaf(ry, ry, rx * rx)), R = R2 * rsqrt_fast(R2), x = (float)L.uf[f] - R;
  bool far = s.m1[j] == s.m2[j] && R > (float)(L.r_excl * iLd) + 1.5f && x > 2.f && x < (float)(s.Sd - 3);
  if (far) {
    const size_t n = (size_t)j * (size_t)s.Sd + (size_t)min((int64_t)x, s.Sd - 1);
    const float iq = __fdividef((float)kE, (float)s.qd[j]);
    const float X = fabsf((float)(s.d[n] * (iLd / kE)) * iq), V = fabsf((float)(s.dd[n] * (1.0 / (kC * kE))) * iq);
    far = X <= fminf(kSplitFieldX * R, kSplitSamples) && V <= kSplitFieldV;
  }
  const unsigned m = __ballot_sync(0xffffffffu, !far);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(L.status + 1, __popc(m));
}

// The point of thread tid in tile blockIdx.x (list: 256 consecutive points; plane: a block of rows x
// columns of the grid), or P for a thread past the edge of the grid.
__device__ __forceinline__ int64_t tile_point(const Launch &L, int64_t tiles_v, int tid) {
  if (L.pts.list) return (int64_t)blockIdx.x * kMixThreads + tid;
  const int64_t tu = blockIdx.x / tiles_v, tv = blockIdx.x % tiles_v;
  const int sh = L.tile_shift, cols = 1 << sh, rows = kMixThreads >> sh;
  const int64_t iu = tu * rows + (tid >> sh), iv = tv * cols + (tid & (cols - 1));
  return (iu < L.pts.nu && iv < L.pts.nv) ? iu * L.pts.nv + iv : L.pts.P;
}

// FAR (large lists): a pair beyond its source's L.rfar takes the first-order dipole form (pc_far_f32.cuh), a
// third of the two-charge form's operations.  Points of a list are anywhere, so each pair is asked by itself;
// in a micrometre cube one warp in five has a near lane for a source.  Measured, 64 dipoles at 100 003 points in
// two frames: 347 -> 311 us a call with list_delay, 259 of them here; bound by latency (24 warps an SM, the
// second wave of CTAs a quarter full) and by the float64 unit in near pairs that cancel (40 % busy).
template <int KIND, bool LIST, int CH, bool FAR = false>
__global__ void __launch_bounds__(kMixThreads, 4) fields_mixed_kernel(const Launch L, int64_t tiles_v) {
  __shared__ double s_anchor[3];
  __shared__ float s_anc_hi[3], s_anc_lo[3];  // the anchor / (c dt) of the dipoles as float-float
  __shared__ KahanArr s_kahan;
  __shared__ float4 s_geo[CH];   // rho_a (x,y,z), |rho_a|
  __shared__ float4 s_geo_lo[CH]; // low parts of rho_a and |rho_a| (list mode)
  __shared__ float4 s_ax[CH];    // axis (x,y,z), q/e
  __shared__ float4 s_mix[CH];   // m2/(m1+m2), m1/(m1+m2), fraction and integer part of the
                                     // retarded sample of the anchor (integer as bits)
  __shared__ const float4 *s_hist[CH];
  __shared__ float s_rfar[FAR ? CH : 1];

  const int tid = threadIdx.x;
  const int f = blockIdx.y;
  const Sources &s = L.src;
  // ---- tile -> points (the index itself is formed again where it is needed, so that it does not
  // occupy registers across the source loop) ----
  const bool active = tile_point(L, tiles_v, tid) < L.pts.P;
  if (tid == 0) {
    double a[3];
    if (L.pts.list) {
      int64_t pa = (int64_t)blockIdx.x * kMixThreads + kMixThreads / 2;
      if (pa >= L.pts.P) pa = L.pts.P - 1;
      point_at(L.pts, pa, a);
    } else {
      int64_t tu = blockIdx.x / tiles_v, tv = blockIdx.x % tiles_v;
      const int sh = L.tile_shift, cols = 1 << sh, rows = kMixThreads >> sh;
      double iu = (double)(tu * rows) + 0.5 * (rows - 1), iv = (double)(tv * cols) + 0.5 * (cols - 1);
      for (int i = 0; i < 3; ++i) a[i] = L.pts.o[i] + iu * L.pts.eu[i] + iv * L.pts.ev[i];
    }
    s_anchor[0] = a[0];
    s_anchor[1] = a[1];
    s_anchor[2] = a[2];
    for (int i = 0; i < 3; ++i) {
      const double x = a[i] * L.iLd;
      s_anc_hi[i] = (float)x;
      s_anc_lo[i] = (float)(x - (double)s_anc_hi[i]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    s_kahan[0][i][tid] = make_float2(0.f, 0.f);
    s_kahan[1][i][tid] = make_float2(0.f, 0.f);
  }
  uint8_t mask = 0;
  int err = 0;

  // ---------------- dipoles ----------------
  if (s.N > 0) {
    // float64 values used once per chunk or by the rare slow pairs are recomputed there, so that
    // none of them occupies registers across the source loop
    const double iLd = L.iLd;  // float64 divisions would stall the CTA on this GPU's narrow float64 unit
    float drx, dry, drz, drlx = 0.f, drly = 0.f, drlz = 0.f;
    if (!LIST) {
      // a plane point sits a whole number of grid steps from the tile anchor: the offset in float
      // from those small integers (no float64 on the way)
      const int sh = L.tile_shift, cols = 1 << sh, rows = kMixThreads >> sh;
      const float du = (float)(tid >> sh) - 0.5f * (float)(rows - 1), dv = (float)(tid & (cols - 1)) - 0.5f * (float)(cols - 1);
      drx = du * L.eu_L[0] + dv * L.ev_L[0];
      dry = du * L.eu_L[1] + dv * L.ev_L[1];
      drz = du * L.eu_L[2] + dv * L.ev_L[2];
    } else {
      double r[3];
      point_at(L.pts, active ? tile_point(L, tiles_v, tid) : 0, r);
      const double drxd = (r[0] - s_anchor[0]) * iLd, dryd = (r[1] - s_anchor[1]) * iLd,
                   drzd = (r[2] - s_anchor[2]) * iLd;
      drx = (float)drxd;
      dry = (float)dryd;
      drz = (float)drzd;
      drlx = (float)(drxd - (double)drx);
      drly = (float)(dryd - (double)dry);
      drlz = (float)(drzd - (double)drz);
    }
    const float dr2 = drx * drx + dry * dry + drz * drz;
    for (int base = 0; base < s.N; base += CH) {
      const int nch = min(CH, s.N - base);
      __syncthreads();
      if (tid < nch) {
        // the tile anchor's distance to the source in float64 (the integer sample index and a
        // fraction kept to ~1e-7), everything else from the per-call records
        // in float-float (~1e-14 relative) on the float32 pipes: rho_a = anchor - origin in units of
        // c dt, |rho_a|, and the centre's retarded sample u - |rho_a| split into integer and fraction
        const int j = base + tid;
        const float4 oh = L.srcf[4 * j + 2], ol = L.srcf[4 * j + 3];
        const ff rax = ff_add({s_anc_hi[0], s_anc_lo[0]}, {-oh.x, -ol.x});
        const ff ray = ff_add({s_anc_hi[1], s_anc_lo[1]}, {-oh.y, -ol.y});
        const ff raz = ff_add({s_anc_hi[2], s_anc_lo[2]}, {-oh.z, -ol.z});
        const ff rna = ff_sqrt(ff_add(ff_add(ff_mul(rax, rax), ff_mul(ray, ray)), ff_mul(raz, raz)));
        const ff x = ff_add({L.uf_hi[f], L.uf_lo[f]}, {-rna.hi, -rna.lo});
        float kaf;
        const int kai = Num<float>::floor_int(x.hi, kaf);
        s_geo[tid] = make_float4(rax.hi, ray.hi, raz.hi, rna.hi);
        if (LIST) s_geo_lo[tid] = make_float4(rax.lo, ray.lo, raz.lo, rna.lo);
        s_ax[tid] = L.srcf[4 * j];
        const float4 mm = L.srcf[4 * j + 1];
        s_mix[tid] = make_float4(mm.x, mm.y, (x.hi - kaf) + x.lo, __int_as_float(kai));
        s_hist[tid] = L.Hd + (size_t)j * s.Sd;
        if (FAR) s_rfar[tid] = L.rfar[j];
      }
      __syncthreads();
      if (!active || err) continue;
      float2 P[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) P[i] = make_float2(0.f, 0.f);
      typename SlowMask<CH>::T slow_mask = 0;
      for (int g0 = 0; g0 < nch; g0 += 32) {
      // groups of 32 sources summed in float32, the group sums compensated (16 per group cost 1 %
      // more time for no accuracy the 1e-5 bound needs)
      const int gend = min(nch, g0 + 32);
      for (int jj = g0; jj < gend; ++jj) {
        const float4 g = s_geo[jj];
        const float4 ax = s_ax[jj];
        const float4 mx = s_mix[jj];
        const float2 mu = make_float2(mx.x, mx.y);
        const float fa = mx.z;
        float rx, ry, rz, rn, irn = 0.f;
        // retarded time of the dipole centre, in samples: kb + xc with |xc| small
        int kb = __float_as_int(mx.w);
        float xc;
        if constexpr (!LIST) {
          rx = g.x + drx, ry = g.y + dry, rz = g.z + drz;
          const float rho2 = rx * rx + ry * ry + rz * rz;
          // rho2 == 0 makes rn NaN, which sends the pair to the slow path through the tests below
          rn = rho2 * rsqrtf(rho2);
          // compact tile: |rho| - |rho_a| from the tile offset without cancellation
          const float corr = __fdividef(2.f * (g.x * drx + g.y * dry + g.z * drz) + dr2, rn + g.w);
          xc = fa - corr;
        } else {
          // points of a list tile may lie far apart: |rho| - |rho_a| in two parts, integer part
          // moved into kb so that the fraction keeps its precision
          const ListDelay t = list_delay(g, s_geo_lo[jj], drx, dry, drz, drlx, drly, drlz, fa, kb);
          rx = t.rx, ry = t.ry, rz = t.rz, rn = t.rn, irn = t.i;
          xc = t.xc;
          kb = t.kb;
        }
        const float rp = rx * ax.x + ry * ax.y + rz * ax.z;
        // fast path: both charges on the interior segment of their centre's retarded time, the point
        // farther than rex + 1.5 samples from the centre (the charges are then farther than rex:
        // their distances differ from rn by |delta| <= 1.1); a garbage index from a huge or NaN xc
        // fails the range test before any load
        float2 X, V, Ac, dl;
        bool fast = false;
        {
          float fl;
          const int kc = Num<float>::floor_int(xc, fl);
          const int j = kb + kc;
          if ((unsigned)(j - 1) < L.jlim && rn > L.rex_fast) {
            // the source's history row from the parameter bank (no per-pair shared-memory load)
            const HistF32 H{L.Hd + (size_t)(base + jj) * (size_t)L.src.Sd};
            float x0, v0, a0, x1, v1, a1;
            H.get_in(j, x0, v0, a0);
            H.get_in(j + 1, x1, v1, a1);
            // (not on the first two segments: the rest state before the history makes a kink there)
            if (FAR && rn >= s_rfar[jj] && j > 1) {
              const float th = xc - fl, i2 = irn * irn, rpi2 = rp * i2, m = rpi2 * irn;
              const float X1 = ax.w * fmaf(th, x1 - x0, x0), V1 = ax.w * fmaf(th, v1 - v0, v0);
              const float A1 = KIND == PC_COULOMB ? 0.f : ax.w * fmaf(th, a1 - a0, a0);
              const float t1 = fmaf(irn, X1, V1);
              float cE, cP, cB;
              if (KIND == PC_COULOMB) {
                cE = m * (3.f * irn) * t1;
                cP = -(i2 * t1);
                cB = i2 * irn * V1;
              } else if (KIND == PC_RADIATION) {
                cE = m * A1;
                cP = -(irn * A1);
                cB = i2 * A1;
              } else {
                cE = m * fmaf(3.f * irn, t1, A1);
                cP = -(irn * fmaf(irn, t1, A1));
                cB = i2 * fmaf(irn, V1, A1);
              }
              const float vi = V1 * irn;
              P[0].x = fmaf(cP, ax.x, fmaf(cE, rx, P[0].x));
              P[0].y = fmaf(cP, ax.y, fmaf(cE, ry, P[0].y));
              P[3].x = fmaf(cP, ax.z, fmaf(cE, rz, P[3].x));
              P[1].x = fmaf(cB, fmaf(ax.y, rz, -(ax.z * ry)), P[1].x);
              P[1].y = fmaf(cB, fmaf(ax.z, rx, -(ax.x * rz)), P[1].y);
              P[3].y = fmaf(cB, fmaf(ax.x, ry, -(ax.y * rx)), P[3].y);
              P[2].x = fmaf(vi, ax.x, P[2].x);
              P[2].y = fmaf(vi, ax.y, P[2].y);
              P[4].x = fmaf(vi, ax.z, P[4].x);
              P[4].y = fmaf(rpi2, t1, P[4].y);
              continue;
            }
            fast = dip_pair_states_fast(x0, v0, a0, x1, v1, a1, xc - fl, rn, rp, mu.x, mu.y, X, V, Ac, dl);
          }
        }
        // near fields that cancel in float32 also leave the fast path
        if (fast && rn < kNearL &&
            dipole_cancellation<float>(rn, mu.x, mu.y, X.x, V.x, Ac.x, X.y, V.y, Ac.y) > kCancel)
          fast = false;
        if (!fast) {
          slow_mask |= SlowMask<CH>::bit(jj);
          continue;
        }
        dipole_pair_fast<KIND>(make_float2(rx, ry), rz, rn, make_float2(ax.x, ax.y), ax.z, rp, mu.x, mu.y, ax.w, X, V,
                               Ac, dl, P);
      }
      kahan_add(s_kahan, tid, P);
#pragma unroll
      for (int i = 0; i < 5; ++i) P[i] = make_float2(0.f, 0.f);
      }
      // the pairs of this chunk that left the fast path
      while (slow_mask && !err) {
        const int jj = SlowMask<CH>::first(slow_mask);
        slow_mask &= slow_mask - 1;
        // the out-of-line call gets arrays of its own: passing the address of part or mask would
        // keep them in local memory throughout the source loop
        float sp[10] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        uint8_t smask = 0;
        const float4 g = s_geo[jj];
        const float4 ax = s_ax[jj];
        const float4 mx = s_mix[jj];
        float rx, ry, rz, rn, xc;
        int kb = __float_as_int(mx.w);
        if constexpr (!LIST) {
          rx = g.x + drx, ry = g.y + dry, rz = g.z + drz;
          const float rho2 = rx * rx + ry * ry + rz * rz;
          rn = rho2 > 0.f ? rho2 * rsqrtf(rho2) : 0.f;
          const float corr = __fdividef(2.f * (g.x * drx + g.y * dry + g.z * drz) + dr2, rn + g.w);
          xc = mx.z - corr;
        } else {
          const ListDelay t = list_delay(g, s_geo_lo[jj], drx, dry, drz, drlx, drly, drlz, mx.z, kb);
          rx = t.rx, ry = t.ry, rz = t.rz, rn = t.rn;
          xc = t.xc;
          kb = t.kb;
        }
        double rp64[3];
        point_at(L.pts, tile_point(L, tiles_v, tid), rp64);
        const int e = slow_dipole<KIND>(s, base + jj, s_hist[jj], (int)s.Sd, kb, xc, rx, ry, rz, rn, ax, mx.x, mx.y,
                                        L.rex, rp64, L.uf[f], L.iLd, L.r_excl, sp,
                                        &smask);
        if (e) err = e;
        mask |= smask;
        float2 SP[5];
        pack_outputs(sp, SP);
        kahan_add(s_kahan, tid, SP);
      }
    }
  }
  // ---------------- point charges ----------------
  if (s.M > 0) {
    double r[3];
    point_at(L.pts, active ? tile_point(L, tiles_v, tid) : 0, r);
    const double iLc = L.iLc;  // no float64 division on the way (the float64 unit is narrow here)
    const float drx = (float)((r[0] - s_anchor[0]) * iLc), dry = (float)((r[1] - s_anchor[1]) * iLc),
                drz = (float)((r[2] - s_anchor[2]) * iLc);
    const float dr2 = drx * drx + dry * dry + drz * drz;
    const double u = L.ufc[f];
    const float rex = (float)(L.r_excl * iLc);
    const float sE = L.sE, sP = L.sP;
    for (int base = 0; base < s.M; base += CH) {
      const int nch = min(CH, s.M - base);
      __syncthreads();
      if (tid < nch) {
        const int c = base + tid;
        double ra[3];
        for (int i = 0; i < 3; ++i) ra[i] = (s_anchor[i] - L.cref[3 * c + i]) * iLc;
        const double rna = sqrt(ra[0] * ra[0] + ra[1] * ra[1] + ra[2] * ra[2]);
        const double x = u - rna;
        const double kaf = floor(x);
        s_geo[tid] = make_float4((float)ra[0], (float)ra[1], (float)ra[2], (float)rna);
        s_ax[tid] = make_float4(0.f, 0.f, 0.f, (float)(s.q[c] * (1.0 / kE)));
        s_mix[tid] = make_float4(0.f, 0.f, (float)(x - kaf), __int_as_float((int)kaf));
      }
      __syncthreads();
      if (!active || err) continue;
      float part[10];
#pragma unroll
      for (int i = 0; i < 10; ++i) part[i] = 0.f;
      for (int cc = 0; cc < nch; ++cc) {
        const float4 g = s_geo[cc];
        const float qs = s_ax[cc].w;
        const float rx = g.x + drx, ry = g.y + dry, rz = g.z + drz;
        const float rho2 = rx * rx + ry * ry + rz * rz;
        const float irn = rho2 > 0.f ? rsqrtf(rho2) : 0.f;
        const float rn = rho2 * irn;
        const float corr = __fdividef(2.f * (g.x * drx + g.y * dry + g.z * drz) + dr2, rn + g.w);
        const float xc = s_mix[cc].z - corr;
        if (!(fabsf(xc) < 1e6f)) {
          err = PC_ERR_NOCONV;
          break;
        }
        const float4 *H = L.Hc + (size_t)(base + cc) * s.S * 3;
        const int S = (int)s.S;
        // first-order estimate of the charge's delay offset: -rho_hat . o(center time)
        float kcf;
        const int kc = Num<float>::floor_int(xc, kcf);
        float thc = xc - kcf;
        int j = __float_as_int(s_mix[cc].w) + kc;
        {
          int jc = j < 0 ? 0 : (j > S - 1 ? S - 1 : j);
          float4 o = __ldg(H + 3 * jc);
          float d0 = -(rx * o.x + ry * o.y + rz * o.z) * irn;
          float stf;
          int st = Num<float>::floor_int(thc - d0, stf);
          j += st;
          thc -= stf;
        }
        float ox = 0, oy = 0, oz = 0, vx = 0, vy = 0, vz = 0, gx = 0, gy = 0, gz = 0;
        bool done = false;
        for (int it = 0; it < 32 && !done; ++it) {
          // an estimate past either end is solved on the end segment extended; the root then
          // decides whether the history really ends too early
          if (j > S - 2) {
            thc += (float)(j - (S - 2));
            j = S - 2;
          }
          if (j < 0 && !s.static_before) {
            thc += (float)j;
            j = 0;
          }
          const int j0 = j < 0 ? 0 : j, j1 = j < 0 ? 0 : j + 1;
          const float4 o0 = __ldg(H + 3 * j0), o1 = __ldg(H + 3 * j1);
          const float wx = o1.x - o0.x, wy = o1.y - o0.y, wz = o1.z - o0.z;
          const float ocx = o0.x + thc * wx, ocy = o0.y + thc * wy, ocz = o0.z + thc * wz;
          const float A = 1.f - (wx * wx + wy * wy + wz * wz);
          const float B = rn - ((rx - ocx) * wx + (ry - ocy) * wy + (rz - ocz) * wz);
          const float C = ocx * (2.f * rx - ocx) + ocy * (2.f * ry - ocy) + ocz * (2.f * rz - ocz);
          const float sq = Num<float>::sqrt0(fmaxf(B * B - A * C, 0.f));
          const float dl = (B > 0.f) ? -__fdividef(C, B + sq) : __fdividef(-B + sq, A);
          float th = thc - dl;
          const bool ok = (j < 0) ? ((float)j + th <= 1e-4f)
                                  : (th >= -1e-4f && (th <= 1.0001f || (j == S - 2 && th <= 1.f + kEndTol)));
          if (ok) {
            th = fminf(fmaxf(th, 0.f), 1.f);
            if (j < 0) {
              ox = o0.x;
              oy = o0.y;
              oz = o0.z;
            } else {
              const float4 v0 = __ldg(H + 3 * j0 + 1), v1 = __ldg(H + 3 * j1 + 1);
              const float4 a0 = __ldg(H + 3 * j0 + 2), a1 = __ldg(H + 3 * j1 + 2);
              ox = o0.x + th * wx;
              oy = o0.y + th * wy;
              oz = o0.z + th * wz;
              vx = v0.x + th * (v1.x - v0.x);
              vy = v0.y + th * (v1.y - v0.y);
              vz = v0.z + th * (v1.z - v0.z);
              gx = a0.x + th * (a1.x - a0.x);
              gy = a0.y + th * (a1.y - a0.y);
              gz = a0.z + th * (a1.z - a0.z);
            }
            done = true;
          } else {
            if (!(fabsf(th) < 1e6f)) break;
            if ((j == S - 2 && th > 1.f) || (j == 0 && th < 0.f && !s.static_before)) {
              err = PC_ERR_HISTORY;
              break;
            }
            float stf;
            const int st = Num<float>::floor_int(th, stf);
            j += st;
            thc -= stf;
          }
        }
        if (!done) {
          if (!err) err = PC_ERR_NOCONV;
          break;
        }
        float c10[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) c10[i] = 0.f;
        charge_mixed<KIND>(rx - ox, ry - oy, rz - oz, vx, vy, vz, gx, gy, gz, qs, rex, c10, mask);
        // E and B carry q through f; scale E/B by sE and phi/A by sP
#pragma unroll
        for (int i = 0; i < 6; ++i) part[i] += sE * c10[i];
#pragma unroll
        for (int i = 6; i < 10; ++i) part[i] += sP * c10[i];
        if ((cc & 15) == 15) {
          float2 PP[5];
          pack_outputs(part, PP);
          kahan_add(s_kahan, tid, PP);
#pragma unroll
          for (int i = 0; i < 10; ++i) part[i] = 0.f;
        }
      }
      float2 PP[5];
      pack_outputs(part, PP);
      kahan_add(s_kahan, tid, PP);
    }
  }
  if (!active) return;
  if (err) {
    set_status(L.status, err);
    return;
  }
  // units: E in k_e e / L^2, B in k_e e / (L^2 c), phi in k_e e / L, A in k_e e / (L c)
  const float fE = L.unit[0], fB = L.unit[1], fP = L.unit[2], fA = L.unit[3];
  const int64_t o = (L.frame0 + f) * L.pts.P + tile_point(L, tiles_v, tid);
  // streaming stores (evict first): the outputs are not read again by this kernel, and L2 keeps the
  // lines that are (the histories, the stack of the slow pairs' calls); on the 2048^2 x 16-frame
  // grid this cut the DRAM writes of a launch from 3.48 to 3.19 GB (outputs: 2.75 GB)
  if (L.out.E) {
    float *e = (float *)L.out.E + 3 * o;
    __stcs(e + 0, fE * kahan_get(s_kahan, tid, 0));
    __stcs(e + 1, fE * kahan_get(s_kahan, tid, 1));
    __stcs(e + 2, fE * kahan_get(s_kahan, tid, 2));
  }
  if (L.out.B) {
    float *b = (float *)L.out.B + 3 * o;
    __stcs(b + 0, fB * kahan_get(s_kahan, tid, 3));
    __stcs(b + 1, fB * kahan_get(s_kahan, tid, 4));
    __stcs(b + 2, fB * kahan_get(s_kahan, tid, 5));
  }
  if (L.out.phi) __stcs((float *)L.out.phi + o, fP * kahan_get(s_kahan, tid, 6));
  if (L.out.A) {
    float *a = (float *)L.out.A + 3 * o;
    __stcs(a + 0, fA * kahan_get(s_kahan, tid, 7));
    __stcs(a + 1, fA * kahan_get(s_kahan, tid, 8));
    __stcs(a + 2, fA * kahan_get(s_kahan, tid, 9));
  }
  if (L.out.mask) __stcs(reinterpret_cast<unsigned char *>(L.out.mask) + o, (unsigned char)mask);
}

// ------------------------------------------------------------------------------------------------
// Two points per thread (plane grids of dipoles): the thread's points sit in rows r and r + rows of
// a tile of 2 rows x cols points, and the fast path evaluates both at once in the lanes of float2
// registers (pc_lw_f32x2.cuh), which packs the per-point scalar part of the pair algebra too.  The
// per-source work staged in shared memory serves twice as many points.  Slow pairs take the
// one-point slow path of their point.
// ------------------------------------------------------------------------------------------------
using KahanArr2 = float2[2][10][kMixThreads];  // [sum, compensation][output][thread], lanes = points

__device__ __forceinline__ void kahan2_add(KahanArr2 &k, int tid, const V2 *P) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const float2 s0 = k[0][i][tid], c0 = k[1][i][tid];
    const float2 y = __fadd2_rn(P[i].v, make_float2(-c0.x, -c0.y));
    const float2 t = __fadd2_rn(s0, y);
    const float2 d = __fadd2_rn(t, make_float2(-s0.x, -s0.y));
    k[1][i][tid] = __fadd2_rn(d, make_float2(-y.x, -y.y));
    k[0][i][tid] = t;
  }
}

// the slow pairs of one point (lane 0 = A, 1 = B) of the chunk, into that point's Kahan lane
template <int KIND, int CH>
__device__ __forceinline__ int slow_pairs2(const Launch &L, int f, int base, typename SlowMask<CH>::T bits, int lane,
                                           float drx, float dry, float drz, float dr2, int64_t p, int Sd32,
                                           float rex, const float4 *s_geo, const float4 *s_ax, const float4 *s_mix,
                                           const float4 *const *s_hist, KahanArr2 &kh, int tid, uint8_t &mask) {
  const Sources &s = L.src;
  int err = 0;
  while (bits && !err) {
    const int jj = SlowMask<CH>::first(bits);
    bits &= bits - 1;
    float sp[10] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    uint8_t smask = 0;
    const float4 g = s_geo[jj];
    const float4 ax = s_ax[jj];
    const float4 mx = s_mix[jj];
    const float rx = g.x + drx, ry = g.y + dry, rz = g.z + drz;
    const float rho2 = rx * rx + ry * ry + rz * rz;
    const float rn = rho2 > 0.f ? rho2 * rsqrtf(rho2) : 0.f;
    const int kb = __float_as_int(mx.w);
    const float corr = __fdividef(2.f * (g.x * drx + g.y * dry + g.z * drz) + dr2, rn + g.w);
    const float xc = mx.z - corr;
    double rp64[3];
    point_at(L.pts, p, rp64);
    err = slow_dipole<KIND>(s, base + jj, s_hist[jj], Sd32, kb, xc, rx, ry, rz, rn, ax, mx.x, mx.y, rex, rp64,
                            L.uf[f], L.iLd, L.r_excl, sp, &smask);
    mask |= smask;
    V2 SP[10];
#pragma unroll
    for (int i = 0; i < 10; ++i) SP[i] = lane == 0 ? V2(sp[i], 0.f) : V2(0.f, sp[i]);
    kahan2_add(kh, tid, SP);
  }
  return err;
}

// the two points' sums to the outputs, in SI units
__device__ __forceinline__ void store_two_points(const Launch &L, int f, int tid, const float2 (*sum)[kMixThreads],
                                                 const float2 (*comp)[kMixThreads], bool actA, bool actB, int64_t pA,
                                                 int64_t pB, uint8_t maskA, uint8_t maskB) {
  const float uE = L.unit[0], uB = L.unit[1], uP = L.unit[2], uA = L.unit[3];
  for (int lane = 0; lane < 2; ++lane) {
    if (!(lane == 0 ? actA : actB)) continue;
    const int64_t o = (L.frame0 + f) * L.pts.P + (lane == 0 ? pA : pB);
    float val[10];
#pragma unroll
    for (int i = 0; i < 10; ++i) {
      const float2 sv = sum[i][tid], cv = comp[i][tid];
      val[i] = lane == 0 ? sv.x - cv.x : sv.y - cv.y;
    }
    // streaming stores, as in the one-point kernel
    if (L.out.E) {
      float *e = (float *)L.out.E + 3 * o;
      __stcs(e + 0, uE * val[0]);
      __stcs(e + 1, uE * val[1]);
      __stcs(e + 2, uE * val[2]);
    }
    if (L.out.B) {
      float *b = (float *)L.out.B + 3 * o;
      __stcs(b + 0, uB * val[3]);
      __stcs(b + 1, uB * val[4]);
      __stcs(b + 2, uB * val[5]);
    }
    if (L.out.phi) __stcs((float *)L.out.phi + o, uP * val[6]);
    if (L.out.A) {
      float *a = (float *)L.out.A + 3 * o;
      __stcs(a + 0, uA * val[7]);
      __stcs(a + 1, uA * val[8]);
      __stcs(a + 2, uA * val[9]);
    }
    if (L.out.mask)
      __stcs(reinterpret_cast<unsigned char *>(L.out.mask) + o, (unsigned char)(lane == 0 ? maskA : maskB));
  }
}

template <int KIND, int CH>
__global__ void __launch_bounds__(kMixThreads, 2) fields_mixed2_kernel(const Launch L, int64_t tiles_v) {
  __shared__ float s_anc_hi[3], s_anc_lo[3];  // the tile anchor / (c dt) as float-float
  __shared__ KahanArr2 s_kahan;
  __shared__ float4 s_geo[CH];  // rho_a (x,y,z), |rho_a|
  __shared__ float4 s_ax[CH];   // axis (x,y,z), q/e
  __shared__ float4 s_mix[CH];  // m2/(m1+m2), m1/(m1+m2), fraction and integer part (bits) of the
                                    // retarded sample of the anchor
  __shared__ const float4 *s_hist[CH];

  const int tid = threadIdx.x;
  const int f = blockIdx.y;
  const Sources &s = L.src;
  const int sh = L.tile_shift, cols = 1 << sh, rows = kMixThreads >> sh;
  const int64_t tu = blockIdx.x / tiles_v, tv = blockIdx.x % tiles_v;
  const int64_t iuA = tu * 2 * rows + (tid >> sh), iuB = iuA + rows, iv = tv * cols + (tid & (cols - 1));
  const bool actA = iuA < L.pts.nu && iv < L.pts.nv, actB = iuB < L.pts.nu && iv < L.pts.nv;
  const int64_t pA = iuA * L.pts.nv + iv, pB = iuB * L.pts.nv + iv;
  if (tid == 0) {
    const double iu = (double)(tu * 2 * rows) + 0.5 * (2 * rows - 1), ivc = (double)(tv * cols) + 0.5 * (cols - 1);
    for (int i = 0; i < 3; ++i) {
      const double x = (L.pts.o[i] + iu * L.pts.eu[i] + ivc * L.pts.ev[i]) * L.iLd;
      s_anc_hi[i] = (float)x;
      s_anc_lo[i] = (float)(x - (double)s_anc_hi[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    s_kahan[0][i][tid] = make_float2(0.f, 0.f);
    s_kahan[1][i][tid] = make_float2(0.f, 0.f);
  }
  __syncthreads();
  uint8_t maskA = 0, maskB = 0;
  int err = 0;
  // offsets of the two points from the anchor, from whole grid steps (no float64 on the way)
  const float duA = (float)(tid >> sh) - 0.5f * (float)(2 * rows - 1), duB = duA + (float)rows;
  const float dvv = (float)(tid & (cols - 1)) - 0.5f * (float)(cols - 1);
  const V2 drx(duA * L.eu_L[0] + dvv * L.ev_L[0], duB * L.eu_L[0] + dvv * L.ev_L[0]);
  const V2 dry(duA * L.eu_L[1] + dvv * L.ev_L[1], duB * L.eu_L[1] + dvv * L.ev_L[1]);
  const V2 drz(duA * L.eu_L[2] + dvv * L.ev_L[2], duB * L.eu_L[2] + dvv * L.ev_L[2]);
  const V2 dr2 = fma2(drz, drz, fma2(dry, dry, drx * drx));
  const float rex = (float)(L.r_excl * L.iLd);
  const float rex_fast = rex + 1.5f;
  const int Sd32 = (int)s.Sd;
  const unsigned jlim = Sd32 > 3 ? (unsigned)(Sd32 - 3) : 0u;  // fast segments 1 <= j <= S-3
  const bool any = actA || actB;
  for (int base = 0; base < s.N; base += CH) {
    const int nch = min(CH, s.N - base);
    __syncthreads();
    if (tid < nch) {
      // the anchor's distance to the source and the centre's retarded sample in float-float
      const int j = base + tid;
      const float4 oh = L.srcf[4 * j + 2], ol = L.srcf[4 * j + 3];
      const ff rax = ff_add({s_anc_hi[0], s_anc_lo[0]}, {-oh.x, -ol.x});
      const ff ray = ff_add({s_anc_hi[1], s_anc_lo[1]}, {-oh.y, -ol.y});
      const ff raz = ff_add({s_anc_hi[2], s_anc_lo[2]}, {-oh.z, -ol.z});
      const ff rna = ff_sqrt(ff_add(ff_add(ff_mul(rax, rax), ff_mul(ray, ray)), ff_mul(raz, raz)));
      const ff x = ff_add({L.uf_hi[f], L.uf_lo[f]}, {-rna.hi, -rna.lo});
      float kaf;
      const int kai = Num<float>::floor_int(x.hi, kaf);
      s_geo[tid] = make_float4(rax.hi, ray.hi, raz.hi, rna.hi);
      s_ax[tid] = L.srcf[4 * j];
      const float4 mm = L.srcf[4 * j + 1];
      s_mix[tid] = make_float4(mm.x, mm.y, (x.hi - kaf) + x.lo, __int_as_float(kai));
      s_hist[tid] = L.Hd + (size_t)j * s.Sd;
    }
    __syncthreads();
    if (!any || err) continue;
    V2 P[10];
#pragma unroll
    for (int i = 0; i < 10; ++i) P[i] = V2(0.f);
    typename SlowMask<CH>::T slowA = 0, slowB = 0;
    for (int g16 = 0; g16 < nch; g16 += 16) {
      // groups of sixteen sources summed in float32, the group sums compensated
      const int gend = min(nch, g16 + 16);
      for (int jj = g16; jj < gend; ++jj) {
        const float4 g = s_geo[jj];
        const float4 ax = s_ax[jj];
        const float4 mx = s_mix[jj];
        V2 rx = V2(g.x) + drx, ry = V2(g.y) + dry, rz = V2(g.z) + drz;
        const V2 rho2 = fma2(rz, rz, fma2(ry, ry, rx * rx));
        // rho2 == 0 makes rn NaN, which fails the tests below
        V2 rn = rho2 * V2(rsqrtf(rho2.v.x), rsqrtf(rho2.v.y));
        const V2 num = fma2(V2(2.f), fma2(V2(g.z), drz, fma2(V2(g.y), dry, V2(g.x) * drx)), dr2);
        V2 xc = V2(mx.z) - num * rcp2(rn + V2(g.w));
        const int kb = __float_as_int(mx.w);
        float flA, flB;
        const int jA = kb + Num<float>::floor_int(xc.v.x, flA), jB = kb + Num<float>::floor_int(xc.v.y, flB);
        bool fA = actA && (unsigned)(jA - 1) < jlim && rn.v.x > rex_fast;
        bool fB = actB && (unsigned)(jB - 1) < jlim && rn.v.y > rex_fast;
        if (!(fA && fB)) {
          if (actA && !fA) slowA |= SlowMask<CH>::bit(jj);
          if (actB && !fB) slowB |= SlowMask<CH>::bit(jj);
          if (!fA && !fB) continue;
          // the point off the fast path takes the other point's geometry: finite values whose
          // results are dropped
          if (!fA) {
            rx.v.x = rx.v.y;
            ry.v.x = ry.v.y;
            rz.v.x = rz.v.y;
            rn.v.x = rn.v.y;
            xc.v.x = xc.v.y;
            flA = flB;
          } else {
            rx.v.y = rx.v.x;
            ry.v.y = ry.v.x;
            rz.v.y = rz.v.x;
            rn.v.y = rn.v.x;
            xc.v.y = xc.v.x;
            flB = flA;
          }
        }
        const V2 rp = fma2(rz, V2(ax.z), fma2(ry, V2(ax.y), rx * V2(ax.x)));
        const HistF32 H{s_hist[jj]};
        const int ja = fA ? jA : jB, jb = fB ? jB : jA;
        const float4 hA0 = H.load(ja), hA1 = H.load(ja + 1), hB0 = H.load(jb), hB1 = H.load(jb + 1);
        const V2 x0(hA0.x, hB0.x), v0(hA0.y, hB0.y), a0(hA0.z, hB0.z);
        const V2 dx = V2(hA1.x, hB1.x) - x0, dv = V2(hA1.y, hB1.y) - v0, da = V2(hA1.z, hB1.z) - a0;
        const V2 thc = xc - V2(flA, flB);
        const V2 Xc = fma2(thc, dx, x0);
        Ch2 cp, cm;
        V2 ep, em;
        const V2 tp = charge2_state(mx.x, x0, dx, v0, dv, a0, da, Xc, thc, rn, rp, cp, ep);
        const V2 tm = charge2_state(-mx.y, x0, dx, v0, dv, a0, da, Xc, thc, rn, rp, cm, em);
        // both charges on interior segments (0.5 +- (0.5 + kExtrap)), the series converged
        const float thh = 0.5f + kExtrap;
        fA = fA && fabsf(tp.v.x - 0.5f) <= thh && fabsf(tm.v.x - 0.5f) <= thh && fabsf(ep.v.x) + fabsf(em.v.x) < 1e-2f;
        fB = fB && fabsf(tp.v.y - 0.5f) <= thh && fabsf(tm.v.y - 0.5f) <= thh && fabsf(ep.v.y) + fabsf(em.v.y) < 1e-2f;
        // near fields that cancel in float32 also leave the fast path
        if (fA && rn.v.x < kNearL &&
            dipole_cancellation<float>(rn.v.x, mx.x, mx.y, cp.X.v.x, cp.V.v.x, cp.Ac.v.x, cm.X.v.x, cm.V.v.x,
                                       cm.Ac.v.x) > kCancel)
          fA = false;
        if (fB && rn.v.y < kNearL &&
            dipole_cancellation<float>(rn.v.y, mx.x, mx.y, cp.X.v.y, cp.V.v.y, cp.Ac.v.y, cm.X.v.y, cm.V.v.y,
                                       cm.Ac.v.y) > kCancel)
          fB = false;
        if (actA && !fA) slowA |= SlowMask<CH>::bit(jj);
        if (actB && !fB) slowB |= SlowMask<CH>::bit(jj);
        if (!fA && !fB) continue;
        dipole2_fast<KIND>(rx, ry, rz, rn, ax.x, ax.y, ax.z, rp, mx.x, mx.y, ax.w, cp, cm, fA, fB, P);
      }
      kahan2_add(s_kahan, tid, P);
#pragma unroll
      for (int i = 0; i < 10; ++i) P[i] = V2(0.f);
    }
    // the pairs of this chunk that left the fast path, per point
    const V2 d2 = dr2;
    if (slowA)
      err = slow_pairs2<KIND, CH>(L, f, base, slowA, 0, drx.v.x, dry.v.x, drz.v.x, d2.v.x, pA, Sd32, rex, s_geo, s_ax,
                              s_mix, s_hist, s_kahan, tid, maskA);
    if (slowB && !err)
      err = slow_pairs2<KIND, CH>(L, f, base, slowB, 1, drx.v.y, dry.v.y, drz.v.y, d2.v.y, pB, Sd32, rex, s_geo, s_ax,
                              s_mix, s_hist, s_kahan, tid, maskB);
  }
  if (!any) return;
  if (err) {
    set_status(L.status, err);
    return;
  }
  store_two_points(L, f, tid, s_kahan[0], s_kahan[1], actA, actB, pA, pB, maskA, maskB);
}

// ------------------------------------------------------------------------------------------------
// Plane grids of dipoles that are mostly far (pc_far_f32.cuh): two points per thread as in
// fields_mixed2_kernel and NF frames (1 or 2) of each, every source of the tile either far for the
// whole tile -- its first-order form, with no test left per pair -- or near, and then evaluated as in
// fields_mixed_kernel.  The far form's geometry (1/R, rho.p, p x rho, the delay) is the same in every
// frame, so a pair of frames forms it once; a CTA walks `reps` groups of NF frames, so that its
// anchor and the staged records are formed once for all of them (one chunk of sources) too.
// Warps cover 4 x 8 points, so that their retarded samples lie close together.
//
// Measured on the field grid (64 dipoles, 2048^2 points, 16 frames): 30.6 -> 10.8 ms.  44 warp
// instructions per pair of a warp (221 before); the float32 pipe is busy 58 % of the cycles and the
// issue slots 51 %, with 16 warps per SM: bound by latency, then by that pipe.  One frame at a time and
// the sums over p x g and dr apart took 14.5 ms; the history as separate (X, V) and A rows the same time
// as float4 records, with fewer L1 wavefronts.  Two of the 16 frames (10 and 12.5 fs, where the moments
// cross zero) spend 1.3 ms each on near pairs in float64.
// ------------------------------------------------------------------------------------------------
constexpr int kFarChunk = 64;  // sources staged at a time
constexpr int kFarRows = 32, kFarCols = 16;  // points of a tile, two per thread: rows r and r + 16

// one (tile anchor, source): rho_a and |rho_a| in c dt and the anchor's retarded sample (integer +
// fraction), in float-float
struct AnchorGeo {
  ff x, y, z, n;
  int k;
  float frac;
};
__device__ __forceinline__ AnchorGeo anchor_geo(const Launch &L, const float *hi, const float *lo, int f, int j) {
  AnchorGeo o;
  const float4 oh = L.srcf[4 * j + 2], ol = L.srcf[4 * j + 3];
  o.x = ff_add({hi[0], lo[0]}, {-oh.x, -ol.x});
  o.y = ff_add({hi[1], lo[1]}, {-oh.y, -ol.y});
  o.z = ff_add({hi[2], lo[2]}, {-oh.z, -ol.z});
  o.n = ff_sqrt(ff_add(ff_add(ff_mul(o.x, o.x), ff_mul(o.y, o.y)), ff_mul(o.z, o.z)));
  const ff x = ff_add({L.uf_hi[f], L.uf_lo[f]}, {-o.n.hi, -o.n.lo});
  float kf;
  o.k = Num<float>::floor_int(x.hi, kf);
  o.frac = (x.hi - kf) + x.lo;
  return o;
}
// whether a source is far for every point within L.tile_r of the anchor, all their retarded samples
// (and, a sample further, the charges') on interior segments of the history
__device__ __forceinline__ bool tile_far(const Launch &L, const AnchorGeo &g, int j) {
  const float rt = L.tile_r;  // at most kFarTile
  const int ir = (int)rt + 2;
  // (anchor samples from 2^22 on are beyond the float floor's range)
  return g.n.hi - rt >= L.rfar[j] && g.k >= ir + 2 && g.k < (1 << 22) && g.k + ir <= (int)L.src.Sd - 5;
}

// the anchor (centre) of plane tile (tu, tv), in c dt, as float-float
__device__ __forceinline__ void tile_anchor(const Launch &L, int64_t tu, int64_t tv, float *hi, float *lo) {
  const double iu = (double)(tu * kFarRows) + 0.5 * (kFarRows - 1), iv = (double)(tv * kFarCols) + 0.5 * (kFarCols - 1);
  for (int i = 0; i < 3; ++i) {
    const double x = (L.pts.o[i] + iu * L.pts.eu[i] + iv * L.pts.ev[i]) * L.iLd;
    hi[i] = (float)x;
    lo[i] = (float)(x - (double)hi[i]);
  }
}

// Kahan sums of the NF frames and two points of each thread: [sum, compensation][frame, output][thread],
// lanes = points
template <int NF>
using KahanFar = float2[2][10 * NF][kMixThreads];
// one point's ten outputs (natural order) of frame slot n into its lane
template <int NF>
__device__ __forceinline__ void kahan_lane_add(KahanFar<NF> &k, int tid, int n, int lane, const float *v) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    float *sp = &k[0][10 * n + i][tid].x + lane, *cp = &k[1][10 * n + i][tid].x + lane;
    const float s0 = *sp, y = v[i] - *cp, t = s0 + y;
    *cp = (t - s0) - y;
    *sp = t;
  }
}

// The near sources (bits, the same for the whole CTA) of one of the thread's two points in one frame
// (slot n): the body of fields_mixed_kernel on the far kernel's staged records, in groups of 32.
template <int KIND, int NF>
__device__ __forceinline__ int near_sources_far(const Launch &L, int f, int n, int base, unsigned long long bits,
                                                int lane, float drx, float dry, float drz, float dr2, int64_t p,
                                                const float4 *s_a, const float2 *s_f, KahanFar<NF> &kh, int tid,
                                                uint8_t &mask) {
  const Sources &s = L.src;
  float2 P[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) P[i] = make_float2(0.f, 0.f);
  unsigned long long slow = 0;
  auto flush = [&](const float2(&Q)[5]) {
    const float v[10] = {Q[0].x, Q[0].y, Q[3].x, Q[1].x, Q[1].y, Q[3].y, Q[4].y, Q[2].x, Q[2].y, Q[4].x};
    kahan_lane_add<NF>(kh, tid, n, lane, v);
  };
  auto geometry = [&](int jj, float &rx, float &ry, float &rz, float &rn, float &xc, int &kb) {
    const float4 g = s_a[jj];
    rx = g.x + drx;
    ry = g.y + dry;
    rz = g.z + drz;
    const float rho2 = rx * rx + ry * ry + rz * rz;
    rn = rho2 > 0.f ? rho2 * rsqrtf(rho2) : 0.f;
    xc = s_f[jj].x - __fdividef(2.f * (g.x * drx + g.y * dry + g.z * drz) + dr2, rn + g.w);
    kb = __float_as_int(s_f[jj].y) + kFloorBits;
  };
  int cnt = 0;
  for (unsigned long long m = bits; m; m &= m - 1) {
    const int jj = __ffsll((long long)m) - 1;
    const float4 ax = L.srcf[4 * (base + jj)], mu = L.srcf[4 * (base + jj) + 1];
    float rx, ry, rz, rn, xc;
    int kb;
    geometry(jj, rx, ry, rz, rn, xc, kb);
    const float rp = rx * ax.x + ry * ax.y + rz * ax.z;
    float2 X, V, Ac, dl;
    bool fast = false;
    float fl;
    const int j = kb + Num<float>::floor_int(xc, fl);
    if ((unsigned)(j - 1) < L.jlim && rn > L.rex_fast) {
      const HistF32 H{L.Hd + (size_t)(base + jj) * (size_t)s.Sd};
      float x0, v0, a0, x1, v1, a1;
      H.get_in(j, x0, v0, a0);
      H.get_in(j + 1, x1, v1, a1);
      fast = dip_pair_states_fast(x0, v0, a0, x1, v1, a1, xc - fl, rn, rp, mu.x, mu.y, X, V, Ac, dl);
    }
    if (fast && rn < kNearL &&
        dipole_cancellation<float>(rn, mu.x, mu.y, X.x, V.x, Ac.x, X.y, V.y, Ac.y) > kCancel)
      fast = false;
    if (fast)
      dipole_pair_fast<KIND>(make_float2(rx, ry), rz, rn, make_float2(ax.x, ax.y), ax.z, rp, mu.x, mu.y, ax.w, X, V,
                             Ac, dl, P);
    else
      slow |= 1ull << jj;
    if (++cnt == 32) {
      flush(P);
#pragma unroll
      for (int i = 0; i < 5; ++i) P[i] = make_float2(0.f, 0.f);
      cnt = 0;
    }
  }
  flush(P);
  int err = 0;
  while (slow && !err) {
    const int jj = __ffsll((long long)slow) - 1;
    slow &= slow - 1;
    float sp[10] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    uint8_t smask = 0;
    const float4 ax = L.srcf[4 * (base + jj)], mu = L.srcf[4 * (base + jj) + 1];
    float rx, ry, rz, rn, xc;
    int kb;
    geometry(jj, rx, ry, rz, rn, xc, kb);
    double rp64[3];
    point_at(L.pts, p, rp64);
    err = slow_dipole<KIND>(s, base + jj, L.Hd + (size_t)(base + jj) * (size_t)s.Sd, (int)s.Sd, kb, xc, rx, ry, rz, rn,
                            ax, mu.x, mu.y, L.rex, rp64, L.uf[f], L.iLd, L.r_excl, sp,
                            &smask);
    mask |= smask;
    float2 Q[5];
    pack_outputs(sp, Q);
    flush(Q);
  }
  return err;
}

// FINE: |rho|^2 as |g|^2 and its difference.  That cancels where a point is much nearer to the source than the
// tile's anchor (with steps of 40 nm the field was 1e-5 off there), so it serves tiles that are small against every
// far distance (far_fine: then |g| <= 1.25 |rho|, and it rounds like the other sum); wider ones add up the squares
// of the components.  (That for all: 10.0 -> 10.25 ms on the field grid.)
template <int KIND, int NF, bool FINE>
__global__ void __launch_bounds__(kMixThreads, 2)
    fields_far_kernel(const __grid_constant__ Launch L, int64_t tiles_v, int reps) {
  __shared__ float s_anc_hi[3], s_anc_lo[3];
  extern __shared__ float2 s_dyn[];
  KahanFar<NF> &s_kahan = *reinterpret_cast<KahanFar<NF> *>(s_dyn);
  __shared__ float4 s_a[kFarChunk];      // g = rho_a (x, y, z), |g|
  __shared__ float4 s_b[kFarChunk];      // q/e p (x, y, z), |g|^2
  __shared__ float2 s_f[NF][kFarChunk];  // the anchor's retarded sample: fraction, integer part less kFloorBits
  __shared__ unsigned s_near[2];

  const int tid = threadIdx.x;
  const Sources &s = L.src;
  // warps of 4 x 8 points, so that a warp's retarded samples lie close together
  const int tr = ((tid >> 6) << 2) | ((tid >> 3) & 3), tc = ((tid >> 5) & 1) * 8 + (tid & 7);
  const int64_t tu = blockIdx.x / tiles_v, tv = blockIdx.x % tiles_v;
  const int64_t iuA = tu * kFarRows + tr, iuB = iuA + kFarRows / 2, iv = tv * kFarCols + tc;
  const bool actA = iuA < L.pts.nu && iv < L.pts.nv, actB = iuB < L.pts.nu && iv < L.pts.nv;
  const int64_t pA = iuA * L.pts.nv + iv, pB = iuB * L.pts.nv + iv;
  if (tid == 0) tile_anchor(L, tu, tv, s_anc_hi, s_anc_lo);
  // twice the offsets of the two points from the anchor, from whole grid steps (points past the grid's
  // edge too: they are within the tile like the others, and only not stored)
  const float duA = (float)(2 * tr - (kFarRows - 1)), duB = duA + (float)kFarRows;
  const float dvv = (float)(2 * tc - (kFarCols - 1));
  const V2 Dx(duA * L.eu_L[0] + dvv * L.ev_L[0], duB * L.eu_L[0] + dvv * L.ev_L[0]);
  const V2 Dy(duA * L.eu_L[1] + dvv * L.ev_L[1], duB * L.eu_L[1] + dvv * L.ev_L[1]);
  const V2 Dz(duA * L.eu_L[2] + dvv * L.ev_L[2], duB * L.eu_L[2] + dvv * L.ev_L[2]);
  const V2 half(0.5f);
  const V2 dr2 = V2(0.25f) * fma2(Dz, Dz, fma2(Dy, Dy, Dx * Dx));
  int err = 0;
  for (int rep = 0; rep < reps; ++rep) {
    const int f0 = (blockIdx.y * reps + rep) * NF;
    if (f0 >= L.T) break;
    uint8_t mask[NF][2];
#pragma unroll
    for (int n = 0; n < NF; ++n) mask[n][0] = mask[n][1] = 0;
#pragma unroll
    for (int i = 0; i < 10 * NF; ++i) {
      s_kahan[0][i][tid] = make_float2(0.f, 0.f);
      s_kahan[1][i][tid] = make_float2(0.f, 0.f);
    }
    for (int base = 0; base < s.N; base += kFarChunk) {
      const int nch = min(kFarChunk, s.N - base);
      __syncthreads();
      if (tid < kFarChunk) {
        bool near = false;
        if (tid < nch) {
          const int j = base + tid;
          AnchorGeo g;
#pragma unroll
          for (int n = 0; n < NF; ++n) {
            g = anchor_geo(L, s_anc_hi, s_anc_lo, f0 + n, j);
            near = near || !tile_far(L, g, j);
            s_f[n][tid] = make_float2(g.frac, __int_as_float(g.k - kFloorBits));
          }
          const float4 ax = L.srcf[4 * j];
          const ff gg = ff_mul(g.n, g.n);
          s_a[tid] = make_float4(g.x.hi, g.y.hi, g.z.hi, g.n.hi);
          s_b[tid] = make_float4(ax.w * ax.x, ax.w * ax.y, ax.w * ax.z, gg.hi);
        }
        const unsigned b = __ballot_sync(0xffffffffu, near);
        if ((tid & 31) == 0) s_near[tid >> 5] = b;
      }
      __syncthreads();
      const unsigned long long near_bits = (unsigned long long)s_near[0] | ((unsigned long long)s_near[1] << 32);
      for (int g0 = 0; g0 < nch; g0 += 32) {
        const unsigned skip = s_near[g0 >> 5];
        const int gend = min(nch, g0 + 32);
        V2 S[NF][10];  // E, B, phi, A of each frame
#pragma unroll
        for (int n = 0; n < NF; ++n)
#pragma unroll
          for (int i = 0; i < 10; ++i) S[n][i] = V2(0.f);
        for (int jj = g0; jj < gend; ++jj) {
          if ((skip >> (jj - g0)) & 1u) continue;
          const float4 a = s_a[jj], b = s_b[jj];
          // |rho|^2 - |g|^2 = 2 g.dr + dr^2, 1/|rho|, |rho| - |g| = (|rho|^2 - |g|^2) / (|rho| + |g|)
          const V2 gx(a.x), gy(a.y), gz(a.z), px(b.x), py(b.y), pz(b.z);
          const V2 num = fma2(gx, Dx, fma2(gy, Dy, fma2(gz, Dz, dr2)));
          const V2 rx = fma2(half, Dx, gx), ry = fma2(half, Dy, gy), rz = fma2(half, Dz, gz);
          const V2 rho2 = FINE ? num + V2(b.w) : fma2(rz, rz, fma2(ry, ry, rx * rx));
          const V2 i(rsqrt_fast(rho2.v.x), rsqrt_fast(rho2.v.y));
          const V2 den = fma2(rho2, i, V2(a.w));
          const V2 corr = num * V2(rcp_fast(den.v.x), rcp_fast(den.v.y));
          // each frame's samples first, so that their loads are all in flight
          V2 th[NF];
          float4 h[NF][4];
          const float4 *H = L.Hd + (size_t)(base + jj) * (size_t)s.Sd;
#pragma unroll
          for (int n = 0; n < NF; ++n) {
            const float2 fr = s_f[n][jj];
            const V2 xc = V2(fr.x) - corr;
            const V2 y = floor_bits2(xc);
            th[n] = xc - (y - V2(kFloorMagic));
            const int kb = __float_as_int(fr.y);
            const float4 *hA = H + (kb + __float_as_int(y.v.x)), *hB = H + (kb + __float_as_int(y.v.y));
            h[n][0] = __ldg(hA);
            h[n][1] = __ldg(hA + 1);
            h[n][2] = __ldg(hB);
            h[n][3] = __ldg(hB + 1);
          }
          const V2 rp = fma2(rz, pz, fma2(ry, py, rx * px));
          const V2 cx = fma2(py, rz, -(pz * ry)), cy = fma2(pz, rx, -(px * rz)), cz = fma2(px, ry, -(py * rx));
          const V2 i2 = i * i, rpi2 = rp * i2, m = rpi2 * i, i3_ = V2(3.f) * i;
#pragma unroll
          for (int n = 0; n < NF; ++n) {
            const float4 A0 = h[n][0], A1 = h[n][1], B0 = h[n][2], B1 = h[n][3];
            const float tA = th[n].v.x, tB = th[n].v.y;
            const V2 X(fmaf(tA, A1.x - A0.x, A0.x), fmaf(tB, B1.x - B0.x, B0.x));
            const V2 V(fmaf(tA, A1.y - A0.y, A0.y), fmaf(tB, B1.y - B0.y, B0.y));
            const V2 t1 = fma2(i, X, V);
            V2(&o)[10] = S[n];
            o[6] = fma2(rpi2, t1, o[6]);
            V2 cE, cP, cB;
            if (KIND == PC_COULOMB) {
              cE = m * i3_ * t1;
              cP = -(i2 * t1);
              cB = i2 * i * V;
            } else {
              const V2 Ac(fmaf(tA, A1.z - A0.z, A0.z), fmaf(tB, B1.z - B0.z, B0.z));
              if (KIND == PC_RADIATION) {
                cE = m * Ac;
                cP = -(i * Ac);
                cB = i2 * Ac;
              } else {
                cE = m * fma2(i3_, t1, Ac);
                cP = -(i * fma2(i, t1, Ac));
                cB = i2 * fma2(i, V, Ac);
              }
            }
            const V2 vi = V * i;
            o[0] = fma2(cP, px, fma2(cE, rx, o[0]));
            o[1] = fma2(cP, py, fma2(cE, ry, o[1]));
            o[2] = fma2(cP, pz, fma2(cE, rz, o[2]));
            o[3] = fma2(cB, cx, o[3]);
            o[4] = fma2(cB, cy, o[4]);
            o[5] = fma2(cB, cz, o[5]);
            o[7] = fma2(vi, px, o[7]);
            o[8] = fma2(vi, py, o[8]);
            o[9] = fma2(vi, pz, o[9]);
          }
        }
#pragma unroll
        for (int n = 0; n < NF; ++n)
#pragma unroll
          for (int i = 0; i < 10; ++i) {
            const float2 s0 = s_kahan[0][10 * n + i][tid], c0 = s_kahan[1][10 * n + i][tid];
            const float2 y = __fadd2_rn(S[n][i].v, make_float2(-c0.x, -c0.y));
            const float2 t = __fadd2_rn(s0, y);
            const float2 d = __fadd2_rn(t, make_float2(-s0.x, -s0.y));
            s_kahan[1][10 * n + i][tid] = __fadd2_rn(d, make_float2(-y.x, -y.y));
            s_kahan[0][10 * n + i][tid] = t;
          }
      }
      if (near_bits && !err) {
#pragma unroll 1
        for (int q = 0; q < 2 * NF && !err; ++q) {
          const int lane = q & 1, n = q >> 1;
          if (!(lane ? actB : actA)) continue;
          const float dx = 0.5f * (lane ? Dx.v.y : Dx.v.x), dy = 0.5f * (lane ? Dy.v.y : Dy.v.x),
                      dz = 0.5f * (lane ? Dz.v.y : Dz.v.x), d2 = lane ? dr2.v.y : dr2.v.x;
          uint8_t mk = 0;
          err = near_sources_far<KIND, NF>(L, f0 + n, n, base, near_bits, lane, dx, dy, dz, d2, lane ? pB : pA, s_a,
                                           s_f[n], s_kahan, tid, mk);
#pragma unroll
          for (int t = 0; t < 2 * NF; ++t)
            if (t == q) mask[t >> 1][t & 1] |= mk;
        }
      }
    }
    if (err) {
      if (actA || actB) set_status(L.status, err);
      err = 0;
    }
#pragma unroll
    for (int n = 0; n < NF; ++n)
      store_two_points(L, f0 + n, tid, &s_kahan[0][10 * n], &s_kahan[1][10 * n], actA, actB, pA, pB, mask[n][0],
                       mask[n][1]);
  }
}

// How many (tile, source, frame) triples are near, over up to kFarSample tiles spread over the grid and
// up to four frames: far[0] += near ones, far[1] += all.
constexpr int kFarSample = 512;
__global__ void far_count_kernel(const __grid_constant__ Launch L, int64_t tiles, int64_t tiles_v, int n_tiles,
                                 int n_frames, int *far) {
  const int64_t n = (int64_t)n_tiles * n_frames * L.src.N;
  int near = 0, all = 0;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(t % L.src.N);
    const int64_t r = t / L.src.N;
    const int f = (int)((r % n_frames) * L.T / n_frames);
    const int64_t tile = (r / n_frames) * tiles / n_tiles;
    float hi[3], lo[3];
    tile_anchor(L, tile / tiles_v, tile % tiles_v, hi, lo);
    near += tile_far(L, anchor_geo(L, hi, lo, f, j), j) ? 0 : 1;
    all += 1;
  }
  near = __reduce_add_sync(0xffffffffu, near);
  all = __reduce_add_sync(0xffffffffu, all);
  if ((threadIdx.x & 31) == 0 && all) {
    atomicAdd(far, near);
    atomicAdd(far + 1, all);
  }
}

// per dipole the distance from which it is far, from the largest moments of its history
__global__ void far_limit_kernel(int N, const unsigned *xvmax, const float4 *srcf, float rex_fast, float *rfar) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= N) return;
  const float4 mu = srcf[4 * j + 1];
  const float x = __uint_as_float(xvmax[2 * j]);
  // not below kNearL (nearer pairs are tested for a near field that cancels), nor where a charge may lie within
  // r_excl; nowhere for charges that may be a sample or more from their centre, as the margins kept at the
  // history's ends and about r_excl are for less
  rfar[j] = x <= kSplitSamples ? fmaxf(fmaxf(kNearL, rex_fast), far_limit(x, __uint_as_float(xvmax[2 * j + 1]), mu.x, mu.y))
                               : __int_as_float(0x7f800000);
}

// ================================================================================================
// host side
// ================================================================================================
static bool finite3(const double *v) { return isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]); }

// mixed-path launches: plane tiles with CH sources per shared-memory stage, one or two points per
// thread; point lists with the full stage
template <int CH>
static void launch_mixed_plane(const Launch &L, dim3 grid, int64_t tiles_v, bool two, int kind, cudaStream_t st) {
  if (two) {
    if (kind == PC_TOTAL) fields_mixed2_kernel<PC_TOTAL, CH><<<grid, kMixThreads, 0, st>>>(L, tiles_v);
    else if (kind == PC_COULOMB) fields_mixed2_kernel<PC_COULOMB, CH><<<grid, kMixThreads, 0, st>>>(L, tiles_v);
    else fields_mixed2_kernel<PC_RADIATION, CH><<<grid, kMixThreads, 0, st>>>(L, tiles_v);
  } else {
    if (kind == PC_TOTAL) fields_mixed_kernel<PC_TOTAL, false, CH><<<grid, kMixThreads, 0, st>>>(L, tiles_v);
    else if (kind == PC_COULOMB) fields_mixed_kernel<PC_COULOMB, false, CH><<<grid, kMixThreads, 0, st>>>(L, tiles_v);
    else fields_mixed_kernel<PC_RADIATION, false, CH><<<grid, kMixThreads, 0, st>>>(L, tiles_v);
  }
}
static void launch_mixed_list(const Launch &L, dim3 grid, int kind, cudaStream_t st) {
  if (L.rfar) {
    if (kind == PC_TOTAL) fields_mixed_kernel<PC_TOTAL, true, kChunk, true><<<grid, kMixThreads, 0, st>>>(L, 1);
    else if (kind == PC_COULOMB) fields_mixed_kernel<PC_COULOMB, true, kChunk, true><<<grid, kMixThreads, 0, st>>>(L, 1);
    else fields_mixed_kernel<PC_RADIATION, true, kChunk, true><<<grid, kMixThreads, 0, st>>>(L, 1);
    return;
  }
  if (kind == PC_TOTAL) fields_mixed_kernel<PC_TOTAL, true, kChunk><<<grid, kMixThreads, 0, st>>>(L, 1);
  else if (kind == PC_COULOMB) fields_mixed_kernel<PC_COULOMB, true, kChunk><<<grid, kMixThreads, 0, st>>>(L, 1);
  else fields_mixed_kernel<PC_RADIATION, true, kChunk><<<grid, kMixThreads, 0, st>>>(L, 1);
}

// Frames in twos, a last odd one by itself; each CTA walks as many of them as leave the grid kFarWaves
// waves of two CTAs per SM.
constexpr int kFarWaves = 8;
template <int KIND, int NF, bool FINE>
static cudaError_t launch_far_nf(const pc_ctx *ctx, const Launch &L, int64_t tiles, int64_t tiles_v, cudaStream_t st) {
  const size_t smem = sizeof(KahanFar<NF>);
  auto *fn = fields_far_kernel<KIND, NF, FINE>;
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t groups = (L.T + NF - 1) / NF, want = (int64_t)kFarWaves * 2 * ctx->num_sms;
  const int reps = (int)std::max<int64_t>(1, std::min<int64_t>(groups, tiles * groups / want));
  fn<<<dim3((unsigned)tiles, (unsigned)((groups + reps - 1) / reps)), kMixThreads, smem, st>>>(L, tiles_v, reps);
  return cudaSuccess;
}
// (no source is far within kNearL, far_limit_kernel)
static bool far_fine(const Launch &L) { return 4.f * L.tile_r <= kNearL; }
template <int KIND>
static cudaError_t launch_far_kind(const pc_ctx *ctx, const Launch &L, int64_t tiles, int64_t tiles_v, cudaStream_t st) {
  Launch M = L;
  M.T = L.T & ~1;
  if (M.T) {
    const cudaError_t e = far_fine(L) ? launch_far_nf<KIND, 2, true>(ctx, M, tiles, tiles_v, st)
                                      : launch_far_nf<KIND, 2, false>(ctx, M, tiles, tiles_v, st);
    if (e != cudaSuccess) return e;
  }
  if (L.T & 1) {
    const int k = L.T - 1;
    M.T = 1;
    M.frame0 = L.frame0 + k;
    M.times[0] = L.times[k];
    M.uf[0] = L.uf[k];
    M.uf_hi[0] = L.uf_hi[k];
    M.uf_lo[0] = L.uf_lo[k];
    return far_fine(L) ? launch_far_nf<KIND, 1, true>(ctx, M, tiles, tiles_v, st)
                       : launch_far_nf<KIND, 1, false>(ctx, M, tiles, tiles_v, st);
  }
  return cudaSuccess;
}
static cudaError_t launch_far(const pc_ctx *ctx, const Launch &L, int kind, cudaStream_t st) {
  const int64_t tiles_v = (L.pts.nv + kFarCols - 1) / kFarCols;
  const int64_t tiles = ((L.pts.nu + kFarRows - 1) / kFarRows) * tiles_v;
  if (kind == PC_TOTAL) return launch_far_kind<PC_TOTAL>(ctx, L, tiles, tiles_v, st);
  if (kind == PC_COULOMB) return launch_far_kind<PC_COULOMB>(ctx, L, tiles, tiles_v, st);
  return launch_far_kind<PC_RADIATION>(ctx, L, tiles, tiles_v, st);
}

// Whether a mixed call of T frames may take fields_far_kernel (then far_chosen decides): plane grids
// of dipoles alone.  Asking the device (three launches and a read-back) takes 28 us, which a call whose
// sources turn out near pays for nothing: below kFarWork (point, dipole, frame) triples that is more than a
// few percent of it.  Sets L.tile_r, the largest distance of a tile's point
// from its anchor (c dt).
constexpr double kFarWork = 1e8;  // fields_mixed_kernel: about 700 us, fields_far_kernel 250
// lists: (point, dipole, frame) triples from which the far distances (a memset and a small kernel, 5 us) pay
constexpr double kFarListWork = 2e6;
// the largest tile (radius, c dt): a tile's float32 offsets from its anchor round at 6e-8 of that, which counts
// where a source is nearer than the anchor.  Against the 16 x 16 tiles of fields_mixed_kernel, on points 405 c dt
// from a source beyond a corner: within 1e-6 of the source scale in both up to 1200 (steps of 20 nm at 1 as), from
// 4 (100 nm) to 2 times its error above
constexpr double kFarTile = 1200.0;
static bool far_candidate(Launch &L, bool plane_of_dipoles, int32_t T) {
  if (!plane_of_dipoles || (double)L.src.N * (double)L.pts.P * (double)T < kFarWork) return false;
  double r2 = 0.0;
  for (int sg = -1; sg <= 1; sg += 2) {
    double q = 0.0;
    for (int i = 0; i < 3; ++i) {
      const double d = (0.5 * (kFarRows - 1) * L.pts.eu[i] + sg * 0.5 * (kFarCols - 1) * L.pts.ev[i]) * L.iLd;
      q += d * d;
    }
    r2 = std::max(r2, q);
  }
  const double r = sqrt(r2) * (1.0 + 1e-6) + 1e-3;
  if (!(r <= kFarTile)) return false;
  L.tile_r = (float)r;
  return true;
}

// The far kernel's near pairs run at half the warps of fields_mixed_kernel, its far ones several times
// as fast: it is taken while at most kFarNearMost of the sampled (tile, source, frame) triples are near.
constexpr double kFarNearMost = 0.4;
static pc_status far_chosen(pc_ctx *ctx, const Launch &L, cudaStream_t st, bool *far) {
  const int64_t tiles_v = (L.pts.nv + kFarCols - 1) / kFarCols;
  const int64_t tiles = ((L.pts.nu + kFarRows - 1) / kFarRows) * tiles_v;
  const int n_tiles = (int)std::min<int64_t>(tiles, kFarSample), n_frames = std::min(L.T, 4);
  const int64_t n = (int64_t)n_tiles * n_frames * L.src.N;
  far_count_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 608), 256, 0, st>>>(L, tiles, tiles_v, n_tiles,
                                                                                     n_frames, ctx->d_status + 1);
  if (cudaMemcpyAsync(ctx->h_status, ctx->d_status, 3 * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return PC_ERR_CUDA;
  *far = ctx->h_status[0] == 0 && (double)ctx->h_status[1] <= kFarNearMost * (double)ctx->h_status[2];
  return PC_OK;
}

// Host outputs that are page-locked are mapped into the device's address space (unified
// addressing): the kernels store into them directly and the stores reach host memory while the
// computation runs.  Returns false (leaving `dev` as it was) if any requested output is not
// page-locked host memory the device can address.
static bool mapped_host_outputs(const pc_field_out *out, Outs &dev) {
  const void *h[5] = {out->E, out->B, out->phi, out->A, out->mask};
  void *d[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  for (int k = 0; k < 5; ++k) {
    if (!h[k]) continue;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, h[k]) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (a.type != cudaMemoryTypeHost || !a.devicePointer) return false;
    d[k] = a.devicePointer;
  }
  dev.E = d[0];
  dev.B = d[1];
  dev.phi = d[2];
  dev.A = d[3];
  dev.mask = (uint8_t *)d[4];
  return true;
}

// Other host outputs: frames are computed in chunks into two device buffers that alternate, and
// each chunk is copied to the host on a second stream while the next chunk computes.
struct HostPipe {
  bool on = false;
  int32_t frames = 1;        // frames per chunk
  size_t bytes_frame = 0;    // device bytes of one frame of every requested output
};

static pc_status fields_impl(pc_ctx *ctx, const pc_charges *ch, const pc_dipole_sources *dp, const double *list,
                             const pc_plane *plane, int64_t P, const double *times, int32_t T, int32_t kind,
                             int32_t precision, double r_excl, const pc_field_out *out, void *stream,
                             bool to_host = false) {
  if (!ctx || !out || !times || T < 1 || P < 0) return PC_ERR_ARG;
  if (kind < PC_TOTAL || kind > PC_RADIATION || (precision != PC_F64 && precision != PC_MIXED)) return PC_ERR_ARG;
  if (!(r_excl >= 0.0)) return PC_ERR_ARG;
  const bool has_ch = ch && ch->M > 0, has_dp = dp && dp->N > 0;
  if (!has_ch && !has_dp) return PC_ERR_ARG;
  if ((ch && ch->M < 0) || (dp && dp->N < 0)) return PC_ERR_ARG;
  if (has_ch && (ch->S < 2 || !(ch->dt > 0.0) || !isfinite(ch->t0) || !ch->q || !ch->pos || !ch->vel || !ch->acc))
    return PC_ERR_ARG;
  if (has_dp && (dp->S < 2 || !(dp->dt > 0.0) || !isfinite(dp->t0) || !dp->origin || !dp->axis || !dp->q ||
                 !dp->m1 || !dp->m2 || !dp->d || !dp->d_dot || !dp->d_ddot))
    return PC_ERR_ARG;
  if (P == 0) return PC_OK;
  if (!list && !plane) return PC_ERR_ARG;
  if (list == nullptr && plane && (plane->nu < 0 || plane->nv < 0 || !finite3(plane->origin) ||
                                   !finite3(plane->eu) || !finite3(plane->ev)))
    return PC_ERR_ARG;
  for (int i = 0; i < T; ++i)
    if (!isfinite(times[i])) return PC_ERR_ARG;
  if (P == 0) return PC_OK;
  DeviceGuard g(ctx->device);
  cudaStream_t st = (cudaStream_t)stream;
  pc_status bs = begin_call(ctx, st);
  if (bs != PC_OK) return bs;

  Launch L;
  memset(&L, 0, sizeof(L));
  L.pts.list = list;
  L.pts.P = P;
  if (!list) {
    for (int i = 0; i < 3; ++i) {
      L.pts.o[i] = plane->origin[i];
      L.pts.eu[i] = plane->eu[i];
      L.pts.ev[i] = plane->ev[i];
    }
    L.pts.nu = plane->nu;
    L.pts.nv = plane->nv;
  }
  Sources &s = L.src;
  if (has_ch) {
    s.M = ch->M;
    s.S = ch->S;
    s.t0 = ch->t0;
    s.dt = ch->dt;
    s.q = ch->q;
    s.pos = ch->pos;
    s.vel = ch->vel;
    s.acc = ch->acc;
    s.static_before = ch->static_before;
  }
  if (has_dp) {
    s.N = dp->N;
    s.Sd = dp->S;
    s.t0d = dp->t0;
    s.dtd = dp->dt;
    s.origin = dp->origin;
    s.axis = dp->axis;
    s.qd = dp->q;
    s.m1 = dp->m1;
    s.m2 = dp->m2;
    s.d = dp->d;
    s.dd = dp->d_dot;
    s.ddd = dp->d_ddot;
  }
  L.out.E = out->E;
  L.out.B = out->B;
  L.out.phi = out->phi;
  L.out.A = out->A;
  L.out.mask = out->mask;
  L.r_excl = r_excl;
  L.status = ctx->d_status;
  L.tile_shift = ctx->tile_shift;

  bool far_try = false, far = false;
  L.iLd = has_dp ? 1.0 / (kC * s.dtd) : 0.0;  // 1/(c dt): first guesses without a division
  L.iLc = has_ch ? 1.0 / (kC * s.dt) : 0.0;
  // dipole sample indices are 32-bit integers in both paths (the difference form's solves)
  if (has_dp && s.Sd > (int64_t)1 << 30) return PC_ERR_ARG;
  // the float64 sum of dipoles alone in the split form, where the pairs outweigh writing the float32 mirror
  // (about 0.01 ns a sample against 0.4 ns a pair saved), and there is the memory for it
  const size_t mirror = ((size_t)s.N * (size_t)s.Sd + 4 * (size_t)s.N) * sizeof(float4);
  const bool split = precision == PC_F64 && has_dp && !has_ch && (double)P * (double)T * s.N >= 1e5 &&
                     (double)P * (double)T >= (double)s.Sd / 16.0 && reserve_optional(ctx->hist_f32, mirror, mirror);
  if (split) {
    const size_t nd = (size_t)s.N * s.Sd;
    float4 *Hd = (float4 *)ctx->hist_f32.ptr;
    L.Hd = Hd;
    launch_prep_dipoles(s, Hd, Hd + nd, nullptr, L.status, st);
  } else if (precision == PC_F64 && has_dp) {
    check_axes_kernel<<<(unsigned)((dp->N + 255) / 256), 256, 0, st>>>(dp->axis, dp->N, L.status);
  }
  if (precision == PC_MIXED) {
    // the float32 path indexes samples with 32-bit integers
    if ((has_dp && s.Sd > (int64_t)1 << 30) || (has_ch && s.S > (int64_t)1 << 30)) return PC_ERR_ARG;
    size_t nd = has_dp ? (size_t)s.N * s.Sd : 0, nc = has_ch ? (size_t)s.M * s.S * 3 : 0;
    const size_t ns = has_dp ? 4 * (size_t)s.N : 0, nf = has_dp ? (size_t)s.N : 0;
    if (ctx->hist_f32.reserve((nd + nc + ns + nf) * sizeof(float4)) != cudaSuccess) return PC_ERR_CUDA;
    if (has_ch && ctx->charge_ref.reserve((size_t)s.M * 3 * sizeof(double)) != cudaSuccess) return PC_ERR_CUDA;
    float4 *Hd = (float4 *)ctx->hist_f32.ptr;
    float4 *Hc = Hd + nd;
    L.Hd = Hd;
    L.Hc = Hc;
    L.cref = (const double *)ctx->charge_ref.ptr;
    L.srcf = Hc + nc;
    L.iLd = has_dp ? 1.0 / (kC * s.dtd) : 0.0;
    set_units(L);
    for (int i = 0; i < 3; ++i) {
      L.eu_L[i] = (float)(L.pts.eu[i] * L.iLd);
      L.ev_L[i] = (float)(L.pts.ev[i] * L.iLd);
    }
    far_try = far_candidate(L, !list && has_dp && !has_ch, T);
    const bool far_lim = far_try || (list && has_dp && (double)s.N * (double)P * (double)T >= kFarListWork);
    unsigned *xvmax = (unsigned *)(Hc + nc + ns);
    if (far_lim && cudaMemsetAsync(xvmax, 0, 2 * (size_t)s.N * sizeof(unsigned), st) != cudaSuccess) return PC_ERR_CUDA;
    if (has_dp) {
      launch_prep_dipoles(s, Hd, Hc + nc, far_lim ? xvmax : nullptr, L.status, st);
    }
    if (far_lim) {
      float *rfar = (float *)(xvmax + 2 * (size_t)s.N);
      far_limit_kernel<<<(unsigned)((s.N + 127) / 128), 128, 0, st>>>(s.N, xvmax, L.srcf, L.rex_fast, rfar);
      L.rfar = rfar;
    }
    if (has_ch) launch_prep_charges(s, Hc, (double *)ctx->charge_ref.ptr, st);
  }
  // host outputs: chunk sizes, device buffers, the copy stream and its events
  const size_t elt = precision == PC_F64 ? sizeof(double) : sizeof(float);
  const size_t b_vec = (size_t)P * 3 * elt, b_sca = (size_t)P * elt, b_msk = (size_t)P;
  HostPipe hp;
  char *slot_base[2] = {nullptr, nullptr};
  if (to_host && !out->E && !out->B && !out->A && !out->phi && !out->mask) return end_call(ctx, st);
  if (to_host && !mapped_host_outputs(out, L.out)) {
    hp.on = true;
    hp.bytes_frame = (out->E ? b_vec : 0) + (out->B ? b_vec : 0) + (out->A ? b_vec : 0) + (out->phi ? b_sca : 0) +
                     (out->mask ? b_msk : 0);
    const size_t target = (size_t)256 << 20;  // about 256 MB per chunk
    hp.frames = (int32_t)std::max<size_t>(1, std::min<size_t>((size_t)kMaxT, target / hp.bytes_frame));
    const size_t slot = hp.bytes_frame * hp.frames;
    if (ctx->out_chunks.reserve(2 * slot) != cudaSuccess) return PC_ERR_CUDA;
    slot_base[0] = (char *)ctx->out_chunks.ptr;
    slot_base[1] = slot_base[0] + slot;
    if (!ctx->copy_stream) {
      if (cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking) != cudaSuccess) return PC_ERR_CUDA;
      for (int k = 0; k < 4; ++k)
        if (cudaEventCreateWithFlags(&ctx->pipe_ev[k], cudaEventDisableTiming) != cudaSuccess) return PC_ERR_CUDA;
    }
  }
  const int32_t step = hp.on ? hp.frames : kMaxT;
  int chunk = 0;
  for (int32_t f0 = 0; f0 < T; f0 += step, ++chunk) {
    set_frames(L, times, f0, min(step, T - f0));
    if (far_try && chunk == 0) {
      const pc_status fs = far_chosen(ctx, L, st, &far);
      if (fs != PC_OK) return fs;
    }
    const int sl = chunk & 1;
    if (hp.on) {
      // this chunk's device slot: wait until the copy of the chunk before last has left it
      if (chunk >= 2 && cudaStreamWaitEvent(st, ctx->pipe_ev[2 + sl], 0) != cudaSuccess) return PC_ERR_CUDA;
      char *c = slot_base[sl];
      const size_t nf = (size_t)L.T;
      L.out.E = out->E ? (void *)c : nullptr;
      c += out->E ? nf * b_vec : 0;
      L.out.B = out->B ? (void *)c : nullptr;
      c += out->B ? nf * b_vec : 0;
      L.out.A = out->A ? (void *)c : nullptr;
      c += out->A ? nf * b_vec : 0;
      L.out.phi = out->phi ? (void *)c : nullptr;
      c += out->phi ? nf * b_sca : 0;
      L.out.mask = out->mask ? (uint8_t *)c : nullptr;
      L.frame0 = 0;
    }
    if (precision == PC_F64) {
      dim3 grid((unsigned)((P + 127) / 128), (unsigned)L.T);
      if (split) {
        // (each launch's frames by themselves: in the first ones the field may not have arrived)
        if (chunk > 0 && cudaMemsetAsync(L.status + 1, 0, sizeof(int), st) != cudaSuccess) return PC_ERR_CUDA;
        L.near_min = (int)(kSplitNearMost * kSplitAsk);
        split_count_kernel<<<kSplitAsk / 128, 128, 0, st>>>(L);
        if (kind == PC_TOTAL) fields_split64_kernel<PC_TOTAL><<<grid, 128, 0, st>>>(L);
        else if (kind == PC_COULOMB) fields_split64_kernel<PC_COULOMB><<<grid, 128, 0, st>>>(L);
        else fields_split64_kernel<PC_RADIATION><<<grid, 128, 0, st>>>(L);
      }
      if (kind == PC_TOTAL) fields_f64_kernel<PC_TOTAL><<<grid, 128, 0, st>>>(L);
      else if (kind == PC_COULOMB) fields_f64_kernel<PC_COULOMB><<<grid, 128, 0, st>>>(L);
      else fields_f64_kernel<PC_RADIATION><<<grid, 128, 0, st>>>(L);
    } else {
      // plane grids of dipoles alone may take two points per thread (the tuned choice)
      const bool two = !list && !has_ch && ctx->pts_per_thread == 2;
      int64_t tiles, tiles_v = 1;
      if (list) {
        tiles = (P + kMixThreads - 1) / kMixThreads;
      } else {
        const int64_t cols = (int64_t)1 << L.tile_shift, rows = (two ? 2 : 1) * (kMixThreads / cols);
        int64_t tu = (L.pts.nu + rows - 1) / rows;
        tiles_v = (L.pts.nv + cols - 1) / cols;
        tiles = tu * tiles_v;
      }
      dim3 grid((unsigned)tiles, (unsigned)L.T);
      if (far) {
        if (launch_far(ctx, L, kind, st) != cudaSuccess) return PC_ERR_CUDA;
      } else if (list) launch_mixed_list(L, grid, kind, st);
      else if (ctx->src_chunk == 32) launch_mixed_plane<32>(L, grid, tiles_v, two, kind, st);
      else launch_mixed_plane<kChunk>(L, grid, tiles_v, two, kind, st);
    }
    if (hp.on) {
      // copy the chunk to the host on the copy stream once its kernel is done
      cudaStream_t cs = ctx->copy_stream;
      if (cudaEventRecord(ctx->pipe_ev[sl], st) != cudaSuccess || cudaStreamWaitEvent(cs, ctx->pipe_ev[sl], 0) != cudaSuccess)
        return PC_ERR_CUDA;
      const size_t nf = (size_t)L.T;
      const size_t o = (size_t)f0;
      bool ok = true;
      if (out->E) ok = ok && cudaMemcpyAsync((char *)out->E + o * b_vec, L.out.E, nf * b_vec, cudaMemcpyDeviceToHost, cs) == cudaSuccess;
      if (out->B) ok = ok && cudaMemcpyAsync((char *)out->B + o * b_vec, L.out.B, nf * b_vec, cudaMemcpyDeviceToHost, cs) == cudaSuccess;
      if (out->A) ok = ok && cudaMemcpyAsync((char *)out->A + o * b_vec, L.out.A, nf * b_vec, cudaMemcpyDeviceToHost, cs) == cudaSuccess;
      if (out->phi)
        ok = ok && cudaMemcpyAsync((char *)out->phi + o * b_sca, L.out.phi, nf * b_sca, cudaMemcpyDeviceToHost, cs) == cudaSuccess;
      if (out->mask)
        ok = ok && cudaMemcpyAsync(out->mask + o * b_msk, L.out.mask, nf * b_msk, cudaMemcpyDeviceToHost, cs) == cudaSuccess;
      if (!ok || cudaEventRecord(ctx->pipe_ev[2 + sl], cs) != cudaSuccess) return PC_ERR_CUDA;
    }
  }
  if (hp.on) {
    // the caller's stream ends after the last copy, so the status read-back below covers them all
    if (cudaEventRecord(ctx->pipe_ev[2], ctx->copy_stream) != cudaSuccess ||
        cudaStreamWaitEvent(st, ctx->pipe_ev[2], 0) != cudaSuccess)
      return PC_ERR_CUDA;
  }
  return end_call(ctx, st);
}

}  // namespace pc

extern "C" pc_status pc_fields(pc_ctx *ctx, const pc_charges *ch, const pc_dipole_sources *dp, const double *points,
                               int64_t P, const double *times, int32_t T, int32_t kind, int32_t precision,
                               double r_excl, const pc_field_out *out, void *stream) {
  if (P > 0 && !points) return PC_ERR_ARG;
  return pc::fields_impl(ctx, ch, dp, points, nullptr, P, times, T, kind, precision, r_excl, out, stream);
}

extern "C" pc_status pc_fields_to_host(pc_ctx *ctx, const pc_charges *ch, const pc_dipole_sources *dp,
                                       const double *points, int64_t P, const double *times, int32_t T, int32_t kind,
                                       int32_t precision, double r_excl, const pc_field_out *out_host, void *stream) {
  if (P > 0 && !points) return PC_ERR_ARG;
  return pc::fields_impl(ctx, ch, dp, points, nullptr, P, times, T, kind, precision, r_excl, out_host, stream, true);
}

extern "C" pc_status pc_fields_plane_to_host(pc_ctx *ctx, const pc_charges *ch, const pc_dipole_sources *dp,
                                             const pc_plane *grid, const double *times, int32_t T, int32_t kind,
                                             int32_t precision, double r_excl, const pc_field_out *out_host,
                                             void *stream) {
  if (!grid || grid->nu < 0 || grid->nv < 0) return PC_ERR_ARG;
  return pc::fields_impl(ctx, ch, dp, nullptr, grid, grid->nu * grid->nv, times, T, kind, precision, r_excl,
                         out_host, stream, true);
}

extern "C" pc_status pc_fields_plane(pc_ctx *ctx, const pc_charges *ch, const pc_dipole_sources *dp,
                                     const pc_plane *grid, const double *times, int32_t T, int32_t kind,
                                     int32_t precision, double r_excl, const pc_field_out *out, void *stream) {
  if (!grid || grid->nu < 0 || grid->nv < 0) return PC_ERR_ARG;
  return pc::fields_impl(ctx, ch, dp, nullptr, grid, grid->nu * grid->nv, times, T, kind, precision, r_excl, out,
                         stream);
}

// ================================================================================================
// pc_fields_noalloc: the mixed-precision point-list evaluation with its scratch in a static device
// array instead of a context workspace, for callers that may not allocate device memory.
// ================================================================================================
#include <mutex>

namespace pc {

// float32 history mirrors (dipoles, then point charges), the point-charge reference positions and
// the status word of every pc_fields_noalloc call live here
constexpr size_t kStaticScratchBytes = (size_t)16 << 20;  // 16 MiB
constexpr size_t kStaticHeader = 256;                     // status word, padded to 256 B
static __device__ __align__(256) unsigned char g_noalloc_scratch[kStaticHeader + kStaticScratchBytes];

constexpr int kMaxDevices = 64;
static void *g_noalloc_addr[kMaxDevices];  // the array's device address per device, once resolved
static std::mutex g_noalloc_mu;            // guards g_noalloc_addr

}  // namespace pc

extern "C" pc_status pc_fields_noalloc(const pc_charges *ch, const pc_dipole_sources *dp, const double *points,
                                       int64_t P, const double *times, int32_t T, int32_t kind, double r_excl,
                                       const pc_field_out *out, void *stream) {
  using namespace pc;
  if (!out || !times || T < 1 || P < 0) return PC_ERR_ARG;
  if (kind < PC_TOTAL || kind > PC_RADIATION || !(r_excl >= 0.0)) return PC_ERR_ARG;
  const bool has_ch = ch && ch->M > 0, has_dp = dp && dp->N > 0;
  if (!has_ch && !has_dp) return PC_ERR_ARG;
  if ((ch && ch->M < 0) || (dp && dp->N < 0)) return PC_ERR_ARG;
  if (has_ch && (ch->S < 2 || !(ch->dt > 0.0) || !isfinite(ch->t0) || !ch->q || !ch->pos || !ch->vel || !ch->acc))
    return PC_ERR_ARG;
  if (has_dp && (dp->S < 2 || !(dp->dt > 0.0) || !isfinite(dp->t0) || !dp->origin || !dp->axis || !dp->q ||
                 !dp->m1 || !dp->m2 || !dp->d || !dp->d_dot || !dp->d_ddot))
    return PC_ERR_ARG;
  for (int i = 0; i < T; ++i)
    if (!isfinite(times[i])) return PC_ERR_ARG;
  if (P == 0) return PC_OK;
  if (!points) return PC_ERR_ARG;
  // the scratch must hold the float32 mirrors and the reference positions
  const size_t nd = has_dp ? (size_t)dp->N * (size_t)dp->S : 0;
  const size_t nc = has_ch ? (size_t)ch->M * (size_t)ch->S * 3 : 0;
  const size_t ns = has_dp ? 4 * (size_t)dp->N : 0;
  const size_t need = (nd + nc + ns) * sizeof(float4) + (has_ch ? (size_t)ch->M * 3 * sizeof(double) : 0);
  if (need > kStaticScratchBytes) return PC_ERR_ARG;
  if ((has_dp && dp->S > (int64_t)1 << 30) || (has_ch && ch->S > (int64_t)1 << 30)) return PC_ERR_ARG;

  // once per device, with that device current: the device address of the static scratch.  Only a
  // resolved address is kept, so a failed first lookup is retried by the next call.
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return PC_ERR_CUDA;
  // the points must live on the current device: the kernels run there
  {
    cudaPointerAttributes pa;
    if (cudaPointerGetAttributes(&pa, points) != cudaSuccess) {
      cudaGetLastError();
      return PC_ERR_ARG;
    }
    if (pa.type != cudaMemoryTypeDevice && pa.type != cudaMemoryTypeManaged) return PC_ERR_ARG;
    if (pa.device != dev) return PC_ERR_ARG;
  }
  unsigned char *base = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
      void *a = nullptr;
      if (cudaGetSymbolAddress(&a, g_noalloc_scratch) != cudaSuccess || !a) {
        cudaGetLastError();
        return PC_ERR_CUDA;
      }
      g_noalloc_addr[dev] = a;
    }
    base = (unsigned char *)g_noalloc_addr[dev];
  }
  int *status = (int *)base;
  float4 *Hd = (float4 *)(base + kStaticHeader);
  float4 *Hc = Hd + nd;
  float4 *srcf = Hc + nc;
  double *cref = (double *)(srcf + ns);

  cudaStream_t st = (cudaStream_t)stream;
  cudaGetLastError();
  // the array keeps the previous call's contents: the status word must start at zero
  if (cudaMemsetAsync(status, 0, sizeof(int), st) != cudaSuccess) return PC_ERR_CUDA;

  Launch L;
  memset(&L, 0, sizeof(L));
  L.pts.list = points;
  L.pts.P = P;
  Sources &s = L.src;
  if (has_ch) {
    s.M = ch->M;
    s.S = ch->S;
    s.t0 = ch->t0;
    s.dt = ch->dt;
    s.q = ch->q;
    s.pos = ch->pos;
    s.vel = ch->vel;
    s.acc = ch->acc;
    s.static_before = ch->static_before;
  }
  if (has_dp) {
    s.N = dp->N;
    s.Sd = dp->S;
    s.t0d = dp->t0;
    s.dtd = dp->dt;
    s.origin = dp->origin;
    s.axis = dp->axis;
    s.qd = dp->q;
    s.m1 = dp->m1;
    s.m2 = dp->m2;
    s.d = dp->d;
    s.dd = dp->d_dot;
    s.ddd = dp->d_ddot;
  }
  L.out.E = out->E;
  L.out.B = out->B;
  L.out.phi = out->phi;
  L.out.A = out->A;
  L.out.mask = out->mask;
  L.r_excl = r_excl;
  L.status = status;
  L.Hd = Hd;
  L.Hc = Hc;
  L.cref = cref;
  L.srcf = srcf;
  L.iLd = has_dp ? 1.0 / (kC * s.dtd) : 0.0;
  set_units(L);
  // the mirrors are rewritten in full by every call
  if (has_dp) launch_prep_dipoles(s, Hd, srcf, nullptr, status, st);
  if (has_ch) launch_prep_charges(s, Hc, cref, st);
  const int64_t tiles = (P + kMixThreads - 1) / kMixThreads;
  for (int32_t f0 = 0; f0 < T; f0 += kMaxT) {
    set_frames(L, times, f0, min(kMaxT, T - f0));
    dim3 grid((unsigned)tiles, (unsigned)L.T);
    launch_mixed_list(L, grid, kind, st);
  }
  if (cudaGetLastError() != cudaSuccess) return PC_ERR_CUDA;
  int h = 0;  // pageable host word: the copy completes before cudaMemcpyAsync returns to the stream order
  if (cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return PC_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return PC_ERR_CUDA;
  return (pc_status)h;
}

// ================================================================================================
// Tile-shape autotuning of the mixed plane evaluation: 256-point tiles of 8 x 32, 16 x 16 or 32 x 8
// (rows x columns) trade the spread of the points' delays within a tile (the history gathers'
// locality) against the width of the output rows each warp stores.  Each candidate runs the
// caller's workload once to warm up and once timed; the fastest is kept in the context for the
// plane calls that follow.
// ================================================================================================
extern "C" pc_status pc_set_plane_tiling(pc_ctx *ctx, const pc_plane_tiling *t) {
  if (!ctx || !t) return PC_ERR_ARG;
  const int32_t rows = t->tile_rows, cols = t->tile_cols;
  if (rows < 1 || cols < 1 || cols > pc::kMixThreads || (cols & (cols - 1))) return PC_ERR_ARG;
  const int64_t pts = (int64_t)rows * cols;
  if (pts != pc::kMixThreads && pts != 2 * pc::kMixThreads) return PC_ERR_ARG;
  if (t->sources_per_stage != 32 && t->sources_per_stage != pc::kChunk) return PC_ERR_ARG;
  int sh = 0;
  while ((1 << sh) < cols) ++sh;
  ctx->tile_shift = sh;
  ctx->pts_per_thread = pts == pc::kMixThreads ? 1 : 2;
  ctx->src_chunk = t->sources_per_stage;
  return PC_OK;
}

extern "C" pc_status pc_autotune_plane(pc_ctx *ctx, const pc_charges *ch, const pc_dipole_sources *dp,
                                       const pc_plane *grid, const double *times, int32_t T, int32_t kind,
                                       double r_excl, const pc_field_out *out, pc_plane_tiling *chosen,
                                       void *stream) {
  if (!ctx || !grid || !out) return PC_ERR_ARG;
  pc::DeviceGuard g(ctx->device);
  cudaStream_t st = (cudaStream_t)stream;
  // (points per thread, log2 columns): 8 x 32, 16 x 16, 32 x 8 tiles of one point per thread, and
  // 16 x 32, 32 x 16, 64 x 8 of two (plane grids of dipoles alone); each with 64 and with 32
  // sources per shared-memory stage
  const int cand[6][2] = {{1, 5}, {1, 4}, {1, 3}, {2, 5}, {2, 4}, {2, 3}};
  const int nshape = (ch && ch->M > 0) ? 3 : 6;
  const int chunks[2] = {pc::kChunk, 32};
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return PC_ERR_CUDA;
  float best = 1e30f;
  int best_c = -1;
  pc_status rs = PC_OK;
  for (int c = 0; c < 2 * nshape && rs == PC_OK; ++c) {
    ctx->pts_per_thread = cand[c % nshape][0];
    ctx->tile_shift = cand[c % nshape][1];
    ctx->src_chunk = chunks[c / nshape];
    rs = pc_fields_plane(ctx, ch, dp, grid, times, T, kind, PC_MIXED, r_excl, out, stream);
    if (rs != PC_OK) break;
    cudaEventRecord(e0, st);
    rs = pc_fields_plane(ctx, ch, dp, grid, times, T, kind, PC_MIXED, r_excl, out, stream);
    cudaEventRecord(e1, st);
    if (rs != PC_OK || cudaEventSynchronize(e1) != cudaSuccess) break;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best) {
      best = ms;
      best_c = c;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (best_c < 0) best_c = 1;
  ctx->pts_per_thread = cand[best_c % nshape][0];
  ctx->tile_shift = cand[best_c % nshape][1];
  ctx->src_chunk = chunks[best_c / nshape];
  if (chosen) {
    chosen->tile_rows = ctx->pts_per_thread * (pc::kMixThreads >> ctx->tile_shift);
    chosen->tile_cols = 1 << ctx->tile_shift;
    chosen->sources_per_stage = ctx->src_chunk;
  }
  return rs;
}
