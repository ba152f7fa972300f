// hydro_fp64.cuh -- FP64 arithmetic of the plain method shared by the FP64
// step kernels: the MC-limited PPM reconstruction (Colella & Woodward 1984),
// contact steepening, the indicator's unlimited reconstruction, and the
// Kurganov-Tadmor point flux with its torques (Sec. III-B).  Every operation
// is explicitly rounded or fused, so that the kernels that inline it agree bit
// for bit.  The oracle's bits: the velocities (prims64), the limited slopes, the
// contact test and its weight, the unlimited values.  Not its bits, by fused
// steps or another order of the same operations: the interface values (ppm_sides64,
// ppm_limit64), the sound speed (rsqrt64) and the point flux; dU/dt then differs
// by about 1e-14 of a field's largest, and the tests hold 1e-12.
#pragma once
#include "hydro_common.cuh"

namespace hyd {

// ---- magnitudes as integers -------------------------------------------------
// The bit patterns of non-negative doubles order like their values, so minima
// and comparisons of magnitudes, doublings, halvings and signs run on the
// integer pipes (GB300 issues FP64 at 1/64 of the FP32 rate).  The masks are
// written as integer instructions: as |x| or -x of a double the compiler
// spends an FP64 addition on each.
__device__ __forceinline__ long long mag64(double x) {
  long long r;
  asm("and.b64 %0, %1, 0x7fffffffffffffff;" : "=l"(r) : "l"(__double_as_longlong(x)));
  return r;
}
// The magnitude m with the sign bit of x (of -x: neg).
__device__ __forceinline__ double sign64(long long m, double x, bool neg = false) {
  long long s;
  asm("and.b64 %0, %1, 0x8000000000000000;" : "=l"(s) : "l"(__double_as_longlong(x)));
  return __longlong_as_double(m | (neg ? s ^ (long long)0x8000000000000000ull : s));
}
// x, or -x
__device__ __forceinline__ double flip64(double x, bool neg) {
  long long r;
  asm("xor.b64 %0, %1, %2;" : "=l"(r) : "l"(__double_as_longlong(x)), "l"(neg ? (long long)0x8000000000000000ull : 0ll));
  return __longlong_as_double(r);
}
__device__ __forceinline__ long long min64(long long a, long long b) { return a < b ? a : b; }
// The same on patterns that may reach beyond those of magnitudes (twice_mag of
// an infinity or a NaN).
__device__ __forceinline__ long long umin64(long long a, long long b) {
  return (unsigned long long)a < (unsigned long long)b ? a : b;
}

__device__ __forceinline__ double max_nonneg(double x, double y) {
  const long long a = __double_as_longlong(x), b = __double_as_longlong(y);
  return __longlong_as_double(a > b ? a : b);
}

// 2x for a finite double of magnitude pattern b, exactly: a normal one gains
// one in the exponent field, a subnormal one (exponent field 0) doubles its
// pattern, which carries into the exponent field where 2x is normal.  Of an
// infinity or a NaN: a pattern above every magnitude's, as unsigned.
__device__ __forceinline__ long long twice_mag(long long b) { return b < (1LL << 52) ? b + b : b + (1LL << 52); }

// Half a magnitude as the FP64 product 0.5 x rounds it (to nearest, ties to
// even): with the exponent field at least 2 the result is normal and the field
// drops by one (infinities and NaNs pass unchanged); below that the pattern is
// the significand with its implicit bit (field 1) or without (zero,
// subnormals), and half of it, rounded to even, is the result's pattern (a
// carry into bit 52 is the smallest normal, correctly encoded).
__device__ __forceinline__ long long half_mag(long long mag) {
  if (mag >= (2LL << 52)) return mag < (0x7ffLL << 52) ? mag - (1LL << 52) : mag;
  return (mag >> 1) + (mag & (mag >> 1) & 1LL);
}
__device__ __forceinline__ double half64(double x) { return sign64(half_mag(mag64(x)), x); }

// x <= 0 for a non-NaN double: +0 has the bit pattern 0 and every value with
// the sign bit set (-0 and the negatives) is negative as a signed integer.
__device__ __forceinline__ bool nonpositive(double x) { return __double_as_longlong(x) <= 0LL; }

// Whether two doubles differ in sign bit.
__device__ __forceinline__ bool signs_differ(double x, double y) {
  return (__double2hiint(x) ^ __double2hiint(y)) < 0;
}

// MC-limited slope of sample j from delta_{j-1} = a and delta_j = b:
// 0 if a b <= 0 (the FP64 product), else sgn(b) min(2|a|, 2|b|, |a + b|/2).
// The product is not formed: with both factors nonzero and of one sign it is
// positive unless it underflows, which needs a subnormal factor or exponent
// fields adding up to less than 972 (it is at least 2^-1074 otherwise), and
// only there the FP64 product decides.
// min(2|a|, 2|b|) = 2 min(|a|, |b|) exactly, the minima, the doubling and the
// halving are taken on the bit patterns, and the sign of the result is the
// sign bit of b: the same bits as the FP64 operations, with one FP64
// instruction (a + b) instead of ten.
__device__ __forceinline__ double slope64(double a, double b) {
  const long long ma = mag64(a), mb = mag64(b), lo = min64(ma, mb);
  if (signs_differ(a, b) || lo == 0LL) return 0.0;
  const unsigned ea = (unsigned)(ma >> 52), eb = (unsigned)(mb >> 52);
  if ((ea + eb < 972u || lo < (1LL << 52)) && nonpositive(rmul(a, b))) return 0.0;
  return sign64(umin64(twice_mag(lo), half_mag(mag64(radd(a, b)))), b);
}

// PPM's interface value between two neighbouring samples of a line, taken from
// both sides: with dl = s_b - s_a and the limited slopes Da, Db,
//   u = value - s_a = dl/2 - (Db - Da)/6,  w = s_b - value = dl/2 + (Db - Da)/6.
// The +d side of a cell and the -d side of its +d neighbour share the slopes'
// difference and dl, so a sweep along the line forms both in three FP64
// instructions (exactly mirrored on the reversed line).
__device__ __forceinline__ void ppm_sides64(double dl, double Da, double Db, double& u, double& w) {
  const double t = rsub(Db, Da), hd = half64(dl);
  u = fma(-1.0 / 6.0, t, hd);
  w = fma(1.0 / 6.0, t, hd);
}

// Contact steepening of the interface values p (+d) and m (-d) of the
// centre sample s2 with weight eta > 0, from its neighbours s1, s3 and their
// slopes D0, D2.
__device__ __forceinline__ void ppm_steep64(double s1, double s3, double D0, double D2, double eta, double& p,
                                            double& m) {
  const double keep = rsub(1.0, eta);
  p = radd(rmul(keep, p), rmul(eta, rsub(s3, half64(D2))));
  m = radd(rmul(keep, m), rmul(eta, radd(s1, half64(D0))));
}

// The same on u = p - s2 and w = s2 - m.
__device__ __forceinline__ void ppm_steep_sides64(double s1, double s2, double s3, double D0, double D2, double eta,
                                                  double& u, double& w) {
  double p = radd(s2, u), m = rsub(s2, w);
  ppm_steep64(s1, s3, D0, D2, eta, p, m);
  u = rsub(p, s2);
  w = rsub(s2, m);
}

// The monotonicity fix-ups of PPM on the interface values s2 + u (+d) and
// s2 - w (-d) of the cell value s2, giving p and m: a local extremum flattens
// the cell, an interface value that would put the parabola's extremum inside
// the cell is moved to 3 s2 - 2 (the other one).  An extremum is u w <= 0, and
// with one sign the parabola test (p - m)(s2 - (p + m)/2) against +-(p - m)^2/6
// reads |w| > 2|u| (m moves to s2 - 2u) and |u| > 2|w| (p moves to s2 + 2w):
// magnitudes cut to twice the other's, on the bit patterns, and two FP64
// additions where the tests and moves took twelve.  The limited values are
// continuous where the tests switch.  For the sides of ordinary tiles (WildTile).
__device__ __forceinline__ void ppm_limit64(double s2, double u, double w, double& p, double& m) {
  const long long au = mag64(u), aw = mag64(w);
  const bool flat = signs_differ(u, w);
  const long long lu = flat ? 0LL : min64(au, twice_mag(aw)), lw = flat ? 0LL : min64(aw, twice_mag(au));
  p = radd(s2, sign64(lu, u));
  m = rsub(s2, sign64(lw, w));
}

// A tile with a primitive of 2^508 or above, an infinity or a NaN has its lines
// by PPM's formula itself (ppm_call64): the formula's squares may overflow and its
// comparisons fail, and a non-finite cell then shows in its neighbours' values
// as the formula has it, which ppm_limit64's cuts would hide.  The test is on the
// tile, where the primitives are formed, because a test in every limit costs
// 2 % of the step (512 sub-grids 7.05 -> 7.23 ms a step of three).
struct WildTile {
  unsigned hi = 0;  // the greatest high word of the magnitudes seen
  __device__ __forceinline__ void see(double x) { hi = max(hi, (unsigned)__double2hiint(x) & 0x7fffffffu); }
  __device__ __forceinline__ bool wild() const { return hi >= (1023u + 508u) << 20; }
};
static __device__ __noinline__ double2 ppm_call64(double s0, double s1, double s2, double s3, double s4, double eta) {
  const double sixth = 1.0 / 6.0;
  const double d0 = rsub(s1, s0), d1 = rsub(s2, s1), d2 = rsub(s3, s2), d3 = rsub(s4, s3);
  const double D0 = slope64(d0, d1), D1 = slope64(d1, d2), D2 = slope64(d2, d3);
  double p = rsub(rmul(0.5, radd(s2, s3)), rmul(rsub(D2, D1), sixth));
  double m = rsub(rmul(0.5, radd(s1, s2)), rmul(rsub(D1, D0), sixth));
  if (eta > 0.0) ppm_steep64(s1, s3, D0, D2, eta, p, m);
  if (rmul(rsub(p, s2), rsub(s2, m)) <= 0.0) return make_double2(s2, s2);
  const double dq = rsub(p, m);
  const double lhs = rmul(dq, rsub(s2, rmul(0.5, radd(p, m)))), rhs = rmul(rmul(dq, dq), sixth);
  if (lhs > rhs)
    m = rsub(rmul(3.0, s2), rmul(2.0, p));
  else if (lhs < -rhs)
    p = rsub(rmul(3.0, s2), rmul(2.0, m));
  return make_double2(p, m);
}

// PPM on the five samples s0..s4 of one line: qp = value at the +d end of the
// centre cell, qm = value at its -d end (limited, monotonised).  kSteep: blend
// both interface values with the neighbours' limited extrapolations by the
// contact-steepening weight eta before the fix-ups (Colella & Woodward 1984):
//   qp <- (1-eta) qp + eta (s3 - D2/2),  qm <- (1-eta) qm + eta (s1 + D0/2).
template <bool kSteep = false>
__device__ __forceinline__ void ppm64(double s0, double s1, double s2, double s3, double s4, double& qp,
                                      double& qm, double eta = 0.0) {
  const double d0 = rsub(s1, s0), d1 = rsub(s2, s1), d2 = rsub(s3, s2), d3 = rsub(s4, s3);
  const double D0 = slope64(d0, d1), D1 = slope64(d1, d2), D2 = slope64(d2, d3);
  double u, w, x;
  ppm_sides64(d2, D1, D2, u, x);
  ppm_sides64(d1, D0, D1, x, w);
  if (kSteep && eta > 0.0) ppm_steep_sides64(s1, s2, s3, D0, D2, eta, u, w);
  ppm_limit64(s2, u, w, qp, qm);
}

// All ten primitives along the line through smem cell index c with stride st.
__device__ __forceinline__ void line10(const double* __restrict__ Q, int c, int st, double qp[F], double qm[F]) {
#pragma unroll
  for (int k = 0; k < F; ++k) {
    const double* q = Q + k * S3 + c;
    ppm64(q[-2 * st], q[-st], q[0], q[st], q[2 * st], qp[k], qm[k]);
  }
}

// Contact-steepening weight of one line from the five samples a0..a4 of the
// steepened field (Colella & Woodward 1984 discontinuity detection; their
// constants eps = 0.01, eta1 = 20, eta2 = 0.05): second differences
// d- = (a0 + a2) - 2 a1 and d+ = (a2 + a4) - 2 a3; no weight without an
// inflection (d- d+ > 0) or with a jump a3 - a1 of at most eps min(|a3|, |a1|);
// else eta~ = -(d+ - d-) / (6 (a3 - a1)) and eta = max(0, min(20 (eta~ - 0.05), 1)).
// Every operation explicitly rounded, in the oracle's order, and the minima
// and maxima as the same comparisons: the oracle's bits.
__device__ __forceinline__ double contact_eta64(double a0, double a1, double a2, double a3, double a4) {
  const double d2m = rsub(radd(a0, a2), rmul(2.0, a1));
  const double d2p = rsub(radd(a2, a4), rmul(2.0, a3));
  if (rmul(d2m, d2p) > 0.0) return 0.0;
  const double jump = rsub(a3, a1);
  const double f3 = fabs(a3), f1 = fabs(a1);
  if (fabs(jump) <= rmul(0.01, f3 < f1 ? f3 : f1)) return 0.0;
  const double et = -rsub(d2p, d2m) / rmul(6.0, jump);
  const double v = rmul(20.0, rsub(et, 0.05));
  const double m = v < 1.0 ? v : 1.0;
  return 0.0 > m ? 0.0 : m;
}

// Whether the line through smem cell c with stride st crosses a contact, not
// a shock: Colella & Woodward's gas-dynamics test over the cell's two
// neighbours on the line (K0 = 0.1), multiplied through by the two positive
// minima (no division):
//   gamma K0 |rho+ - rho-| min(p) >= |p+ - p-| min(rho),  p = (gamma-1) eps.
__device__ __forceinline__ bool contact_line64(const double* __restrict__ Q, int c, int st, const StepParams& P) {
  const double r0 = Q[RHO * S3 + c - st], r1 = Q[RHO * S3 + c + st];
  const double p0 = rmul(P.gm1, Q[EGAS * S3 + c - st]), p1 = rmul(P.gm1, Q[EGAS * S3 + c + st]);
  const double drho = fabs(rsub(r1, r0)), dp = fabs(rsub(p1, p0));
  return !(rmul(rmul(rmul(P.gamma, 0.1), drho), p0 < p1 ? p0 : p1) < rmul(dp, r0 < r1 ? r0 : r1));
}

// line10 with contact steepening of the density and species lines where the
// line crosses a contact.
__device__ __forceinline__ void line10c(const double* __restrict__ Q, int c, int st, const StepParams& P,
                                        double qp[F], double qm[F]) {
  const bool contact = contact_line64(Q, c, st, P);
#pragma unroll
  for (int k = 0; k < F; ++k) {
    const double* q = Q + k * S3 + c;
    if (k == RHO || k >= SP0) {
      const double eta = contact ? contact_eta64(q[-2 * st], q[-st], q[0], q[st], q[2 * st]) : 0.0;
      ppm64<true>(q[-2 * st], q[-st], q[0], q[st], q[2 * st], qp[k], qm[k], eta);
    } else {
      ppm64(q[-2 * st], q[-st], q[0], q[st], q[2 * st], qp[k], qm[k]);
    }
  }
}

// Lines of a cell the learned indicator marks smooth: the unlimited 4-point
// interface values q+ = 7/12 (q0 + q1) - 1/12 (q-1 + q2) towards +d (and the
// mirror towards -d) for every field but the spin, which stays limited.
__device__ __forceinline__ void line10u(const double* __restrict__ Q, int c, int st, double qp[F], double qm[F]) {
  const double c7 = 7.0 / 12.0, c1 = 1.0 / 12.0;
#pragma unroll
  for (int k = 0; k < F; ++k) {
    const double* q = Q + k * S3 + c;
    if (k == ZX || k == ZY || k == ZZ) {
      ppm64(q[-2 * st], q[-st], q[0], q[st], q[2 * st], qp[k], qm[k]);
    } else {
      qp[k] = rsub(rmul(c7, radd(q[0], q[st])), rmul(c1, radd(q[-st], q[2 * st])));
      qm[k] = rsub(rmul(c7, radd(q[0], q[-st])), rmul(c1, radd(q[st], q[-2 * st])));
    }
  }
}

// line10, line10c (contact) or line10u (smooth) of a wild tile.
static __device__ __noinline__ void line10_wild(const double* __restrict__ Q, int c, int st, bool smooth, bool contact,
                                                const StepParams& P, double qp[F], double qm[F]) {
  const bool steep = contact && !smooth && contact_line64(Q, c, st, P);
#pragma unroll 1
  for (int k = 0; k < F; ++k) {
    const double* q = Q + k * S3 + c;
    const double s0 = q[-2 * st], s1 = q[-st], s2 = q[0], s3 = q[st], s4 = q[2 * st];
    double2 v;
    if (smooth && !(k == ZX || k == ZY || k == ZZ)) {
      const double c7 = 7.0 / 12.0, c1 = 1.0 / 12.0;
      v.x = rsub(rmul(c7, radd(s2, s3)), rmul(c1, radd(s1, s4)));
      v.y = rsub(rmul(c7, radd(s2, s1)), rmul(c1, radd(s3, s0)));
    } else {
      v = ppm_call64(s0, s1, s2, s3, s4, steep && (k == RHO || k >= SP0) ? contact_eta64(s0, s1, s2, s3, s4) : 0.0);
    }
    qp[k] = v.x;
    qm[k] = v.y;
  }
}

// 1 / sqrt(x) for x > 0: the FP32 value y refined by one step of Halley's
// third-order iteration, y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2 (the FP32
// value's error of 2^-22 leaves 2^-64), five FP64 instructions.  y has 24 bits, so
// y^2 is exact and e is rounded once: at most 0.501 ulp in all (4e6 values; the
// library's function 0.508; with e from a rounded x y it was 0.997, rms 0.331
// against 0.289).  Outside FP32's normal range the library's function, in a call.
static __device__ __noinline__ double rsqrt_call(double x) { return rsqrt(x); }
__device__ __forceinline__ double rsqrt64(double x) {
  if ((unsigned)__double2hiint(x) - 0x38100000u >= 0x0fd00000u) return rsqrt_call(x);
  const double y = widen(rsqrtf(narrow(x)));
  const double e = fma(-x, rmul(y, y), 1.0);
  return fma(rmul(e, y), fma(0.375, e, 0.5), y);
}

// The primitives of one cell from its conserved rho, s, E in u (v and eps in
// place) and the tracer; false for a non-physical cell.  The three quotients
// by rho from one reciprocal, each with Markstein's correction (the remainder
// s - q rho, exact in a fused step, times 1/rho): the division's bits wherever
// the reciprocal, the quotient and the remainder neither overflow nor
// underflow, as with rho in [2^-120, 2^120) and |s| in [2^-900, 2^900) or zero
// (compared over 1.4e7 quotients as near to a rounding boundary as they get).
// Elsewhere, and for rho <= 0, infinities and NaN, the division.  The range is
// wide in s: ahead of a blast the momenta fall by many orders per cell, and with
// those below 2^-520 divided a step of an early 512-sub-grid Sedov blast took
// 7.35 ms in place of 7.19.
static __device__ __noinline__ double div_call(double a, double b) { return a / b; }
__device__ __forceinline__ bool prims64(double u[EGAS + 1], double tau, const StepParams& P) {
  const double rho = u[RHO];
  bool fast = (unsigned)__double2hiint(rho) - ((1023u - 120u) << 20) < 240u << 20;
  bool zero[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const unsigned hs = (unsigned)__double2hiint(u[SX + m]) & 0x7fffffffu;
    zero[m] = (hs | (unsigned)__double2loint(u[SX + m])) == 0u;
    fast &= zero[m] | (hs - ((1023u - 900u) << 20) < 1800u << 20);
  }
  double v[3];
  if (fast) {
    const double ri = __drcp_rn(rho);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double q = rmul(u[SX + m], ri);
      v[m] = zero[m] ? u[SX + m] : fma(fma(-q, rho, u[SX + m]), ri, q);  // a zero keeps its sign
    }
  } else {
#pragma unroll 1
    for (int m = 0; m < 3; ++m) {
      const double q = div_call(u[SX], rho);  // (the three in turn, without an index)
      u[SX] = u[SY];
      u[SY] = u[SZ];
      u[SZ] = q;
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) v[m] = u[SX + m];
  }
  const double E = u[EGAS];
  const double ek = rmul(half64(rho), radd(radd(rmul(v[0], v[0]), rmul(v[1], v[1])), rmul(v[2], v[2])));
  const double eE = rsub(E, ek);
  const double eps = (eE > rmul(P.eta1, E)) ? eE : pow(tau, P.gamma);
#pragma unroll
  for (int m = 0; m < 3; ++m) u[SX + m] = v[m];
  u[EGAS] = eps;
  return (rho > 0.0) && (eps > 0.0);
}

// What the flux needs of a reconstructed state besides its fields: the
// pressure p, the energy E = eps + rho |v|^2 / 2 and the sound speed.
// c = sqrt(gamma p / rho) = gamma p / sqrt(gamma p rho): one reciprocal square
// root instead of a division and a square root (a few ulps from the correctly
// rounded value); c = 0 where p <= 0 (a non-physical state).  A state is the
// end of one line and serves up to three faces, so a kernel that keeps line
// ends keeps these with them.
struct End64 {
  double p, E, c;
};
__device__ __forceinline__ End64 end64(double rho, double vx, double vy, double vz, double eps, const StepParams& P) {
  End64 e;
  e.p = rmul(P.gm1, eps);
  e.E = fma(half64(rho), fma(vz, vz, fma(vy, vy, rmul(vx, vx))), eps);
  const double gp = rmul(P.gamma, e.p);
  e.c = (__double_as_longlong(gp) <= 0LL) ? 0.0 : rmul(gp, rsqrt64(rmul(gp, rho)));
  return e;
}

// d x for an integer d in {-1, 0, 1}, by sign selection.
__device__ __forceinline__ double signed_pick(int d, double x) { return d == 0 ? 0.0 : flip64(x, d < 0); }

// Spin feedback at a cell's point x_c + (h/2) d: the velocity there of the
// cell's rigid rotation omega = z / I, I = rho h^2 / 6 (a uniform cube about
// its centre), omega x (h/2) d = (3 / (rho h)) z x d, for the cell's
// primitives rho, eps and z and k3h = 3 / h, gg1 = gamma (gamma - 1).  The
// rotation is subsonic: where its corner speed sqrt(3) (3 / (rho h)) |z|
// exceeds the sound speed c = sqrt(gg1 eps / rho), the factor 3 / (rho h) is
// replaced by the one that reaches c there, c / (sqrt(3) |z|) (none for
// eps <= 0).  The test compares rho c^2 with rho times the corner speed
// squared, so that only a capped cell divides again.  z x d by sign
// selection (d in {-1, 0, 1}^3), so the increment at x_c - (h/2) d is
// exactly the negative.  Explicitly rounded (no contraction), so that every
// kernel that adds it gets the same bits.
__device__ __forceinline__ void spin_dv64(double rho, double eps, double zx, double zy, double zz, double k3h,
                                          double gg1, int dx, int dy, int dz, double dv[3]) {
  double k = k3h / rho;
  const double z2 = radd(radd(rmul(zx, zx), rmul(zy, zy)), rmul(zz, zz));
  const double rc2 = rmul(gg1, eps);
  if (rc2 < rmul(rmul(3.0, rmul(k3h, k)), z2)) k = rc2 > 0.0 ? sqrt(rc2 / rmul(rmul(3.0, rho), z2)) : 0.0;
  dv[0] = rmul(k, rsub(signed_pick(dz, zy), signed_pick(dy, zz)));
  dv[1] = rmul(k, rsub(signed_pick(dx, zz), signed_pick(dz, zx)));
  dv[2] = rmul(k, rsub(signed_pick(dy, zx), signed_pick(dx, zy)));
}

// Kurganov-Tadmor flux at one point with half its Simpson weight hw = w/2,
// accumulated per field into the face sum:
//   w F_q = hw (F_L + F_R) - hw a_q (U_R - U_L),  F = U u_n (+ p e_a, + p v_a)
//         = U_L A + (U_R - U_L) B (+ the pressure terms),
//   A = hw (u_nL + u_nR),  B = hw u_nR - hw a_q:
// two fused steps and one difference per field, and a uniform state, whose
// differences are zero, still has no dissipation to cancel.  rho u_n, v (three
// components each): the reconstructed fields; eL, eR: end64 of the two sides;
// un = v_a + wn, wn = omega y_q along x, -omega x_q along y (rotating frame,
// u = v - omega z_hat x x_q).  The point lies at x_L + (h/2) d from the left
// cell's centre, d = e_a + u1 e_b + u2 e_c (b < c the transverse axes); M
// accumulates the moments of the momentum flux g = w F_q that the face's
// torques need besides the face sum: u1 g_a, u1 g_c, u2 g_a, u2 g_b.  Every
// operation is explicitly rounded or fused, so that the kernels that inline
// it agree bit for bit.
__device__ __forceinline__ void point64(const double qL[F], const End64& eL, const double qR[F], const End64& eR,
                                        int a, double om, double r, double hw, int u1, int u2, double fsum[F],
                                        double M[4], double& amax) {
  const double vaL = (a == 0) ? qL[SX] : (a == 1) ? qL[SY] : qL[SZ];
  const double vaR = (a == 0) ? qR[SX] : (a == 1) ? qR[SY] : qR[SZ];
  const double unL = fma(om, r, vaL), unR = fma(om, r, vaR);
  const double aq = max_nonneg(radd(fabs(unL), eL.c), radd(fabs(unR), eR.c));  // signal speeds are >= 0
  amax = max_nonneg(amax, aq);
  const double A = rmul(hw, radd(unL, unR)), B = rmul(hw, rsub(unR, aq));
  const double hpp = rmul(hw, radd(eL.p, eR.p));
  double g[3];
#pragma unroll
  for (int k = 0; k < F; ++k) {
    if (k >= SX && k <= SZ) {
      const double uL = rmul(qL[RHO], qL[k]), uR = rmul(qR[RHO], qR[k]);
      g[k - SX] = fma(uL, A, fma(rsub(uR, uL), B, (a == k - SX) ? hpp : 0.0));
      fsum[k] = radd(fsum[k], g[k - SX]);
    } else if (k == EGAS) {
      const double pv = fma(eL.p, vaL, rmul(eR.p, vaR));
      fsum[k] = fma(eL.E, A, fma(rsub(eR.E, eL.E), B, fma(hw, pv, fsum[k])));
    } else {
      fsum[k] = fma(qL[k], A, fma(rsub(qR[k], qL[k]), B, fsum[k]));
    }
  }
  const double ga = a == 0 ? g[0] : a == 1 ? g[1] : g[2];
  if (u1 != 0) {
    M[0] = radd(M[0], flip64(ga, u1 < 0));
    M[1] = radd(M[1], flip64(a == 2 ? g[1] : g[2], u1 < 0));
  }
  if (u2 != 0) {
    M[2] = radd(M[2], flip64(ga, u2 < 0));
    M[3] = radd(M[3], flip64(a == 0 ? g[1] : g[0], u2 < 0));
  }
}

// The rotating frame's part of u_n at a point: un = v_a + om r, om = omega
// and r = y_q along x, om = -omega and r = x_q along y, none along z.
__device__ __forceinline__ double frame_om(int a, const StepParams& P) {
  return (a == 0) ? P.omega : (a == 1) ? -P.omega : 0.0;
}

// The face's torques about the left and right cell centres from point64's
// moments M and face sum fsum: tl = (h/2) T with T = sum of d x g, and
// tr = (h/2) (T - 2 e_a x m) about the centre at x_L + h e_a, m the momentum
// part of fsum.  With d = e_a + u1 e_b + u2 e_c and m the sum of g, T has
// along a the component +-(M[1] - M[3]), along b and c differences of M[2],
// M[0] and m.
__device__ __forceinline__ void face_torques64(const double M[4], const double fsum[F], int a, double half_h,
                                               double tl[3], double tr[3]) {
  const double mx = fsum[SX], my = fsum[SY], mz = fsum[SZ];
  double T[3];
  if (a == 0) {  // d = (1, u1, u2)
    T[0] = rsub(M[1], M[3]);
    T[1] = rsub(M[2], mz);
    T[2] = rsub(my, M[0]);
  } else if (a == 1) {  // d = (u1, 1, u2)
    T[0] = rsub(mz, M[2]);
    T[1] = rsub(M[3], M[1]);
    T[2] = rsub(M[0], mx);
  } else {  // d = (u1, u2, 1)
    T[0] = rsub(M[2], my);
    T[1] = rsub(mx, M[0]);
    T[2] = rsub(M[1], M[3]);
  }
  // e_a x m
  const double ex = (a == 0) ? 0.0 : (a == 1) ? mz : flip64(my, true);
  const double ey = (a == 0) ? flip64(mz, true) : (a == 1) ? 0.0 : mx;
  const double ez = (a == 0) ? my : (a == 1) ? flip64(mx, true) : 0.0;
  tl[0] = rmul(half_h, T[0]);
  tl[1] = rmul(half_h, T[1]);
  tl[2] = rmul(half_h, T[2]);
  tr[0] = rmul(half_h, fma(-2.0, ex, T[0]));
  tr[1] = rmul(half_h, fma(-2.0, ey, T[1]));
  tr[2] = rmul(half_h, fma(-2.0, ez, T[2]));
}

}  // namespace hyd
