// particles64.cu -- the plain FP64 particle path: one thread per particle,
// gather straight from the FP64 field arrays, push and move in the particle's
// local orthonormal frame, Villasenor-Buneman deposit with FP64 global
// atomics.  Also: stable removal of deleted particles and the particle
// reductions used by the diagnostics.
#include "pic_internal.h"

namespace pic {

namespace {

// ---- FP64 arithmetic of the particle step -------------------------------------
// This part issues FP64 at 2 lanes a clock and SM: a warp's FP64 operation
// takes the pipe as long as 64 FP32 ones, so the kernel's cost is the number
// of FP64 operations (conversions, compares and floor among them).  The step
// therefore works in the particle's local frame on small arguments: positions
// as cell + offset, r and theta from node tables turned by short series, the
// moves as increments (log1p, arcsine series), and reciprocals and square
// roots as one third-order step (Householder; Halley) from the hardware's
// approximations; compares are made on the integer halves of a double.
// Measured on 512 x 512, 2e7 particles: 634 FP64 instructions a particle and
// 22.6 ms a step with exp, log, sincos, atan2, hypot and divisions in global
// coordinates; 300 and 11.2 ms so; 285 and 10.7 ms with FP32 last terms of the series
// and one code for the last path segment of crossing and other lanes (the FP64
// pipe at its 86 % limit throughout).
// The local form is also the more exact one: against 50 digits, a move's
// position error falls from 1.2e-14 to 3.5e-15 cell, and next to a pole (1e-6
// to 1 cell from it) the momenta's from 1e-10 to 2e-15.

__device__ __forceinline__ int hi_word(double x) { return __double2hiint(x); }
__device__ __forceinline__ bool finite64(double x) { return (hi_word(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool is_zero64(double x) { return (__double_as_longlong(x) << 1) == 0; }

// 1 / x: the approximation's relative error e < 2^-19 becomes e^3
__device__ __forceinline__ double recip64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  const double r = fma(y, fma(e, e, e), y);
  // normal x with a normal reciprocal; otherwise the approximation's 0, infinity or NaN
  return (unsigned)(hi_word(x) & 0x7fffffff) - 0x00100000u < 0x7fc00000u ? r : y;
}

// 1 / sqrt(x): y (1 + e / 2 + 3 e^2 / 8) with e = 1 - x y^2
__device__ __forceinline__ double rsqrt64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  const double r = fma(y * e, fma(0.375, e, 0.5), y);
  return (unsigned)hi_word(x) - 0x00100000u < 0x7fe00000u ? r : y;  // normal, positive, finite x
}

// sqrt(x) = g + d y (1 / 2 + 3 d y^2 / 8), g = x y with y the approximation of
// 1 / sqrt(x), d = x - g^2 exact: the rounding of g does not stay in the result
__device__ __forceinline__ double sqrt64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = x * y, t = fma(-g, g, x) * y;
  const double r = fma(t, fma(0.375, t * y, 0.5), g);
  return (unsigned)hi_word(x) - 0x00100000u < 0x7fe00000u ? r : sqrt(x);
}

// The last terms of a series, too small for their 24 bits to show in a double,
// are summed in FP32; the arguments are converted with integer operations
// (toward zero; a subnormal float becomes 0), as a conversion instruction
// costs as much of the FP64 pipe as a term.
__device__ __forceinline__ float low32(double x) {  // |x| < 2
  const int e = (hi_word(x) & 0x7fffffff) - 0x38000000;
  const float f = __uint_as_float(__funnelshift_l((unsigned)__double2loint(x), (unsigned)(e < 0x00100000 ? 0 : e), 3));
  return hi_word(x) < 0 ? -f : f;
}
__device__ __forceinline__ double high64(float x) {  // normal, positive x
  const unsigned b = __float_as_uint(x);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// arcsine for |t| < 1/8: t sum (2k)! / (4^k k!^2 (2k+1)) t^2k, truncated below
// 2^-60 relative; FP32 from t^10 on (2^-35 of t)
__device__ __forceinline__ double asin_series64(double t) {
  const double z = t * t;
  const float y = low32(z);
  float q = 6435.0f / 557056.0f;
  q = fmaf(q, y, 143.0f / 10240.0f);
  q = fmaf(q, y, 231.0f / 13312.0f);
  q = fmaf(q, y, 63.0f / 2816.0f);
  double p = high64(q);
  p = fma(p, z, 35.0 / 1152.0);
  p = fma(p, z, 5.0 / 112.0);
  p = fma(p, z, 3.0 / 40.0);
  p = fma(p, z, 1.0 / 6.0);
  return fma(t * z, p, t);
}

// (1/2) log1p(s) = atanh(t), t = s / (2 + s), for |s| < 1/16, truncated below
// 2^-60; FP32 from t^8 on (2^-43 of t)
__device__ __forceinline__ double half_log1p64(double s) {
  if (!((hi_word(s) & 0x7fffffff) < 0x3fb00000)) return 0.5 * log1p(s);
  const double t = s * recip64(2.0 + s), z = t * t;
  const float y = low32(z);
  double p = high64(fmaf(1.0f / 11.0f, y, 1.0f / 9.0f));
  p = fma(p, z, 1.0 / 7.0);
  p = fma(p, z, 1.0 / 5.0);
  p = fma(p, z, 1.0 / 3.0);
  return fma(t * z, p, t);
}

// exp(x) for |x| <= 1/32, truncated below 2^-60; FP32 from x^6 on (2^-39)
__device__ __forceinline__ double exp_series64(double x) {
  const float y = low32(x);
  double p = high64(fmaf(fmaf(1.0f / 40320.0f, y, 1.0f / 5040.0f), y, 1.0f / 720.0f));
  p = fma(p, x, 1.0 / 120.0);
  p = fma(p, x, 1.0 / 24.0);
  p = fma(p, x, 1.0 / 6.0);
  p = fma(p, x, 0.5);
  return fma(fma(p, x, 1.0), x, 1.0);
}

// sin and cos of (n, b) = node angle + b, |b| <= pi / 64; FP32 for the last two
// terms of each series (2^-38 of sin b; 2^-35)
__device__ __forceinline__ void turn64(double2 n, double b, double &st, double &ct) {
  const double z = b * b;
  const float y = low32(z);
  double p = high64(fmaf(-1.0f / 362880.0f, y, 1.0f / 5040.0f)), q = high64(fmaf(-1.0f / 40320.0f, y, 1.0f / 720.0f));
  p = fma(-p, z, 1.0 / 120.0);
  p = fma(p, z, -1.0 / 6.0);
  const double sb = fma(b * z, p, b);
  q = fma(-q, z, 1.0 / 24.0);
  q = fma(q, z, -0.5);
  const double cb1 = q * z;  // cos b - 1
  st = fma(n.y, sb, fma(n.x, cb1, n.x));
  ct = fma(-n.x, sb, fma(n.y, cb1, n.y));
}

// floor of a grid coordinate |x| < 2^31 as an integer and as a double: two
// additions with 1.5 2^52, rounded down
__device__ __forceinline__ int floor64(double x, double &f) {
  const double m = __dadd_rd(x, 6755399441055744.0);
  f = __dsub_rn(m, 6755399441055744.0);
  return __double2loint(m);
}

// bilinear interpolation of a component at array offset o, offsets (a, b):
// three linear interpolations
__device__ __forceinline__ double lerp64(const double *__restrict__ p, size_t o, int LD, double a, double b) {
  const double f00 = p[o], f10 = p[o + LD], f01 = p[o + 1], f11 = p[o + LD + 1];
  const double v0 = fma(a, f10 - f00, f00), v1 = fma(a, f11 - f01, f01);
  return fma(b, v1 - v0, v0);
}

// the analytic field (vacuum_field) from 1 / r, added to E and B
__device__ __forceinline__ void add_vacuum64(const Grid &G, double r0W, double ir, double st, double ct, bool inside,
                                             double E[3], double B[3]) {
  if (G.vacuum == PIC_VAC_NONE) return;
  const double b0 = G.b0, r0 = G.r_min, q = r0 * ir, bq2 = b0 * q * q;
  switch (G.vacuum) {
    case PIC_VAC_MONOPOLE:
      B[0] += bq2;
      break;
    case PIC_VAC_MONOPOLE_ROTATOR: {
      B[0] += bq2;
      if (!inside) {
        const double a = bq2 * (q * r0W);
        E[0] = fma(-2.0 * a, ct, E[0]);
        E[1] = fma(-a, st, E[1]);
      } else {
        E[1] = fma(-b0 * q * r0W, st, E[1]);
      }
      break;
    }
    case PIC_VAC_UNIFORM_BZ:
      B[0] = fma(b0, ct, B[0]);
      B[1] = fma(-b0, st, B[1]);
      break;
    case PIC_VAC_DIPOLE_COROT:
    case PIC_VAC_DIPOLE_ROTATOR: {
      const double m3 = bq2 * q, mW = b0 * r0W * (q * q);  // mu / r^3, mu W / r^2
      B[0] = fma(2.0 * m3, ct, B[0]);
      B[1] = fma(m3, st, B[1]);
      if (inside || G.vacuum == PIC_VAC_DIPOLE_COROT) {
        E[0] = fma(mW * st, st, E[0]);
        E[1] = fma(-2.0 * mW * st, ct, E[1]);
      } else {
        const double a = mW * (q * q);  // Omega mu r0^2 / r^4
        E[0] = fma(-a, fma(3.0 * ct, ct, -1.0), E[0]);
        E[1] = fma(-2.0 * a * st, ct, E[1]);
      }
      break;
    }
    default:
      break;
  }
}

// Vay (2008) and Boris (1970) pushes, Sec. 2, in a right-handed orthonormal
// basis; qmdt = (q / m) dt, u = gamma v updated in place
__device__ __forceinline__ void vay64(double qmdt, const double E[3], const double B[3], double u[3]) {
  const double h = 0.5 * qmdt;
  const double ig0 = rsqrt64(fma(u[0], u[0], fma(u[1], u[1], fma(u[2], u[2], 1.0))));
  const double tau0 = h * B[0], tau1 = h * B[1], tau2 = h * B[2];
  const double v0 = u[0] * ig0, v1 = u[1] * ig0, v2 = u[2] * ig0;
  const double a0 = fma(v1, tau2, fma(-v2, tau1, fma(qmdt, E[0], u[0])));
  const double a1 = fma(v2, tau0, fma(-v0, tau2, fma(qmdt, E[1], u[1])));
  const double a2 = fma(v0, tau1, fma(-v1, tau0, fma(qmdt, E[2], u[2])));
  const double t2 = fma(tau0, tau0, fma(tau1, tau1, tau2 * tau2));
  const double us = fma(a0, tau0, fma(a1, tau1, a2 * tau2));
  const double sg = fma(a0, a0, fma(a1, a1, fma(a2, a2, 1.0))) - t2;
  const double root = sqrt64(fma(sg, sg, 4.0 * fma(us, us, t2)));
  const double ig = rsqrt64(0.5 * (sg + root));
  const double w0 = tau0 * ig, w1 = tau1 * ig, w2 = tau2 * ig;
  const double sc = recip64(fma(t2 * ig, ig, 1.0)), at = us * ig;
  u[0] = sc * fma(a1, w2, fma(-a2, w1, fma(at, w0, a0)));
  u[1] = sc * fma(a2, w0, fma(-a0, w2, fma(at, w1, a1)));
  u[2] = sc * fma(a0, w1, fma(-a1, w0, fma(at, w2, a2)));
}

__device__ __forceinline__ void boris64(double qmdt, const double E[3], const double B[3], double u[3]) {
  const double h = 0.5 * qmdt;
  const double m0 = fma(h, E[0], u[0]), m1 = fma(h, E[1], u[1]), m2 = fma(h, E[2], u[2]);
  const double ig = h * rsqrt64(fma(m0, m0, fma(m1, m1, fma(m2, m2, 1.0))));
  const double t0 = ig * B[0], t1 = ig * B[1], t2 = ig * B[2];
  const double f = 2.0 * recip64(fma(t0, t0, fma(t1, t1, fma(t2, t2, 1.0))));
  const double p0 = fma(m1, t2, fma(-m2, t1, m0)), p1 = fma(m2, t0, fma(-m0, t2, m1)),
               p2 = fma(m0, t1, fma(-m1, t0, m2));
  const double s0 = f * t0, s1 = f * t1, s2 = f * t2;
  u[0] = fma(h, E[0], fma(p1, s2, fma(-p2, s1, m0)));
  u[1] = fma(h, E[1], fma(p2, s0, fma(-p0, s2, m1)));
  u[2] = fma(h, E[2], fma(p0, s1, fma(-p1, s0, m2)));
}

// charge crossing the four dual faces around the cell at array offset o for a
// straight path p -> p + d inside it (local coordinates, Villasenor-Buneman,
// Eq. Jcons)
__device__ __forceinline__ void vb_seg64(double *Fr, double *Ft, size_t o, int LD, double qw, double p1, double p2,
                                         double d1, double d2) {
  const double A = qw * d1, B = qw * d2;
  const double Am = A * fma(0.5, d2, p2), Bm = B * fma(0.5, d1, p1);
  atomicAdd(Fr + o, A - Am);
  atomicAdd(Fr + o + 1, Am);
  atomicAdd(Ft + o, B - Bm);
  atomicAdd(Ft + o + LD, Bm);
}

__device__ __forceinline__ double clamp01(double v) {
  return hi_word(v) < 0 ? 0.0 : (hi_word(v) >= 0x3ff00000 ? 1.0 : v);
}

struct Fields64 { const double *f[6]; };
struct Flux64 { double *Fr, *Ft, *Fp; };
struct Args64 {
  Grid G;
  double r0W, qmdt;        // r_min Omega at the step's start; (q / m) dt
  double inv_dxi, k_th;    // 1 / dxi; nth / pi (linear theta) or nth / 2 (equal area)
  double pi_nth, inv_nth, nth;
  bool series_r, series_t; // dxi <= 1/16; nth >= 32: the tables' short series
  const double2 *th_n;     // (sin, cos) of the node angles per padded column (linear theta)
};

__global__ void __launch_bounds__(256) k_particles64(const __grid_constant__ Args64 A, Parts64 P, int64_t n,
                                                     Fields64 F, Flux64 D, int *err, long long *cnt, AxisTies ties) {
  follow();
  const Grid &G = A.G;
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double qw = P.qw[k];
  if (is_zero64(qw)) return;  // free slot
  const double x1 = P.x1[k], x2 = P.x2[k];
  double u[3] = {P.ur[k], P.ut[k], P.up[k]};
  const bool ea = G.th_map == PIC_TH_EQUAL_AREA, lg = G.r_map == PIC_R_LOG;
  // cell and offsets (particles hold whole-grid coordinates, arrays local rows)
  double fi, fj;
  const int ci = floor64(x1, fi);
  int cj = floor64(x2, fj);
  const double dx = x1 - fi;
  double dy = x2 - fj;
  if (cj > G.nth - 1) { cj = G.nth - 1; dy = 1.0; }  // on the south axis
  const bool hx = hi_word(dx) >= 0x3fe00000, hy = hi_word(dy) >= 0x3fe00000;  // offset >= 1/2
  const int li = ci - G.i0;
  const int LD = G.LD;
  const size_t o = (size_t)(li + G.PI) * LD + (size_t)(cj + G.PJ);
  const double ah = dx + (hx ? -0.5 : 0.5), bh = dy + (hy ? -0.5 : 0.5);  // offsets from the half-integer nodes
  // ---- 1 / r, sin and cos of theta --------------------------------------------
  double ir, st, ct;
  if (lg && A.series_r) ir = G.m.inv_r_n[li + G.PI + hx] * exp_series64((hx ? 1.0 - dx : -dx) * G.dxi);
  else ir = recip64(map_r(G, x1));
  if (ea) {
    const double rest = A.nth - x2;
    ct = (rest - x2) * A.inv_nth;
    st = sqrt64(x2 * rest) * (2.0 * A.inv_nth);
  } else if (A.series_t) {
    turn64(A.th_n[cj + G.PJ + hy], (hy ? dy - 1.0 : dy) * A.pi_nth, st, ct);
  } else {
    sincospi(x2 * A.inv_nth, &st, &ct);
  }
  // ---- gather and push (ballistic inside the outer conductor) -------------------
  if (ci < G.nr_glob) {
    double E[3] = {0.0, 0.0, 0.0}, B[3] = {0.0, 0.0, 0.0};
    if (ci >= 0) {  // no plasma field inside the inner conductor
      const size_t oi = hx ? o : o - LD, oj = hy ? o : o - 1, oij = hy ? oi : oi - 1;
      E[0] = lerp64(F.f[ER], oi, LD, ah, dy);
      E[1] = lerp64(F.f[ETH], oj, LD, dx, bh);
      E[2] = lerp64(F.f[EPH], o, LD, dx, dy);
      B[0] = lerp64(F.f[BR], oj, LD, dx, bh);
      B[1] = lerp64(F.f[BTH], oi, LD, ah, dy);
      B[2] = lerp64(F.f[BPH], oij, LD, ah, bh);
    }
    add_vacuum64(G, A.r0W, ir, st, ct, ci < 0, E, B);
    const double qmdt = hi_word(qw) >= 0 ? A.qmdt : -A.qmdt;
    if (G.pusher == PIC_BORIS) boris64(qmdt, E, B, u);
    else vay64(qmdt, E, B, u);
  }
  // ---- straight 3-D move in the local frame, in units of r (Sec. 3.3) ------------
  const double v = rsqrt64(fma(u[0], u[0], fma(u[1], u[1], fma(u[2], u[2], 1.0)))) * (G.dt * ir);
  const double a = u[0] * v, b = u[1] * v, c = u[2] * v;
  const double s = fma(a, 2.0 + a, fma(b, b, c * c));  // (r'/r)^2 - 1
  const double inv_rn = rsqrt64(1.0 + s);              // r / r'
  double D1, m = 0.0;
  if (ea || !lg) m = s * recip64(1.0 + (1.0 + s) * inv_rn);  // r'/r - 1
  if (lg) D1 = half_log1p64(s) * A.inv_dxi;
  else D1 = m * recip64(ir) * A.inv_dxi;
  const double Px = fma(a, st, fma(b, ct, st)), Pz = fma(a, ct, fma(-b, st, ct));  // before rotating back
  const double R2 = fma(Px, Px, c * c);
  // off the axis by more than rounds to nothing (a square below the normal
  // numbers: Px, c, u_th and u_ph all under 1e-150); across it
  const bool off = hi_word(R2) >= 0x00100000, back = hi_word(Px) < 0;
  const double iR = off ? rsqrt64(R2) : 0.0, R = R2 * iR;
  const double stn = R * inv_rn, ctn = Pz * inv_rn;
  double D2;
  if (ea) {  // nth / 2 (cos th - cos th'), the differences formed without cancellation
    D2 = A.k_th * inv_rn * fma(ct, m - a, b * st);
  } else {   // sin of the turning angle: (b + ct (R - Px)) r / r'
    const double kap = back ? R - Px : (off ? c * c * recip64(R + Px) : 0.0);
    const double num = fma(ct, kap, b), den = fma(st, kap, 1.0 + a), sd = num * inv_rn;
    const bool small = (hi_word(sd) & 0x7fffffff) < 0x3fc00000 && hi_word(den) >= 0;
    D2 = (small ? asin_series64(sd) : atan2(num, den)) * A.k_th;
  }
  // azimuth swept, and the momentum in the new local frame
  const double cp = off ? Px * iR : 1.0, sp = off ? c * iR : 0.0;
  double phi = !back && off && (hi_word(sp) & 0x7fffffff) < 0x3fc00000 ? asin_series64(sp) : atan2(c, Px);
  const double ux = fma(u[0], st, u[1] * ct), uz = fma(u[0], ct, -(u[1] * st));
  if (back) {  // rare: see AxisTies
    const double w2 = u[2] * u[2];
    if (w2 <= (AXIS_TIE * AXIS_TIE) * (fma(u[0], u[0], u[1] * u[1]) + w2)) phi = axis_tie(ties, P.id[k], phi);
  }
  const double uR = fma(cp, ux, sp * u[2]), nup = fma(cp, u[2], -(sp * ux));
  const double nur = fma(uR, stn, uz * ctn), nut = fma(uR, ctn, -(uz * stn));
  const double nx1 = x1 + D1;
  double nx2 = x2 + D2;
  if (!(finite64(nx1) && finite64(nx2) && finite64(nur) && finite64(nut) && finite64(nup))) {
    set_err(err, ERR_NAN);
    P.qw[k] = 0.0;
    return;
  }
  double fni, fnj;
  int ni = floor64(nx1, fni);
  if ((hi_word(nx1) & 0x7fffffff) >= 0x41d00000) ni = hi_word(nx1) < 0 ? -(1 << 30) : 1 << 30;  // beyond 2^30
  if (hi_word(nx2) < 0) nx2 = 0.0;
  int nj = floor64(nx2, fnj);
  if (nj > G.nth - 1 || (hi_word(nx2) & 0x7fffffff) >= 0x41d00000) { nj = G.nth - 1; nx2 = A.nth; fnj = A.nth - 1.0; }
  const bool in = ni >= -G.g && ni < G.nr_glob + G.g;
  const int kx = ni - ci, ky = nj - cj;
  if (!in || kx < -1 || kx > 1 || ky < -1 || ky > 1) {
    set_err(err, ERR_COURANT);
  } else {
    // the path between the stored positions (exact differences: the flux
    // closes the charge's continuity to the rounding of its products), split
    // where it crosses grid lines
    const double d1 = nx1 - x1, d2 = nx2 - x2;
    double mx = fma(0.5, d1, dx), my = fma(0.5, d2, dy);  // the path's midpoint in the old cell's frame
    // the last segment, the only one of most paths: one code for all lanes
    double px = dx, py = dy, q1 = d1, q2 = d2;
    size_t om = o;
    if (kx | ky) {
      const double ex = nx1 - fni, ey = nx2 - fnj;  // end point in the new cell's frame
      const double Xo = kx > 0 ? 1.0 : 0.0, Xn = 1.0 - Xo, Yo = ky > 0 ? 1.0 : 0.0, Yn = 1.0 - Yo;
      double sx = 2.0, sy = 2.0;  // crossing parameters, 0 to 1 (2: no crossing)
      if (kx) sx = (Xo - dx) * recip64(d1);
      if (ky) sy = (Yo - dy) * recip64(d2);
      const bool xf = __double_as_longlong(sx) <= __double_as_longlong(sy);
      // first crossing, in the old cell's frame; the middle cell and its entry point
      const double c1 = clamp01(fma(xf ? sx : sy, xf ? d2 : d1, xf ? dy : dx)), c1x = xf ? Xo : c1, c1y = xf ? c1 : Yo;
      vb_seg64(D.Fr, D.Ft, o, LD, qw, dx, dy, c1x - dx, c1y - dy);
      px = xf ? Xn : c1x;
      py = xf ? c1y : Yn;
      om = o + (size_t)((ptrdiff_t)(xf ? kx : 0) * LD + (xf ? 0 : ky));
      if (kx && ky) {  // second crossing, in the middle cell's frame
        const double c2 = clamp01(fma((xf ? sy : sx) - 1.0, xf ? d1 : d2, xf ? ex : ey)), c2x = xf ? c2 : Xo,
                     c2y = xf ? Yo : c2;
        vb_seg64(D.Fr, D.Ft, om, LD, qw, px, py, c2x - px, c2y - py);
        px = xf ? c2x : Xn;
        py = xf ? Yn : c2y;
        om = o + (size_t)((ptrdiff_t)kx * LD + ky);
      }
      q1 = ex - px;
      q2 = ey - py;
    }
    vb_seg64(D.Fr, D.Ft, om, LD, qw, px, py, q1, q2);
    // azimuthal flux: charge crossing the meridional half-plane, area weights
    // at the midpoint of the grid-coordinate path (reading of the paper)
    size_t oa = o;
    if (hi_word(mx) < 0) { mx += 1.0; oa -= LD; }
    else if (hi_word(mx) >= 0x3ff00000) { mx -= 1.0; oa += LD; }
    if (hi_word(my) < 0) { my += 1.0; oa -= 1; }
    else if (hi_word(my) >= 0x3ff00000) { my -= 1.0; oa += 1; }
    const double w = qw * phi * (0.5 / PI_D);
    const double wx = w * mx, w0 = w - wx, w01 = w0 * my, w11 = wx * my;
    atomicAdd(D.Fp + oa, w0 - w01);
    atomicAdd(D.Fp + oa + LD, wx - w11);
    atomicAdd(D.Fp + oa + 1, w01);
    atomicAdd(D.Fp + oa + LD + 1, w11);
  }
  // removal once the filtered shape lies inside a conductor (Sec. 3.4.2)
  if (ni < -(G.n_filt + 1) || ni >= G.nr_glob + G.n_filt + 1) {
    P.qw[k] = 0.0;
    add_ll(cnt + CNT_DELETED, 1LL);
    return;
  }
  P.x1[k] = nx1;
  P.x2[k] = nx2;
  P.ur[k] = nur;
  P.ut[k] = nut;
  P.up[k] = nup;
}

// ---- stable removal of free slots (block counts, one-block scan, scatter) ----
constexpr int CB = 256;

__global__ void k_count_live(const double *__restrict__ qw, int64_t n, long long *bc) {
  const int64_t k = blockIdx.x * (int64_t)CB + threadIdx.x;
  int live = (k < n && qw[k] != 0.0) ? 1 : 0;
  int s = __syncthreads_count(live);
  if (threadIdx.x == 0) bc[blockIdx.x] = s;
}

__global__ void k_scan_blocks(long long *bc, int64_t nb, long long *total) {
  // exclusive scan of nb block counts by one block of 1024 threads
  __shared__ long long part[1024];
  const int t = threadIdx.x;
  const int64_t per = (nb + 1023) / 1024, b0 = t * per, b1 = min(nb, b0 + per);
  long long s = 0;
  for (int64_t b = b0; b < b1; ++b) s += bc[b];
  part[t] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    long long v = t >= off ? part[t - off] : 0;
    __syncthreads();
    part[t] += v;
    __syncthreads();
  }
  long long run = part[t] - s;
  for (int64_t b = b0; b < b1; ++b) {
    long long c = bc[b];
    bc[b] = run;
    run += c;
  }
  if (t == 1023) *total = part[1023];
}

__global__ void k_scatter_live(Parts64 S, Parts64 D, int64_t n, const long long *__restrict__ boff) {
  __shared__ int wsum[CB / 32];
  const int64_t k = blockIdx.x * (int64_t)CB + threadIdx.x;
  const int live = (k < n && S.qw[k] != 0.0) ? 1 : 0;
  const unsigned m = __ballot_sync(0xffffffffu, live);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int before = __popc(m & ((1u << lane) - 1u));
  if (lane == 0) wsum[w] = __popc(m);
  __syncthreads();
  int base = 0;
  for (int q = 0; q < w; ++q) base += wsum[q];
  if (live) {
    const int64_t d = boff[blockIdx.x] + base + before;
    D.x1[d] = S.x1[k]; D.x2[d] = S.x2[k];
    D.ur[d] = S.ur[k]; D.ut[d] = S.ut[k]; D.up[d] = S.up[k];
    D.qw[d] = S.qw[k]; D.id[d] = S.id[k];
  }
}

__global__ void k_charge64(Grid G, const double *__restrict__ x1, const double *__restrict__ x2,
                           const double *__restrict__ qw, int64_t n, double *Q, double *Qa) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double q = qw[k];
  if (q == 0.0) return;
  const double a = x1[k] - (double)G.i0, b = x2[k], fi = floor(a), fj = floor(b), w1 = a - fi, w2 = b - fj;
  const size_t o = gidx(G, (int)fi, (int)fj);
  const double c00 = (1 - w1) * (1 - w2), c10 = w1 * (1 - w2), c01 = (1 - w1) * w2, c11 = w1 * w2;
  atomicAdd(Q + o, q * c00); atomicAdd(Q + o + G.LD, q * c10);
  atomicAdd(Q + o + 1, q * c01); atomicAdd(Q + o + G.LD + 1, q * c11);
  const double aq = fabs(q);
  atomicAdd(Qa + o, aq * c00); atomicAdd(Qa + o + G.LD, aq * c10);
  atomicAdd(Qa + o + 1, aq * c01); atomicAdd(Qa + o + G.LD + 1, aq * c11);
}

__global__ void k_reduce64(Parts64 P, int64_t n, double qm, double *acc, long long *live) {
  double kin = 0.0, ch = 0.0;
  long long l = 0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    if (P.qw[k] == 0.0) continue;
    const double q = P.qw[k], u2 = P.ur[k] * P.ur[k] + P.ut[k] * P.ut[k] + P.up[k] * P.up[k];
    kin += fabs(q) / qm * (sqrt(1.0 + u2) - 1.0);
    ch += q;
    l += 1;
  }
  block_sum3(kin, ch, l, acc + ACC_KIN, acc + ACC_CHARGE, live);
}

}  // namespace

void particles64(pic_ctx *c, double t) {
  if (c->n_used == 0) return;
  Fields64 F;
  for (int k = 0; k < 6; ++k) F.f[k] = c->f[k];
  Flux64 D{c->Ft[0], c->Ft[1], c->Ft[2]};  // the deposit planes, cleared by the last step
  const Grid &G = c->G;
  Args64 A;
  A.G = G;
  A.r0W = G.r_min * omega_at(G.omega, G.t_spin, t);
  A.qmdt = G.qm * G.dt;
  A.nth = G.nth;
  A.inv_dxi = 1.0 / G.dxi;
  A.k_th = G.th_map == PIC_TH_EQUAL_AREA ? 0.5 * G.nth : G.nth / PI_D;
  A.pi_nth = PI_D / G.nth;
  A.inv_nth = 1.0 / G.nth;
  A.series_r = G.dxi <= 1.0 / 16;
  A.series_t = G.nth >= 32;
  A.th_n = c->th_n64;
  const int64_t blocks = (c->n_used + 255) / 256;
  ++c->launches, launch_on(c->stream, c->overlap, k_particles64, (unsigned)blocks, 256, A, c->p64, c->n_used, F, D,
                           c->d_err, c->d_cnt, axis_ties(c));
}

int64_t compact64(pic_ctx *c) {
  const int64_t n = c->n_used;
  if (n == 0) return 0;
  const int64_t nb = (n + CB - 1) / CB;
  long long *bc = (long long *)c->scratch;
  ++c->launches, k_count_live<<<(unsigned)nb, CB, 0, c->stream>>>(c->p64.qw, n, bc);
  ++c->launches, k_scan_blocks<<<1, 1024, 0, c->stream>>>(bc, nb, c->d_cnt + CNT_SORTED);
  ++c->launches, k_scatter_live<<<(unsigned)nb, CB, 0, c->stream>>>(c->p64, c->q64, n, bc);
  cudaMemcpyAsync(c->h_pinned, c->d_cnt + CNT_SORTED, sizeof(long long), cudaMemcpyDeviceToHost, c->stream);
  cudaStreamSynchronize(c->stream);
  const int64_t live = *c->h_pinned;
  Parts64 t = c->p64;
  c->p64 = c->q64;
  c->q64 = t;
  c->n_used = live;
  return live;
}

void charge64(pic_ctx *c) {
  for (double *p : {c->Q, c->Qa}) cudaMemsetAsync(p, 0, c->grid_elems * sizeof(double), c->stream);
  if (c->n_used == 0) return;
  ++c->launches, k_charge64<<<(unsigned)((c->n_used + 255) / 256), 256, 0, c->stream>>>(c->G, c->p64.x1, c->p64.x2, c->p64.qw,
                                                                        c->n_used, c->Q, c->Qa);
}

void reduce_particles64(pic_ctx *c) {
  if (c->n_used == 0) return;
  // a fixed grid (4 blocks per SM) keeps the same-address atomics few
  ++c->launches, k_reduce64<<<4 * 152, 256, 0, c->stream>>>(c->p64, c->n_used, c->G.qm, c->d_acc,
                                                                        c->d_cnt + CNT_LIVE);
}

}  // namespace pic
