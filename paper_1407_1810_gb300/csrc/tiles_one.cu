// tiles_one.cu -- the FP32 tile kernel with one particle a thread: the form of
// grids of up to PACK_CELLS cells (use_packed in particles32.cu says where the
// line lies).
#include "tiles32.cuh"

namespace pic {
namespace t32 {
namespace {

template <int WJ, int WN>
struct SmemAcc {  // window accessors (shared memory)
  const float *f;           // 6 * WN
  int *hi;                  // 3 * WN : sums of the high parts
  int *lo;                  // 3 * WN : sums of the low parts
  const float *rn;          // f_r(i) of the window's rows
  const float2 *tn;         // (sin, cos) of the node angles of the window's columns
  int wi0, wj0;
  float fs;                 // flux units per unit charge, 2^(KFIX - e)
  __device__ float fld(int c, int i, int j) const { return f[c * WN + (i - wi0) * WJ + (j - wj0)]; }
  __device__ float rad(int i) const { return rn[i - wi0]; }
  __device__ float2 ang(int j) const { return tn[j - wj0]; }
  // unconditional: a test for zero terms would branch around every atomic,
  // which costs more than adding the rare zero
  __device__ void add(int k, int i, int j, int h, int l) const {
    const int e = k * WN + (i - wi0) * WJ + (j - wj0);
    atomicAdd(&hi[e], h);
    atomicAdd(&lo[e], l);
  }
};

struct GlobAcc {  // global-memory accessors (particles outside the window)
  const Args32 *A;
  float fs;
  __device__ float fld(int c, int i, int j) const { return A->f[c][pidx(*A, i, j)]; }
  __device__ float rad(int i) const { return A->r_n[i + A->PI]; }
  __device__ float2 ang(int j) const { return A->th_n[j + A->PJ]; }
  __device__ void add(int k, int i, int j, int h, int l) const {
    const long long v = ((long long)h << SPLIT) + (long long)l;
    if (v) atomicAdd(reinterpret_cast<unsigned long long *>(A->acc[k] + pidx(*A, i, j)), (unsigned long long)v);
  }
};

// Fixed-point split of a flux term cs (in quanta, |cs| <= 2^36) into integers
// h, l with h 2^SPLIT + l = rint(cs), |h| <= 2^18, |l| <= 2^17.  Rounding to
// an integer by adding 1.5 * 2^23 is exact for |x| < 2^22; the subtraction
// cs - h 2^SPLIT is exact (Sterbenz).  Only FP32 adds and integer ops, no
// 64-bit conversions.
__device__ inline void split_fix(float cs, int &h, int &l) {
  const float MAGIC = 12582912.0f, MAGIC_H = 3298534883328.0f;  // 1.5 2^23, 1.5 2^41 (ulp 2^SPLIT)
  const float hm = __fadd_rn(cs, MAGIC_H);                        // cs rounded to a multiple of 2^18
  h = __float_as_int(hm) - 0x54400000;
  const float lf = __fsub_rn(cs, __fsub_rn(hm, MAGIC_H));       // exact
  l = __float_as_int(__fadd_rn(lf, MAGIC)) - 0x4B400000;
}

// bilinear interpolation of field c in cell (i, j) at offsets (a, b).  LERP:
// two linear interpolations along i and one along j (six operations, no
// weights); otherwise the four weights, shared by the components that share a
// staggered point (the form the kernels that hold more live values keep: the
// other one makes them spill)
template <bool LERP, class W>
__device__ inline float bilin(const W &w, int c, int i, int j, float a, float b) {
  if (LERP) {
    const float v0 = fmaf(a, w.fld(c, i + 1, j) - w.fld(c, i, j), w.fld(c, i, j));
    const float v1 = fmaf(a, w.fld(c, i + 1, j + 1) - w.fld(c, i, j + 1), w.fld(c, i, j + 1));
    return fmaf(b, v1 - v0, v0);
  }
  return (1.f - a) * (1.f - b) * w.fld(c, i, j) + a * (1.f - b) * w.fld(c, i + 1, j) +
         (1.f - a) * b * w.fld(c, i, j + 1) + a * b * w.fld(c, i + 1, j + 1);
}

// Villasenor-Buneman fluxes of a straight path p -> q inside cell (i, j)
// (local coordinates in [0, 1], Eq. Jcons, Sec. 3.3).  GUARD skips the terms
// of a zero component, which the segments of a split path often have; a zero
// term adds nothing to the exact sums, so either form gives the same bits.
template <bool GUARD = true, class W>
__device__ inline void vb_seg(const W &w, float scale, int i, int j, float p1, float p2, float q1, float q2) {
  const float d1 = q1 - p1, d2 = q2 - p2, m1 = 0.5f * (p1 + q1), m2 = 0.5f * (p2 + q2);
  const float a = scale * d1, b = scale * d2;
  int h, l;
  if (!GUARD || a != 0.f) {
    split_fix(a * (1.f - m2), h, l);
    w.add(0, i, j, h, l);
    split_fix(a * m2, h, l);
    w.add(0, i, j + 1, h, l);
  }
  if (!GUARD || b != 0.f) {
    split_fix(b * (1.f - m1), h, l);
    w.add(1, i, j, h, l);
    split_fix(b * m1, h, l);
    w.add(1, i + 1, j, h, l);
  }
}

// log1p, atan and expm1 for the small arguments of a single step: truncated
// Taylor series (relative truncation s^6/7, t^8/9 and y^6/720: below 1.3e-10
// for |x| < 1/32), otherwise the library functions
// (the _series forms alone when the arguments are known to be small)
__device__ inline float log1p_series(float s) {
  return s * (1.f - s * (0.5f - s * (0.33333334f - s * (0.25f - s * (0.2f - s * 0.16666667f)))));
}
__device__ inline float atan_series(float y, float x) {
  const float t = y * rcp_(x), t2 = t * t;
  return t * (1.f - t2 * (0.33333334f - t2 * (0.2f - t2 * 0.14285715f)));
}
__device__ inline float exp_series(float y) {
  return 1.f + y * (1.f + y * (0.5f + y * (0.16666667f + y * (0.041666668f + y * 0.008333334f))));
}
__device__ inline float log1p_small(float s) { return fabsf(s) < 0.03125f ? log1p_series(s) : log1pf(s); }
__device__ inline float atan2_small(float y, float x) {
  return x > 0.f && fabsf(y) < 0.03125f * x ? atan_series(y, x) : atan2f(y, x);
}
__device__ inline float exp_small(float y) { return fabsf(y) < 0.03125f ? exp_series(y) : expf(y); }

__device__ inline float clamp01(float v) { return fminf(fmaxf(v, 0.f), 1.f); }



// ---- momentum in increments ----------------------------------------------
// The FP32 step computes each change of the momentum -- the push, then the
// rotation into the particle's new local frame -- as an increment du whose
// rounding errors are relative to |du|, not to |u|: for a particle turning by
// a small angle per step they are that much smaller, and the step adds to u
// only the rounding of the one sum u + du that stores it.
//
// This arithmetic is written with explicitly rounded operations: the step is
// inlined twice (shared-memory window and global memory), and a product the
// compiler fused into an FMA in one copy but not in the other would make the
// two paths differ in the last bit.

__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// a x b - c x d (one component of a cross product)
__device__ __forceinline__ float cross_(float a, float b, float c, float d) { return fma_(a, b, -mul_(c, d)); }
__device__ __forceinline__ float dot3_(float a0, float a1, float a2, float b0, float b1, float b2) {
  return fma_(a0, b0, fma_(a1, b1, mul_(a2, b2)));
}
// sin x and cos x - 1 of a small angle: x (1 - x^2/6 + x^4/120) and
// -x^2/2 (1 - x^2/12 + x^4/360), relative truncation below x^6/5040 (under
// 2^-28 for |x| < 0.16)
__device__ __forceinline__ void sin_cosm1_series(float x, float &s, float &cm1) {
  const float x2 = mul_(x, x);
  s = mul_(x, fma_(-x2, fma_(-x2, 0.008333334f, 0.16666667f), 1.f));
  cm1 = mul_(mul_(-0.5f, x2), fma_(-x2, fma_(-x2, 0.0027777778f, 0.083333336f), 1.f));
}

// Vay (2008) push, Sec. 2, as u' - u: with a = u + (q dt/m) E + v x tau and
// t = tau / gamma', u' = s (a + (a.t) t + a x t), s = 1 / (1 + t^2), i.e.
// u' - a = s ((a.t) t + a x t - t^2 a).
__device__ inline void vay_delta(float qmdt, const float E[3], const float B[3], const float u[3], float du[3]) {
  const float h = mul_(0.5f, qmdt);
  const float ig0 = rsqrt_(add_(1.f, dot3_(u[0], u[1], u[2], u[0], u[1], u[2])));
  const float tau0 = mul_(h, B[0]), tau1 = mul_(h, B[1]), tau2 = mul_(h, B[2]);
  const float v0 = mul_(u[0], ig0), v1 = mul_(u[1], ig0), v2 = mul_(u[2], ig0);
  const float d0 = fma_(qmdt, E[0], cross_(v1, tau2, v2, tau1));
  const float d1 = fma_(qmdt, E[1], cross_(v2, tau0, v0, tau2));
  const float d2 = fma_(qmdt, E[2], cross_(v0, tau1, v1, tau0));
  const float a0 = add_(u[0], d0), a1 = add_(u[1], d1), a2 = add_(u[2], d2);
  const float tau2s = dot3_(tau0, tau1, tau2, tau0, tau1, tau2);
  const float ustar = dot3_(a0, a1, a2, tau0, tau1, tau2);
  const float sigma = sub_(add_(1.f, dot3_(a0, a1, a2, a0, a1, a2)), tau2s);
  const float disc = fma_(sigma, sigma, mul_(4.f, fma_(ustar, ustar, tau2s)));
  const float g2 = mul_(0.5f, add_(sigma, sqrtf(disc)));
  const float ig = rsqrt_(g2);
  const float t0 = mul_(tau0, ig), t1 = mul_(tau1, ig), t2 = mul_(tau2, ig);
  const float tt = dot3_(t0, t1, t2, t0, t1, t2);
  const float sc = rcp_(add_(1.f, tt));
  const float at = dot3_(a0, a1, a2, t0, t1, t2);
  du[0] = fma_(sc, sub_(fma_(at, t0, cross_(a1, t2, a2, t1)), mul_(tt, a0)), d0);
  du[1] = fma_(sc, sub_(fma_(at, t1, cross_(a2, t0, a0, t2)), mul_(tt, a1)), d1);
  du[2] = fma_(sc, sub_(fma_(at, t2, cross_(a0, t1, a1, t0)), mul_(tt, a2)), d2);
}

// Boris (1970) push, Sec. 2, as u' - u: half electric kick h E, rotation
// u- -> u+ = u- + (u- + u- x t) x s, half kick; u' - u = 2 h E + (u- + u- x t) x s.
__device__ inline void boris_delta(float qmdt, const float E[3], const float B[3], const float u[3], float du[3]) {
  const float h = mul_(0.5f, qmdt);
  const float he0 = mul_(h, E[0]), he1 = mul_(h, E[1]), he2 = mul_(h, E[2]);
  const float um0 = add_(u[0], he0), um1 = add_(u[1], he1), um2 = add_(u[2], he2);
  const float ig = rsqrt_(add_(1.f, dot3_(um0, um1, um2, um0, um1, um2)));
  const float hi = mul_(h, ig);
  const float t0 = mul_(hi, B[0]), t1 = mul_(hi, B[1]), t2 = mul_(hi, B[2]);
  const float f = mul_(2.f, rcp_(add_(1.f, dot3_(t0, t1, t2, t0, t1, t2))));
  const float p0 = add_(um0, cross_(um1, t2, um2, t1)), p1 = add_(um1, cross_(um2, t0, um0, t2)),
              p2 = add_(um2, cross_(um0, t1, um1, t0));
  const float s0 = mul_(f, t0), s1 = mul_(f, t1), s2 = mul_(f, t2);
  du[0] = fma_(2.f, he0, cross_(p1, s2, p2, s1));
  du[1] = fma_(2.f, he1, cross_(p2, s0, p0, s2));
  du[2] = fma_(2.f, he2, cross_(p0, s1, p1, s0));
}

// One particle step.  Returns false when the particle is removed.
template <int SPEC, class W>
__device__ inline bool step32(const Args32 &A, const W &w, int64_t k, uint32_t &cell, float &dx, float &dy, float &ur,
                              float &ut, float &up, const float qw) {
  const Flags<SPEC> F(A);
  const int ci = (int)(cell >> 16) - CELL_BIAS, cj = (int)(cell & 0xffffu);
  // ---- geometry of the particle's position (Sec. 3.2) -----------------------
  const float rn = w.rad(ci);
  constexpr bool series = SPEC != SPEC_GENERIC;  // arguments below 1/32: no fallback
  const float r = F.r_log ? rn * (series ? exp_series(dx * A.dxi) : exp_small(dx * A.dxi)) : rn + dx * A.dxi;
  // sin and cos of theta from the distance to the nearer pole, which both
  // offsets resolve to FP32 relative precision (1 - x2/nth would cancel)
  const float x2 = (float)cj + dy;                 // distance to the north pole
  const float rest = (float)(A.nth - cj) - dy;     // distance to the south pole
  float st, ct;
  if (F.th_ea) {  // cos th = 1 - 2 x2/nth, sin th = 2 sqrt(x2 (nth - x2))/nth
    ct = (rest - x2) * A.inv_nth;
    st = 2.f * sqrtf(fmaxf(x2 * rest, 0.f)) * A.inv_nth;
  } else if (series) {
    // linear map: the node angle's sine and cosine from the column table,
    // turned by the offset's angle (at most pi / nth, nth >= 32 on the
    // specialised grids: short series).  The node taken is the one on the
    // pole's side of the particle in its hemisphere, so both terms of sin th
    // have one sign and sin th keeps FP32 relative precision up to the poles.
    const bool north = 2 * cj < A.nth;
    const float2 n = w.ang(north ? cj : cj + 1);
    float sb, cb1;
    sin_cosm1_series(mul_(north ? dy : dy - 1.f, A.pi_nth), sb, cb1);
    st = fma_(n.y, sb, fma_(n.x, cb1, n.x));   // sin th_n cos b + cos th_n sin b
    ct = fma_(-n.x, sb, fma_(n.y, cb1, n.y));  // cos th_n cos b - sin th_n sin b
  } else if (x2 <= rest) {
    sincospif(x2 * A.inv_nth, &st, &ct);
  } else {
    sincospif(rest * A.inv_nth, &st, &ct);
    ct = -ct;
  }
  // ---- gather + push (ballistic inside the outer conductor) -----------------
  float du[3] = {0.f, 0.f, 0.f};  // momentum change of the step: push, then frame rotation
  if (ci < A.nr) {
    float E[3], B[3];
    const Vac<float> V{F.vacuum, A.b0, A.r_min, A.omega_t};
    vacuum_field<float>(V, r, st, ct, ci < 0, E, B);
    if (F.vacuum == PIC_VAC_MONOPOLE || F.vacuum == PIC_VAC_MONOPOLE_ROTATOR) {  // monopole B_r = b0 (r0/r)^2 with b0 to ~1e-14
      const float q = A.r_min * rcp_(r);
      B[0] = fmaf(A.b0_lo, q * q, B[0]);
    }
    if (ci >= 0) {  // plasma field only outside the inner conductor
      const bool hx = dx >= 0.5f, hy = dy >= 0.5f;
      const int ih = hx ? ci : ci - 1, jh = hy ? cj : cj - 1;
      const float ah = hx ? dx - 0.5f : dx + 0.5f, bh = hy ? dy - 0.5f : dy + 0.5f;
      constexpr bool L = SPEC == SPEC_MONOPOLE;
      E[0] += bilin<L>(w, ER, ih, cj, ah, dy);
      E[1] += bilin<L>(w, ETH, ci, jh, dx, bh);
      E[2] += bilin<L>(w, EPH, ci, cj, dx, dy);
      B[0] += bilin<L>(w, BR, ci, jh, dx, bh);
      B[1] += bilin<L>(w, BTH, ih, cj, ah, dy);
      B[2] += bilin<L>(w, BPH, ih, jh, ah, bh);
    }
    const float u[3] = {ur, ut, up};
    // local (r, th, ph) is a right-handed orthonormal frame: the Cartesian
    // push formulas apply to its components unchanged
    const float qmdt = qw > 0.f ? A.qmdt : -A.qmdt;
    if (F.pusher == PIC_BORIS) boris_delta(qmdt, E, B, u, du);
    else vay_delta(qmdt, E, B, u, du);
  }
  // u^{n+1/2} in FP32, for the move
  const float pr = add_(ur, du[0]), pt = add_(ut, du[1]), pp = add_(up, du[2]);
  // ---- move in the local frame (Sec. 3.3) -----------------------------------
  const float ig = rsqrt_(1.f + pr * pr + pt * pt + pp * pp);
  const float vr = pr * ig, vt = pt * ig, vp = pp * ig;
  const float Dr = fmaf(vr, A.dt, vr * A.dt_lo), Dt = fmaf(vt, A.dt, vt * A.dt_lo), Dp = fmaf(vp, A.dt, vp * A.dt_lo);
  const float ir = rcp_(r);
  const float a = Dr * ir, b = Dt * ir, c = Dp * ir;
  const float s = a * (2.f + a) + b * b + c * c;  // (r'/r)^2 - 1
  const float L1 = F.r_log ? 0.5f * (series ? log1p_series(s) : log1p_small(s)) : r * s * rcp_(1.f + sqrtf(1.f + s));
  const float D1 = fmaf(L1, A.inv_dxi, L1 * A.inv_dxi_lo);
  const float p = r + Dr, q = Dt;
  const float Px = p * st + q * ct, Pz = p * ct - q * st;  // displaced point, (R, z) before rotating back
  const float Rn = sqrtf(Px * Px + Dp * Dp);
  const float kap = Px >= 0.f ? (Rn + Px > 0.f ? Dp * Dp * rcp_(Rn + Px) : 0.f) : Rn - Px;  // R' - Px
  const float dth = series ? atan_series(q + ct * kap, p + st * kap) : atan2_small(q + ct * kap, p + st * kap);
  // sin(dth) and cos(dth) - 1 of the meridional rotation, from the half angle
  // (or, for the small angles of the specialised grids, short series)
  float D2, sd, cd1;
  if (F.th_ea || !series) {
    float sh, ch;
    sincosf(0.5f * dth, &sh, &ch);
    sd = mul_(2.f, mul_(sh, ch));
    cd1 = mul_(-2.f, mul_(sh, sh));
    D2 = F.th_ea ? A.nth_f * (st * ch + ct * sh) * sh : fmaf(dth, A.k2_hi, dth * A.k2_lo);
  } else {
    sin_cosm1_series(dth, sd, cd1);
    D2 = fmaf(dth, A.k2_hi, dth * A.k2_lo);
  }
  // new cell and offsets (carries are exact integers)
  float tx = dx + D1, ty = dy + D2;
  int kx = (int)floorf(tx), ky = (int)floorf(ty);
  float nx = tx - (float)kx, ny = ty - (float)ky;
  if (nx >= 1.f) { nx = 0.f; ++kx; }
  if (ny >= 1.f) { ny = 0.f; ++ky; }
  int ncj = cj + ky;
  if (ncj < 0) { ncj = 0; ky = -cj; ny = 0.f; }                       // rounding below the axis
  if (ncj > A.nth - 1) { ncj = A.nth - 1; ky = ncj - cj; ny = 1.f; }   // rounding past the south axis
  // momentum into the new local frame, as an increment: Cartesian at phi = 0
  // (x along R), rotated back about z by -phi' (cos phi' - 1 = -kap / R',
  // sin phi' = Dp / R'), then into (r', th') at th' = th + dth:
  //   u_r' = u_r cos dth + u_th sin dth + dx st',  u_th' = -u_r sin dth + u_th cos dth + dx ct',
  //   u_ph' = u_ph + dy,  with (dx, dy) the change of (u_x, u_ph) under the azimuthal rotation
  {
    const float ux = fma_(pr, st, mul_(pt, ct));
    const float iRn = Rn > 0.f ? rcp_(Rn) : 0.f;
    const float cm1 = mul_(-kap, iRn), sph = mul_(Dp, iRn);
    const float dxr = fma_(ux, cm1, mul_(sph, pp)), dyr = fma_(pp, cm1, -mul_(sph, ux));
    const float irn = rsqrtf(fmaxf(fma_(Rn, Rn, mul_(Pz, Pz)), 1e-30f));
    const float stn = mul_(Rn, irn), ctn = mul_(Pz, irn);
    du[0] = add_(du[0], fma_(pr, cd1, fma_(pt, sd, mul_(dxr, stn))));
    du[1] = add_(du[1], fma_(pt, cd1, fma_(-pr, sd, mul_(dxr, ctn))));
    du[2] = add_(du[2], dyr);
  }
  const float nur = add_(ur, du[0]), nut = add_(ut, du[1]), nup = add_(up, du[2]);
  if (!(isfinite(nx) && isfinite(ny) && isfinite(nur) && isfinite(nut) && isfinite(nup)) || kx < -1 || kx > 1 ||
      ky < -1 || ky > 1) {
    atomicOr(A.err, (isfinite(nx) && isfinite(nur)) ? ERR_COURANT : ERR_NAN);
    return false;
  }
  // ---- Villasenor-Buneman deposit along the grid-coordinate path -----------
  // Three segments, split where the path crosses the x and y grid lines in
  // the order it meets them; a line not crossed puts its segment at zero
  // length (zero terms are skipped).  Branch-free, so lanes that cross and
  // lanes that do not run the same instructions -- except for two votes of
  // the converged group: when no lane crosses a line the path is its one
  // nonzero segment (the same terms as in the general form, without the
  // zero-component tests: a zero term adds nothing), and when no lane crosses
  // both lines the third segment is empty for every lane.  Each lane's terms
  // are the same whichever form its group takes.  The move of one step is a small
  // fraction of a cell away from the inner boundary (about 0.35 / r of one at
  // 4096 log cells), so most warps take it there.
  const float scale = qw * w.fs;  // exact: fs is a power of two
  const unsigned grp = __activemask();
  if (__all_sync(grp, (kx | ky) == 0)) {
    vb_seg<false>(w, scale, ci, cj, dx, dy, nx, ny);
  } else {
  const float Dxs = kx == 0 ? nx - dx : (kx > 0 ? (1.f - dx) + nx : -(dx + (1.f - nx)));
  const float Dys = ky == 0 ? ny - dy : (ky > 0 ? (1.f - dy) + ny : -(dy + (1.f - ny)));
  // crossing parameters: any point on the crossed grid line keeps charge
  // conservation exact, so an approximate reciprocal is enough here
  const float sx = kx > 0 ? (1.f - dx) * rcp_(Dxs) : (kx < 0 ? -dx * rcp_(Dxs) : 2.f);
  const float sy = ky > 0 ? (1.f - dy) * rcp_(Dys) : (ky < 0 ? -dy * rcp_(Dys) : 2.f);
  const float Xo = kx > 0 ? 1.f : 0.f, Xn = 1.f - Xo;  // crossed x line in the old / new x frame
  const float Yo = ky > 0 ? 1.f : 0.f, Yn = 1.f - Yo;
  const bool xfirst = sx <= sy;
  // first crossing point, in the frame of the cell the path leaves
  float c1x, c1y;
  if (xfirst) { c1x = kx ? Xo : nx; c1y = kx ? clamp01(dy + sx * Dys) : ny; }
  else        { c1y = Yo; c1x = clamp01(dx + sy * Dxs); }
  // cell of the middle segment and the entry point there
  const int mi = ci + (xfirst ? kx : 0), mj = cj + (xfirst ? 0 : ky);
  const float e1x = (xfirst && kx) ? Xn : c1x, e1y = (!xfirst) ? Yn : c1y;
  vb_seg(w, scale, ci, cj, dx, dy, c1x, c1y);
  if (__all_sync(grp, (kx & ky) == 0)) {
    // no lane of the group crosses both lines (kx & ky is nonzero only when
    // both are): the middle segment ends at the end point and the third has
    // zero length, as in the general form below
    vb_seg(w, scale, mi, mj, e1x, e1y, nx, ny);
  } else {
  // second crossing point, in the frame of the middle cell
  float c2x, c2y;
  if (kx && ky) {
    if (xfirst) { c2y = Yo; c2x = clamp01(nx - (1.f - sy) * Dxs); }
    else        { c2x = Xo; c2y = clamp01(ny - (1.f - sx) * Dys); }
  } else {
    c2x = nx; c2y = ny;
  }
  const float e2x = (kx && ky && !xfirst) ? Xn : c2x, e2y = (kx && ky && xfirst) ? Yn : c2y;
  vb_seg(w, scale, mi, mj, e1x, e1y, c2x, c2y);
  vb_seg(w, scale, ci + kx, cj + ky, e2x, e2y, nx, ny);
  }
  }
  // azimuthal flux: charge crossing the meridional half-plane, qw dphi / 2 pi,
  // area weights at the midpoint of the grid path
  {
    float phi = atan2_small(Dp, Px);
    if (Px < 0.f && pp * pp <= (float)(AXIS_TIE * AXIS_TIE) * (pr * pr + pt * pt + pp * pp))
      phi = axis_tie(A.ties, A.ids[k], phi);  // rare: see AxisTies
    const float v = scale * phi * 0.15915494309189535f;
    const float mx = 0.5f * (dx + (float)kx + nx), my = 0.5f * (dy + (float)ky + ny);
    const float fx = floorf(mx), fy = floorf(my);
    const float wx = mx - fx, wy = my - fy;
    const int i0 = ci + (int)fx, j0 = cj + (int)fy;
    {  // v is nonzero for nearly every particle: no test
      int h, l;
      split_fix(v * (1.f - wx) * (1.f - wy), h, l);
      w.add(2, i0, j0, h, l);
      split_fix(v * wx * (1.f - wy), h, l);
      w.add(2, i0 + 1, j0, h, l);
      split_fix(v * (1.f - wx) * wy, h, l);
      w.add(2, i0, j0 + 1, h, l);
      split_fix(v * wx * wy, h, l);
      w.add(2, i0 + 1, j0 + 1, h, l);
    }
  }
  // ---- store; removal once the filtered shape is inside a conductor ---------
  const int nci = ci + kx;
  if (nci < -(A.n_filt + 1) || nci >= A.nr + A.n_filt + 1) return false;
  cell = ((uint32_t)(nci + CELL_BIAS) << 16) | (uint32_t)ncj;
  dx = nx; dy = ny; ur = nur; ut = nut; up = nup;
  return true;
}

// the rare path: a particle outside its tile's window (inlined: an
// out-of-line call costs register spills around it in the hot loop)
template <int SPEC>
__device__ inline bool step32_global(const Args32 &A, float fs, int64_t k, uint32_t &cell, float &dx, float &dy,
                                     float &ur, float &ut, float &up, const float qw) {
  const GlobAcc gw{&A, fs};
  return step32<SPEC>(A, gw, k, cell, dx, dy, ur, ut, up, qw);
}

template <int SPEC, class SW>
__device__ inline void process_v(const Args32 &A, Parts32 P, int64_t k, bool win, const SW &sw,
                                 int wi_lo, int wi_hi, int wj_lo, int wj_hi, int &dead, const float qw,
                                 uint32_t cell, float dx, float dy, float ur, float ut, float up) {
  if (qw == 0.f) return;
  const int ci = (int)(cell >> 16) - CELL_BIAS, cj = (int)(cell & 0xffffu);
  bool alive;
  if (win && ci >= wi_lo && ci < wi_hi && cj >= wj_lo && cj < wj_hi)
    alive = step32<SPEC>(A, sw, k, cell, dx, dy, ur, ut, up, qw);
  else
    alive = step32_global<SPEC>(A, sw.fs, k, cell, dx, dy, ur, ut, up, qw);
  if (!alive) { P.qw[k] = 0.f; ++dead; return; }
  P.cell[k] = cell;
  P.dx[k] = dx; P.dy[k] = dy;
  P.ur[k] = ur; P.ut[k] = ut; P.up[k] = up;
}

template <int SPEC, class SW>
__device__ inline void process(const Args32 &A, Parts32 P, int64_t k, bool win, const SW &sw,
                               int wi_lo, int wi_hi, int wj_lo, int wj_hi, int &dead) {
  process_v<SPEC>(A, P, k, win, sw, wi_lo, wi_hi, wj_lo, wj_hi, dead, P.qw[k], P.cell[k], P.dx[k], P.dy[k], P.ur[k],
                  P.ut[k], P.up[k]);
}

// per-thread asynchronous copy of 4 bytes global -> shared (no registers held)
__device__ inline void cp_async4(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ inline void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ inline void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }


// One tile CTA (or one block of unbinned particles) of the FP32 step: block
// `blk` of the member whose arguments are A and P, its six field tensor maps
// at `maps` (kernel parameters, or global memory when GMAPS).
template <int TI, int TJ, int SPEC, bool GMAPS>
__device__ __forceinline__ void tiles32_block(const Args32 &A, const Parts32 &P, const CUtensorMap *maps,
                                              unsigned blk) {
  using BX_ = Box<TI, TJ>;
  constexpr int WI = BX_::WI, WJ = BX_::WJ, WN = BX_::WN, WB = BX_::WB, SLOT = BX_::SLOT;
  __shared__ __align__(128) float sbuf[BX_::SF + BX_::U1];
  __shared__ __align__(16) uint32_t spf[2][7][NT];  // each thread's next particle, copied ahead
  float *const sf = sbuf;                                      // 6 WN: the window
  float *const stage = sbuf + BX_::SF;                         // 6 SLOT: the boxes, first
  int *const shi = reinterpret_cast<int *>(sbuf + BX_::SF);    // 3 WN: then the accumulators
  int *const slo = shi + 3 * WN;                               // 3 WN
  __shared__ float srn[WI];
  __shared__ float2 stn[WJ];
  __shared__ int sdead, sok;
  __shared__ __align__(8) uint64_t sbar;
  int dead = 0;
  const float fs = __int_as_float((127 + KFIX - qexp_value(A.qexp)) << 23);  // 2^(KFIX - e)
  if (blk < (uint64_t)A.nunits) {
    int t;
    int64_t b0, b1;
    unit_range(A, A.units[blk], t, b0, b1);
    if (b1 <= b0) return;
    const int i0 = A.row0 + (t / A.ntj) * TI, j0 = (t % A.ntj) * TJ;
    const int wi0 = i0 - H - 1, wj0 = j0 - H - 1;
    if (threadIdx.x == 0) {
      sdead = 0;
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sbar)));
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&sbar)),
                   "r"((uint32_t)(6 * WI * WB * sizeof(float)))
                   : "memory");
      const int x = wj0 - WOFF + A.PJ, y = wi0 + A.PI;  // x: a multiple of 4 (static_assert above)
      if (GMAPS) {
#pragma unroll
        for (int c = 0; c < 6; ++c) tensormap_acquire(maps + c);
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) tma_window(stage + c * SLOT, maps + c, x, y, &sbar);
      // bounded wait: on a timeout the error is latched, the copies get a
      // second bounded wait (they write into this block's shared memory) and
      // the tile is skipped
      bool ok = window_wait(&sbar, 1ll << 26);
      if (!ok) {
        atomicOr(A.err, ERR_TIMEOUT);
        window_wait(&sbar, 1ll << 26);
      }
      sok = ok ? 1 : 0;
    }
    for (int e = threadIdx.x; e < WI; e += NT) srn[e] = A.r_n[wi0 + e + A.PI];
    if (SPEC != SPEC_GENERIC)
      for (int e = threadIdx.x; e < WJ; e += NT) stn[e] = A.th_n[wj0 + e + A.PJ];
    __syncthreads();
    if (!sok) return;
    for (int e = threadIdx.x; e < WN; e += NT) {
      const int r = e / WJ, q = e % WJ;
#pragma unroll
      for (int c = 0; c < 6; ++c) sf[c * WN + e] = stage[c * SLOT + r * WB + q + WOFF];
    }
    __syncthreads();  // the staging area becomes the accumulators
    for (int e = threadIdx.x; e < 3 * WN; e += NT) { shi[e] = 0; slo[e] = 0; }
    __syncthreads();
    const SmemAcc<WJ, WN> sw{sf, shi, slo, srn, stn, wi0, wj0, fs};
    {
      const int t = threadIdx.x;
      auto fetch = [&](int buf, int64_t k) {
        cp_async4(&spf[buf][0][t], P.qw + k); cp_async4(&spf[buf][1][t], P.cell + k);
        cp_async4(&spf[buf][2][t], P.dx + k); cp_async4(&spf[buf][3][t], P.dy + k);
        cp_async4(&spf[buf][4][t], P.ur + k); cp_async4(&spf[buf][5][t], P.ut + k);
        cp_async4(&spf[buf][6][t], P.up + k);
      };
      int64_t k = b0 + t;
      if (k < b1) fetch(0, k);
      cp_commit();
      for (int buf = 0; k < b1; k += NT, buf ^= 1) {
        if (k + NT < b1) fetch(buf ^ 1, k + NT);
        cp_commit();
        cp_wait<1>();  // this particle's copies (the next one's may still be in flight)
        process_v<SPEC>(A, P, k, true, sw, i0 - H, i0 + TI + H, j0 - H, j0 + TJ + H, dead,
                        __uint_as_float(spf[buf][0][t]), spf[buf][1][t], __uint_as_float(spf[buf][2][t]),
                        __uint_as_float(spf[buf][3][t]), __uint_as_float(spf[buf][4][t]),
                        __uint_as_float(spf[buf][5][t]), __uint_as_float(spf[buf][6][t]));
      }
      cp_wait<0>();
    }
    if (dead) atomicAdd(&sdead, dead);
    __syncthreads();
    for (int e = threadIdx.x; e < WN; e += NT) {
      const size_t o = pidx(A, wi0 + e / WJ, wj0 + e % WJ);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int hsum = shi[c * WN + e], lsum = slo[c * WN + e];
        if (sums_full(hsum, lsum, b1 - b0)) atomicOr(A.err, ERR_CAPACITY);
        const long long v = ((long long)hsum << SPLIT) + (long long)lsum;
        if (v) atomicAdd(reinterpret_cast<unsigned long long *>(A.acc[c] + o), (unsigned long long)v);
      }
    }
    if (threadIdx.x == 0 && sdead) add_ll(A.cnt + CNT_DELETED, sdead);
  } else {  // particles outside any bin (injected since the last sort)
    const SmemAcc<WJ, WN> none{nullptr, nullptr, nullptr, nullptr, nullptr, 0, 0, fs};
    const int64_t k = A.sorted_end + (int64_t)(blk - A.nunits) * NT + threadIdx.x;
    if (k < A.n_used) process<SPEC>(A, P, k, false, none, 0, 0, 0, 0, dead);
    if (dead) add_ll(A.cnt + CNT_DELETED, dead);
  }
}

template <int TI, int TJ, int SPEC>
__global__ void __launch_bounds__(NT, 4) k_tiles32(Args32 A, Parts32 P, const __grid_constant__ TileMaps maps) {
  follow();
  tiles32_block<TI, TJ, SPEC, false>(A, P, maps.m, blockIdx.x);
}

// the tile kernel over several members of an ensemble in one grid; see
// ens_tiles32 for what its launches do to each other
template <int TI, int TJ, int SPEC>
__global__ void __launch_bounds__(NT, 4) k_ens_tiles32(const __grid_constant__ EnsTileBatch B) {
  next_may_start();
  int lo = 0, hi = B.n - 1;  // the member owning this block
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((unsigned)B.off[mid] <= blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const EnsTileArg &T = B.a[lo];
  tiles32_block<TI, TJ, SPEC, true>(T.A, T.P, T.maps, blockIdx.x - (unsigned)B.off[lo]);
  follow();
}

template <int SPEC>
void launch(int shape, unsigned blocks, cudaStream_t s, bool overlap, const Args32 &A, const Parts32 &P, const TileMaps &M) {
  if (shape == 1) launch_on(s, overlap, k_tiles32<8, 32, SPEC>, blocks, NT, A, P, M);
  else if (shape == 2) launch_on(s, overlap, k_tiles32<32, 8, SPEC>, blocks, NT, A, P, M);
  else launch_on(s, overlap, k_tiles32<16, 16, SPEC>, blocks, NT, A, P, M);
}

template <int SPEC>
void launch_ens(int shape, unsigned blocks, cudaStream_t s, bool beside, const EnsTileBatch &B) {
  if (shape == 1) launch_on(s, beside, k_ens_tiles32<8, 32, SPEC>, blocks, NT, B);
  else if (shape == 2) launch_on(s, beside, k_ens_tiles32<32, 8, SPEC>, blocks, NT, B);
  else launch_on(s, beside, k_ens_tiles32<16, 16, SPEC>, blocks, NT, B);
}

}  // namespace

void launch_one(int spec, int shape, unsigned blocks, cudaStream_t s, bool overlap, const Args32 &A, const Parts32 &P,
                const TileMaps &M) {
  if (spec == SPEC_MONOPOLE) launch<SPEC_MONOPOLE>(shape, blocks, s, overlap, A, P, M);
  else if (spec == SPEC_ROTATOR) launch<SPEC_ROTATOR>(shape, blocks, s, overlap, A, P, M);
  else launch<SPEC_GENERIC>(shape, blocks, s, overlap, A, P, M);
}

void launch_ens_one(int spec, int shape, unsigned blocks, cudaStream_t s, bool beside,
                    const EnsTileBatch &B) {
  if (spec == SPEC_MONOPOLE) launch_ens<SPEC_MONOPOLE>(shape, blocks, s, beside, B);
  else if (spec == SPEC_ROTATOR) launch_ens<SPEC_ROTATOR>(shape, blocks, s, beside, B);
  else launch_ens<SPEC_GENERIC>(shape, blocks, s, beside, B);
}

}  // namespace t32
}  // namespace pic
