// tiles_two.cu -- the FP32 tile kernel with two particles a thread in packed
// FP32 instructions: the form of large grids.
#include "tiles32.cuh"

namespace pic {
namespace t32 {
namespace {

// ---- arithmetic on the particles of a thread -----------------------------------
// A thread of the tile kernel steps two particles.  Blackwell's packed FP32
// instructions (fma, add, mul on a register pair) do both particles' operation
// in one issue slot; the kernel is bound by issue slots (676 a particle and
// 91 % of them used with one particle a thread), so the step is written on
// Vf<NL>, the NL particles of a thread: NL = 2 in the tile's window, NL = 1
// for the rare particle outside it.  Every operation is explicitly rounded, so
// both forms give the same bits.  The packed instructions have no operand
// negation: differences are fma(b, -1, a), and products are arranged so that
// the sign sits in a constant.  The compiler contracts a packed product and
// sum into one fma whatever their rounding modifiers, and a scalar pair of
// intrinsics never: add_ is therefore never given a product (fma_ is, or the
// negated product is subtracted, which no instruction fuses).
//
// Measured (1024 x 1024 monopole, 6.3e7 particles, first step after a sort by
// cell): 1.17 -> 0.91 ms, 407 issue slots a particle (70 % of the issue slots,
// 76 % of the shared-memory wavefronts used); once the order inside the tiles
// has mixed, 1.06 ms, bound by the bank conflicts of the gather's loads and the
// deposit's atomics (random cells: 72 + 57 wavefronts a warp).  More CTAs do
// not help (5 an SM at 96 registers: 2 % slower).
using pic::rcp_;
using pic::rsqrt_;
template <int NL>
struct Vf {
  float v[NL];
  __device__ __forceinline__ float &operator[](int l) { return v[l]; }
  __device__ __forceinline__ float operator[](int l) const { return v[l]; }
};
template <int NL>
__device__ __forceinline__ Vf<NL> bc(float c) {
  Vf<NL> r;
#pragma unroll
  for (int l = 0; l < NL; ++l) r[l] = c;
  return r;
}
__device__ __forceinline__ float2 pk(const Vf<2> &a) { return make_float2(a.v[0], a.v[1]); }
__device__ __forceinline__ Vf<2> up(float2 a) { return Vf<2>{{a.x, a.y}}; }
template <int NL>
__device__ __forceinline__ Vf<NL> fma_(const Vf<NL> &a, const Vf<NL> &b, const Vf<NL> &c) {
  if constexpr (NL == 2) return up(__ffma2_rn(pk(a), pk(b), pk(c)));
  else return Vf<NL>{{__fmaf_rn(a[0], b[0], c[0])}};
}
template <int NL>
__device__ __forceinline__ Vf<NL> mul_(const Vf<NL> &a, const Vf<NL> &b) {
  if constexpr (NL == 2) return up(__fmul2_rn(pk(a), pk(b)));
  else return Vf<NL>{{__fmul_rn(a[0], b[0])}};
}
template <int NL>
__device__ __forceinline__ Vf<NL> add_(const Vf<NL> &a, const Vf<NL> &b) {
  if constexpr (NL == 2) return up(__fadd2_rn(pk(a), pk(b)));
  else return Vf<NL>{{__fadd_rn(a[0], b[0])}};
}
template <int NL>
__device__ __forceinline__ Vf<NL> add_rd(const Vf<NL> &a, const Vf<NL> &b) {  // rounded down
  if constexpr (NL == 2) return up(__fadd2_rd(pk(a), pk(b)));
  else return Vf<NL>{{__fadd_rd(a[0], b[0])}};
}
template <int NL>
__device__ __forceinline__ Vf<NL> sub_(const Vf<NL> &a, const Vf<NL> &b) {  // a - b, one rounding
  return fma_(b, bc<NL>(-1.f), a);
}
// with a constant (the same for every particle)
template <int NL>
__device__ __forceinline__ Vf<NL> mul_(const Vf<NL> &a, float c) { return mul_(a, bc<NL>(c)); }
template <int NL>
__device__ __forceinline__ Vf<NL> add_(const Vf<NL> &a, float c) { return add_(a, bc<NL>(c)); }
template <int NL>
__device__ __forceinline__ Vf<NL> fma_(const Vf<NL> &a, const Vf<NL> &b, float c) { return fma_(a, b, bc<NL>(c)); }
template <int NL>
__device__ __forceinline__ Vf<NL> fma_(const Vf<NL> &a, float b, const Vf<NL> &c) { return fma_(a, bc<NL>(b), c); }
template <int NL>
__device__ __forceinline__ Vf<NL> fma_(const Vf<NL> &a, float b, float c) { return fma_(a, bc<NL>(b), bc<NL>(c)); }
template <int NL>
__device__ __forceinline__ Vf<NL> rcp_(const Vf<NL> &a) {
  Vf<NL> r;
#pragma unroll
  for (int l = 0; l < NL; ++l) r[l] = rcp_(a[l]);
  return r;
}
template <int NL>
__device__ __forceinline__ Vf<NL> rsqrt_(const Vf<NL> &a) {
  Vf<NL> r;
#pragma unroll
  for (int l = 0; l < NL; ++l) r[l] = rsqrt_(a[l]);
  return r;
}
template <int NL>
__device__ __forceinline__ Vf<NL> sqrt_(const Vf<NL> &a) {
  Vf<NL> r;
#pragma unroll
  for (int l = 0; l < NL; ++l) r[l] = sqrtf(a[l]);
  return r;
}
template <int NL>
__device__ __forceinline__ Vf<NL> dot3_(const Vf<NL> a[3], const Vf<NL> b[3]) {
  return fma_(a[0], b[0], fma_(a[1], b[1], mul_(a[2], b[2])));
}
// floor through the sum with 1.5 2^23 rounded down: the integer sits in its low bits
constexpr float FLOOR_MAGIC = 12582912.0f;
constexpr int FLOOR_BITS = 0x4B400000;
template <int NL>
__device__ __forceinline__ Vf<NL> floor_(const Vf<NL> &t, int k[NL]) {
  const Vf<NL> m = add_rd(t, bc<NL>(FLOOR_MAGIC));
#pragma unroll
  for (int l = 0; l < NL; ++l) k[l] = __float_as_int(m[l]) - FLOOR_BITS;
  return add_(m, -FLOOR_MAGIC);
}

// ---- field and deposit accessors --------------------------------------------------
// The six components sit in four arrays: E_r and B_th share their staggered
// point, and so do E_th and B_r, so each of those pairs is one 8-byte load and
// one packed interpolation.
template <int WJ, int WN>
struct SmemAcc {  // window accessors (shared memory)
  using Index = int;
  const float2 *fa, *fb;    // (E_r, B_th), (E_th, B_r)
  const float *fc, *fd;     // E_ph, B_ph
  int *hi;                  // 3 * WN : sums of the high parts
  int *lo;                  // 3 * WN : sums of the low parts
  const float *rn;          // radius table of the window's rows
  const float2 *tn;         // (sin, cos) of the node angles of the window's columns
  int wi0, wj0;
  static __device__ __forceinline__ int stride() { return WJ; }
  __device__ __forceinline__ int index(int i, int j) const { return (i - wi0) * WJ + (j - wj0); }
  __device__ __forceinline__ float2 a(int o) const { return fa[o]; }
  __device__ __forceinline__ float2 b(int o) const { return fb[o]; }
  __device__ __forceinline__ float c(int o) const { return fc[o]; }
  __device__ __forceinline__ float d(int o) const { return fd[o]; }
  __device__ __forceinline__ float rad(int i) const { return rn[i - wi0]; }
  __device__ __forceinline__ float2 ang(int j) const { return tn[j - wj0]; }
  // unconditional: a test for zero terms would branch around every atomic,
  // which costs more than adding the rare zero
  __device__ __forceinline__ void add(int k, int o, int h, int l) const {
    atomicAdd(&hi[k * WN + o], h);
    atomicAdd(&lo[k * WN + o], l);
  }
};

struct GlobAcc {  // global-memory accessors (particles outside the window)
  using Index = size_t;
  const Args32 *A;
  __device__ __forceinline__ size_t stride() const { return (size_t)A->LD; }
  __device__ __forceinline__ size_t index(int i, int j) const { return pidx(*A, i, j); }
  __device__ __forceinline__ float2 a(size_t o) const { return make_float2(A->f[ER][o], A->f[BTH][o]); }
  __device__ __forceinline__ float2 b(size_t o) const { return make_float2(A->f[ETH][o], A->f[BR][o]); }
  __device__ __forceinline__ float c(size_t o) const { return A->f[EPH][o]; }
  __device__ __forceinline__ float d(size_t o) const { return A->f[BPH][o]; }
  __device__ __forceinline__ float rad(int i) const { return A->ir_n[i + A->PI]; }
  __device__ __forceinline__ float2 ang(int j) const { return A->th_n[j + A->PJ]; }
  __device__ __forceinline__ void add(int k, size_t o, int h, int l) const {
    const long long v = ((long long)h << SPLIT) + (long long)l;
    if (v) atomicAdd(reinterpret_cast<unsigned long long *>(A->acc[k] + o), (unsigned long long)v);
  }
};

// Fixed-point split of flux terms cs (in quanta, |cs| <= 2^36) into integers
// h, l with h 2^SPLIT + l = rint(cs), |h| <= 2^18, |l| <= 2^17.  Rounding to
// an integer by adding 1.5 * 2^23 is exact for |x| < 2^22; the subtraction
// cs - h 2^SPLIT is exact (Sterbenz).  Only FP32 adds and integer ops, no
// 64-bit conversions.  The term comes negated (ncs = -cs): see Vf.
template <int NL>
__device__ __forceinline__ void split_fix(const Vf<NL> &ncs, int h[NL], int l[NL]) {
  constexpr float MAGIC = 12582912.0f, MAGIC_H = 3298534883328.0f;  // 1.5 2^23, 1.5 2^41 (ulp 2^SPLIT)
  const Vf<NL> hm = fma_(ncs, -1.f, MAGIC_H);                        // cs rounded to a multiple of 2^18
  const Vf<NL> lm = add_(sub_(fma_(hm, -1.f, MAGIC_H), ncs), MAGIC);  // exact differences
#pragma unroll
  for (int q = 0; q < NL; ++q) {
    h[q] = __float_as_int(hm[q]) - 0x54400000;
    l[q] = __float_as_int(lm[q]) - 0x4B400000;
  }
}

template <int NL, class W>
__device__ __forceinline__ void deposit(const W &w, int k, const typename W::Index o[NL], typename W::Index off,
                                        const Vf<NL> &ncs) {
  int h[NL], l[NL];
  split_fix<NL>(ncs, h, l);
#pragma unroll
  for (int q = 0; q < NL; ++q) w.add(k, o[q] + off, h[q], l[q]);
}

// Villasenor-Buneman fluxes of straight paths p -> q inside the cells at o
// (local coordinates in [0, 1], Eq. Jcons, Sec. 3.3); nscale: minus the charge
// in flux units
template <int NL, class W>
__device__ __forceinline__ void vb_seg(const W &w, const Vf<NL> &nscale, const typename W::Index o[NL], const Vf<NL> &p1,
                                       const Vf<NL> &p2, const Vf<NL> &q1, const Vf<NL> &q2) {
  const Vf<NL> m1 = mul_(add_(p1, q1), 0.5f), m2 = mul_(add_(p2, q2), 0.5f);
  const Vf<NL> a = mul_(nscale, sub_(q1, p1)), b = mul_(nscale, sub_(q2, p2));
  const Vf<NL> n1 = fma_(m1, -1.f, 1.f), n2 = fma_(m2, -1.f, 1.f);
  const typename W::Index S = w.stride();
  deposit<NL>(w, 0, o, 0, mul_(a, n2));
  deposit<NL>(w, 0, o, 1, mul_(a, m2));
  deposit<NL>(w, 1, o, 0, mul_(b, n1));
  deposit<NL>(w, 1, o, S, mul_(b, m1));
}

__device__ __forceinline__ float clamp01(float v) { return fminf(fmaxf(v, 0.f), 1.f); }

// The path of a particle that crosses a grid line in x (kx = +-1), in y or in
// both: (dx, dy) in the cell at o to (nx, ny) in the cell (kx, ky) from it,
// split where it crosses the lines in the order it meets them.
template <class W>
__device__ __forceinline__ void vb_path(const W &w, float nscale, typename W::Index o, float dx, float dy, float nx,
                                        float ny, int kx, int ky) {
  using I = typename W::Index;
  const I S = w.stride();
  const float Xo = kx > 0 ? 1.f : 0.f, Xn = 1.f - Xo;  // crossed x line in the old / new x frame
  const float Yo = ky > 0 ? 1.f : 0.f, Yn = 1.f - Yo;
  const float Dxs = __fadd_rn(__fsub_rn(nx, dx), (float)kx), Dys = __fadd_rn(__fsub_rn(ny, dy), (float)ky);
  // crossing parameters: any point on the crossed grid line keeps charge
  // conservation exact, so an approximate reciprocal is enough here
  const float sx = kx ? __fmul_rn(__fsub_rn(Xo, dx), rcp_(Dxs)) : 2.f;
  const float sy = ky ? __fmul_rn(__fsub_rn(Yo, dy), rcp_(Dys)) : 2.f;
  const bool xfirst = sx <= sy;
  // first crossing point, in the frame of the cell the path leaves
  const float c1x = xfirst ? Xo : clamp01(__fmaf_rn(sy, Dxs, dx)), c1y = xfirst ? clamp01(__fmaf_rn(sx, Dys, dy)) : Yo;
  using V = Vf<1>;
  const V s{{nscale}}, ex{{nx}}, ey{{ny}};
  V px{{dx}}, py{{dy}};
  I c[1] = {o};
  vb_seg<1>(w, s, c, px, py, V{{c1x}}, V{{c1y}});
  // cell of the middle segment and the entry point there
  px[0] = xfirst ? Xn : c1x;
  py[0] = xfirst ? c1y : Yn;
  c[0] = o + (xfirst ? (kx > 0 ? S : (I)0 - S) : (I)ky);
  if (kx && ky) {
    // second crossing point, in the frame of the middle cell
    const float c2x = xfirst ? clamp01(__fmaf_rn(__fsub_rn(sy, 1.f), Dxs, nx)) : Xo;
    const float c2y = xfirst ? Yo : clamp01(__fmaf_rn(__fsub_rn(sx, 1.f), Dys, ny));
    vb_seg<1>(w, s, c, px, py, V{{c2x}}, V{{c2y}});
    px[0] = xfirst ? c2x : Xn;
    py[0] = xfirst ? Yn : c2y;
    c[0] = o + (kx > 0 ? S : (I)0 - S) + (I)ky;
  }
  vb_seg<1>(w, s, c, px, py, ex, ey);
}

// exp, log1p, arcsine and arctangent for the small arguments of a single step:
// truncated Taylor series (relative truncation below 2^-28 at the bounds that
// pic_ctx::small_steps states), otherwise the library functions
template <int NL>
__device__ __forceinline__ Vf<NL> exp_series(const Vf<NL> &y) {
  Vf<NL> p = fma_(y, 0.008333334f, 0.041666668f);
  p = fma_(y, p, 0.16666667f);
  p = fma_(y, p, 0.5f);
  p = fma_(y, p, 1.f);
  return fma_(y, p, 1.f);
}
template <int NL>
__device__ __forceinline__ Vf<NL> log1p_series(const Vf<NL> &s) {
  Vf<NL> p = fma_(s, -0.16666667f, 0.2f);
  p = fma_(s, p, -0.25f);
  p = fma_(s, p, 0.33333334f);
  p = fma_(s, p, -0.5f);
  p = fma_(s, p, 1.f);
  return mul_(s, p);
}
// |t| < 1/4
template <int NL>
__device__ __forceinline__ Vf<NL> asin_series(const Vf<NL> &t) {
  const Vf<NL> z = mul_(t, t);
  Vf<NL> p = fma_(z, 0.022372159f, 0.030381944f);
  p = fma_(z, p, 0.044642857f);
  p = fma_(z, p, 0.075f);
  p = fma_(z, p, 0.16666667f);
  return fma_(mul_(t, z), p, t);
}
// arcsine of the meridional turn, |t| <= 1/40
template <int NL>
__device__ __forceinline__ Vf<NL> asin_small(const Vf<NL> &t, const Vf<NL> &z) {
  return fma_(mul_(t, z), fma_(z, 0.075f, 0.16666667f), t);
}
// cos - 1 from the sine of that turn: sqrt(1 - z) - 1
template <int NL>
__device__ __forceinline__ Vf<NL> cosm1_small(const Vf<NL> &z) {
  return mul_(z, fma_(z, fma_(z, -0.0625f, -0.125f), -0.5f));
}
// (1 + s)^-1/2 - 1 for the relative displacement of a step, |s| <= 0.052
template <int NL>
__device__ __forceinline__ Vf<NL> inv_sqrt1p(const Vf<NL> &s) {
  Vf<NL> p = fma_(s, 0.22558594f, -0.24609375f);
  p = fma_(s, p, 0.2734375f);
  p = fma_(s, p, -0.3125f);
  p = fma_(s, p, 0.375f);
  p = fma_(s, p, -0.5f);
  return fma_(s, p, 1.f);
}
// sin x and cos x - 1 of a small angle: x (1 - x^2/6 + x^4/120) and
// -x^2/2 (1 - x^2/12 + x^4/360), relative truncation below x^6/5040 (under
// 2^-28 for |x| < 0.16)
template <int NL>
__device__ __forceinline__ void sin_cosm1_series(const Vf<NL> &x, Vf<NL> &s, Vf<NL> &cm1) {
  const Vf<NL> x2 = mul_(x, x);
  s = mul_(x, fma_(x2, fma_(x2, 0.008333334f, -0.16666667f), 1.f));
  cm1 = mul_(x2, fma_(x2, fma_(x2, -0.0013888889f, 0.041666668f), -0.5f));
}
// atan2(y, x) with R = hypot(x, y), in explicitly rounded operations: three
// halvings of the angle (tan(a/2) = sin a / (1 + cos a)) bring the tangent
// below 1/5, where the series to t^11 truncates below 2^-28
__device__ __forceinline__ float azimuth(float y, float x, float R) {
  float t = __fmul_rn(fabsf(y), rcp_(__fadd_rn(__fadd_rn(R, fabsf(x)), 1e-30f)));  // tan of half the angle from the x axis
#pragma unroll
  for (int k = 0; k < 2; ++k) t = __fmul_rn(t, rcp_(__fadd_rn(1.f, sqrtf(__fmaf_rn(t, t, 1.f)))));
  const float z = __fmul_rn(t, t);
  float p = __fmaf_rn(z, -0.090909092f, 0.11111111f);
  p = __fmaf_rn(z, p, -0.14285715f);
  p = __fmaf_rn(z, p, 0.2f);
  p = __fmaf_rn(z, p, -0.33333334f);
  const float a = __fmul_rn(8.f, __fmaf_rn(__fmul_rn(t, z), p, t));
  // beyond pi/2 from the other side of the axis, pi as two FP32 numbers
  const float b = x < 0.f ? __fadd_rn(3.1415927f, -__fadd_rn(a, 8.7422777e-8f)) : a;
  return copysignf(b, y);
}
__device__ __forceinline__ float log1p_small(float s) {
  return fabsf(s) < 0.03125f ? log1p_series(Vf<1>{{s}})[0] : log1pf(s);
}
__device__ __forceinline__ float exp_small(float y) { return fabsf(y) < 0.03125f ? exp_series(Vf<1>{{y}})[0] : expf(y); }

// ---- momentum in increments ----------------------------------------------
// The FP32 step computes each change of the momentum -- the push, then the
// rotation into the particle's new local frame -- as an increment du whose
// rounding errors are relative to |du|, not to |u|: for a particle turning by
// a small angle per step they are that much smaller, and the step adds to u
// only the rounding of the one sum u + du that stores it.

// Vay (2008) push, Sec. 2, as u' - u: with a = u + (q dt/m) E + v x tau and
// t = tau / gamma', u' = s (a + (a.t) t + a x t), s = 1 / (1 + t^2), i.e.
// u' - a = s ((a.t) t + a x t - t^2 a).
template <int NL>
__device__ __forceinline__ void vay_delta(const Vf<NL> &qmdt, const Vf<NL> E[3], const Vf<NL> B[3], const Vf<NL> u[3],
                                          Vf<NL> du[3]) {
  using V = Vf<NL>;
  const V h = mul_(qmdt, 0.5f);
  const V ig0 = rsqrt_(add_(dot3_(u, u), 1.f)), nig0 = mul_(ig0, -1.f);
  const V tau[3] = {mul_(h, B[0]), mul_(h, B[1]), mul_(h, B[2])};
  const V v[3] = {mul_(u[0], ig0), mul_(u[1], ig0), mul_(u[2], ig0)};
  const V nv[3] = {mul_(u[0], nig0), mul_(u[1], nig0), mul_(u[2], nig0)};
  V d[3], a[3], na[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {  // (q dt / m) E + v x tau
    const int i = (k + 1) % 3, j = (k + 2) % 3;
    d[k] = fma_(v[i], tau[j], fma_(nv[j], tau[i], mul_(qmdt, E[k])));
    a[k] = add_(u[k], d[k]);
    na[k] = mul_(a[k], -1.f);
  }
  const V tau2 = dot3_(tau, tau), ustar = dot3_(a, tau);
  const V sigma = sub_(add_(dot3_(a, a), 1.f), tau2);
  const V disc = fma_(sigma, sigma, mul_(fma_(ustar, ustar, tau2), 4.f));
  const V ig = rsqrt_(mul_(add_(sigma, sqrt_(disc)), 0.5f));
  const V t[3] = {mul_(tau[0], ig), mul_(tau[1], ig), mul_(tau[2], ig)};
  const V tt = dot3_(t, t), sc = rcp_(add_(tt, 1.f)), at = mul_(ustar, ig);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = (k + 1) % 3, j = (k + 2) % 3;
    du[k] = fma_(sc, fma_(tt, na[k], fma_(at, t[k], fma_(a[i], t[j], mul_(na[j], t[i])))), d[k]);
  }
}

// Boris (1970) push, Sec. 2, as u' - u: half electric kick h E, rotation
// u- -> u+ = u- + (u- + u- x t) x s, half kick; u' - u = 2 h E + (u- + u- x t) x s.
template <int NL>
__device__ __forceinline__ void boris_delta(const Vf<NL> &qmdt, const Vf<NL> E[3], const Vf<NL> B[3],
                                            const Vf<NL> u[3], Vf<NL> du[3]) {
  using V = Vf<NL>;
  const V h = mul_(qmdt, 0.5f);
  V um[3], n[3], p[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    um[k] = fma_(h, E[k], u[k]);
    n[k] = mul_(um[k], -1.f);
  }
  const V hi = mul_(h, rsqrt_(add_(dot3_(um, um), 1.f)));
  const V t[3] = {mul_(hi, B[0]), mul_(hi, B[1]), mul_(hi, B[2])};
  const V f = mul_(rcp_(add_(dot3_(t, t), 1.f)), 2.f);
  const V s[3] = {mul_(f, t[0]), mul_(f, t[1]), mul_(f, t[2])};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = (k + 1) % 3, j = (k + 2) % 3;
    p[k] = add_(um[k], fma_(um[i], t[j], mul_(n[j], t[i])));
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = (k + 1) % 3, j = (k + 2) % 3;
    du[k] = fma_(p[i], s[j], fma_(mul_(p[j], -1.f), s[i], mul_(qmdt, E[k])));
  }
}

// bilinear interpolation, two lines along i and one along j: both components
// of a float2 array, or one array for the NL particles
template <class W>
__device__ __forceinline__ float2 lerp2(const W &, float2 f00, float2 f10, float2 f01, float2 f11, float a, float b) {
  const Vf<2> va = bc<2>(a);
  const Vf<2> v0 = fma_(va, sub_(up(f10), up(f00)), up(f00)), v1 = fma_(va, sub_(up(f11), up(f01)), up(f01));
  return pk(fma_(bc<2>(b), sub_(v1, v0), v0));
}
template <int NL>
__device__ __forceinline__ Vf<NL> lerp1(const Vf<NL> f[4], const Vf<NL> &a, const Vf<NL> &b) {
  const Vf<NL> v0 = fma_(a, sub_(f[1], f[0]), f[0]), v1 = fma_(a, sub_(f[3], f[2]), f[2]);
  return fma_(b, sub_(v1, v0), v0);
}

// One step of the NL particles of a thread.  In: their cells and state (k0:
// the first one's slot, read only for an axis-crossing tie); on[l]: the particle exists.  Out:
// the new state, ok[l]: it stays in the simulation.  A path that crosses no
// grid line is deposited here; for the others `cross(l, o, ...)` is called.
template <int SPEC, int NL, class W, class Cross>
__device__ __forceinline__ void step32(const Args32 &A, const W &w, float fs, int64_t k0, const bool on[NL],
                                       uint32_t cell[NL], Vf<NL> &dx, Vf<NL> &dy, Vf<NL> &ur, Vf<NL> &ut, Vf<NL> &up_,
                                       const Vf<NL> &qw, bool ok[NL], const Cross &cross) {
  using V = Vf<NL>;
  using I = typename W::Index;
  const Flags<SPEC> F(A);
  constexpr bool series = SPEC != SPEC_GENERIC;  // arguments below the series' bounds: no fallback
  int ci[NL], cj[NL];
  I o[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    ci[l] = (int)(cell[l] >> 16) - CELL_BIAS;
    cj[l] = (int)(cell[l] & 0xffffu);
    o[l] = w.index(ci[l], cj[l]);
  }
  // ---- geometry of the particle's position (Sec. 3.2) -----------------------
  // 1 / r (the table holds 1 / f_r(i) on a log grid, f_r(i) on a linear one)
  V rt, ir;
#pragma unroll
  for (int l = 0; l < NL; ++l) rt[l] = w.rad(ci[l]);
  if (F.r_log) {
    const V y = mul_(dx, -A.dxi);
    if (series) {
      ir = mul_(rt, exp_series(y));
    } else {
#pragma unroll
      for (int l = 0; l < NL; ++l) ir[l] = __fmul_rn(rt[l], exp_small(y[l]));
    }
  } else {
    ir = rcp_(fma_(dx, A.dxi, rt));
  }
  // sin and cos of theta from the distance to the nearer pole, which both
  // offsets resolve to FP32 relative precision (1 - x2/nth would cancel)
  V st, ct;
  if (F.th_ea) {  // cos th = 1 - 2 x2/nth, sin th = 2 sqrt(x2 (nth - x2))/nth
    V fj;
#pragma unroll
    for (int l = 0; l < NL; ++l) fj[l] = __int_as_float(0x4B000000 + cj[l]);  // 2^23 + cj
    fj = add_(fj, -8388608.f);
    const V x2 = add_(fj, dy), rest = sub_(fma_(fj, -1.f, A.nth_f), dy);
    ct = mul_(sub_(rest, x2), A.inv_nth);
    st = mul_(sqrt_(mul_(x2, rest)), 2.f * A.inv_nth);
  } else if (series) {
    // linear map: the node angle's sine and cosine from the column table,
    // turned by the offset's angle (at most pi / nth, nth >= 32 on the
    // specialised grids: short series).  The node taken is the one on the
    // pole's side of the particle in its hemisphere, so both terms of sin th
    // have one sign and sin th keeps FP32 relative precision up to the poles.
    V b, n0, n1, sb, cb1;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const bool north = 2 * cj[l] < A.nth;
      const float2 n = w.ang(north ? cj[l] : cj[l] + 1);
      n0[l] = n.x;
      n1[l] = n.y;
      b[l] = north ? dy[l] : __fadd_rn(dy[l], -1.f);
    }
    sin_cosm1_series(mul_(b, A.pi_nth), sb, cb1);
    st = fma_(n1, sb, fma_(n0, cb1, n0));              // sin th_n cos b + cos th_n sin b
    ct = sub_(fma_(n1, cb1, n1), mul_(n0, sb));        // cos th_n cos b - sin th_n sin b
  } else {
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const float x2 = __fadd_rn((float)cj[l], dy[l]), rest = __fsub_rn((float)(A.nth - cj[l]), dy[l]);
      sincospif((x2 <= rest ? x2 : rest) * A.inv_nth, &st[l], &ct[l]);
      if (x2 > rest) ct[l] = -ct[l];
    }
  }
  // ---- gather + push (ballistic inside the outer conductor) -----------------
  V E[3], B[3], qmdt;
  {
    V ah, bh, f0[4], f1[4];
    const I S = w.stride();
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const bool hx = dx[l] >= 0.5f, hy = dy[l] >= 0.5f;
      const I oi = hx ? o[l] : o[l] - S, oj = hy ? o[l] : o[l] - 1, oij = hy ? oi : oi - 1;
      ah[l] = __fadd_rn(dx[l], hx ? -0.5f : 0.5f);
      bh[l] = __fadd_rn(dy[l], hy ? -0.5f : 0.5f);
      const float2 a = lerp2(w, w.a(oi), w.a(oi + S), w.a(oi + 1), w.a(oi + S + 1), ah[l], dy[l]);
      const float2 b = lerp2(w, w.b(oj), w.b(oj + S), w.b(oj + 1), w.b(oj + S + 1), dx[l], bh[l]);
      E[0][l] = a.x; B[1][l] = a.y;
      E[1][l] = b.x; B[0][l] = b.y;
      f0[0][l] = w.c(o[l]); f0[1][l] = w.c(o[l] + S); f0[2][l] = w.c(o[l] + 1); f0[3][l] = w.c(o[l] + S + 1);
      f1[0][l] = w.d(oij); f1[1][l] = w.d(oij + S); f1[2][l] = w.d(oij + 1); f1[3][l] = w.d(oij + S + 1);
      qmdt[l] = __int_as_float(__float_as_int(A.qmdt) ^ (__float_as_int(qw[l]) & 0x80000000));
    }
    E[2] = lerp1<NL>(f0, dx, dy);
    B[2] = lerp1<NL>(f1, ah, bh);
    bool edge = false;
#pragma unroll
    for (int l = 0; l < NL; ++l) edge |= (unsigned)ci[l] >= (unsigned)A.nr;
    if (edge) {
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        if (ci[l] < 0)  // plasma field only outside the inner conductor
          for (int q = 0; q < 3; ++q) { E[q][l] = 0.f; B[q][l] = 0.f; }
        if (ci[l] >= A.nr) qmdt[l] = 0.f;  // no field, no push
      }
    }
  }
  if (F.vacuum == PIC_VAC_MONOPOLE || F.vacuum == PIC_VAC_MONOPOLE_ROTATOR) {  // B_r = b0 (r0/r)^2, b0 to ~1e-14
    const V q = mul_(ir, A.r_min), q2 = mul_(q, q);
    B[0] = add_(B[0], fma_(q2, A.b0, mul_(q2, A.b0_lo)));
    if (F.vacuum == PIC_VAC_MONOPOLE_ROTATOR) {
      V w1 = mul_(mul_(q, q2), A.nbrw);  // -b0 r0^4 Omega / r^3
      V w0 = mul_(w1, 2.f);
#pragma unroll
      for (int l = 0; l < NL; ++l)
        if (ci[l] < 0) {  // inside the star: -b0 r0^2 Omega / r
          w0[l] = 0.f;
          w1[l] = __fmul_rn(q[l], A.nbrw);
        }
      E[0] = fma_(w0, ct, E[0]);
      E[1] = fma_(w1, st, E[1]);
    }
  } else if (F.vacuum != PIC_VAC_NONE) {
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      float e[3], b[3];
      const Vac<float> Vc{F.vacuum, A.b0, A.r_min, A.omega_t};
      vacuum_field<float>(Vc, rcp_(ir[l]), st[l], ct[l], ci[l] < 0, e, b);
      for (int q = 0; q < 3; ++q) {
        E[q][l] = __fadd_rn(E[q][l], e[q]);
        B[q][l] = __fadd_rn(B[q][l], b[q]);
      }
    }
  }
  const V u[3] = {ur, ut, up_};
  V du[3];  // momentum change of the step: push, then frame rotation
  // local (r, th, ph) is a right-handed orthonormal frame: the Cartesian push
  // formulas apply to its components unchanged
  if (F.pusher == PIC_BORIS) boris_delta<NL>(qmdt, E, B, u, du);
  else vay_delta<NL>(qmdt, E, B, u, du);
  // u^{n+1/2} in FP32, for the move
  const V p[3] = {add_(u[0], du[0]), add_(u[1], du[1]), add_(u[2], du[2])};
  // ---- move in the local frame, in units of r (Sec. 3.3) ----------------------
  const V g = mul_(rsqrt_(add_(dot3_(p, p), 1.f)), ir), gdt = fma_(g, A.dt, mul_(g, A.dt_lo));
  const V a = mul_(p[0], gdt), b = mul_(p[1], gdt), c = mul_(p[2], gdt);
  const V c2 = mul_(c, c), bc2 = fma_(b, b, c2);
  const V s = fma_(a, fma_(p[0], gdt, bc<NL>(2.f)), bc2);  // (r'/r)^2 - 1
  V D1, irn;                               // radial increment in cells; r / r'
  if (series) {
    irn = inv_sqrt1p(s);
    const V L = log1p_series(s);
    D1 = fma_(L, A.hinv_dxi, mul_(L, A.hinv_dxi_lo));
  } else {
    irn = rsqrt_(add_(s, 1.f));
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const float L = F.r_log ? 0.5f * log1p_small(s[l])
                              : __fmul_rn(__fmul_rn(rcp_(ir[l]), s[l]), rcp_(1.f + sqrtf(1.f + s[l])));
      D1[l] = __fmaf_rn(L, A.inv_dxi, __fmul_rn(L, A.inv_dxi_lo));
    }
  }
  // displaced point, (R, z) before rotating back; kap = R' - Px
  const V Px = fma_(a, st, fma_(b, ct, st)), Pz = sub_(fma_(a, ct, ct), mul_(b, st));
  const V R2 = fma_(Px, Px, fma_(c, c, 2e-38f));  // (the constant, a normal number: no 0 / 0 on the axis)
  const V iRn = rsqrt_(R2), Rn = mul_(R2, iRn);
  V kap = mul_(c2, rcp_(fma_(R2, iRn, Px)));
  const V sph = mul_(c, iRn);        // sine of the azimuth swept
  V phi = asin_series(sph);
  {
    bool far = false;  // across the axis, on it, or turning by a large azimuth next to it
#pragma unroll
    for (int l = 0; l < NL; ++l) far |= !(Px[l] > 1e-17f && fabsf(sph[l]) < 0.25f);
    if (far) {
#pragma unroll
      for (int l = 0; l < NL; ++l)
        if (on[l] && !(Px[l] > 1e-17f && fabsf(sph[l]) < 0.25f)) {
          if (!(Px[l] > 0.f)) kap[l] = Px[l] < 0.f ? __fsub_rn(Rn[l], Px[l]) : (R2[l] > 2.2e-38f ? Rn[l] : 0.f);
          float x = Px[l], y = c[l], R = Rn[l];
          if (R2[l] < 1e-20f) {  // lengths whose squares lose bits: 2^60 times them
            x = __fmul_rn(x, 0x1p60f);
            y = __fmul_rn(y, 0x1p60f);
            R = sqrtf(__fmaf_rn(x, x, __fmul_rn(y, y)));
          }
          phi[l] = azimuth(y, x, R);
          if (Px[l] < 0.f && p[2][l] * p[2][l] <= (float)(AXIS_TIE * AXIS_TIE) *
                                                       (p[0][l] * p[0][l] + p[1][l] * p[1][l] + p[2][l] * p[2][l]))
            phi[l] = axis_tie(A.ties, A.ids[k0 + l], phi[l]);  // rare: see AxisTies
        }
    }
  }
  // meridional turn: its sine (b + ct kap) r / r' and cosine - 1
  const V num = fma_(ct, kap, b), sd = mul_(num, irn);
  const V a1 = fma_(p[0], gdt, bc<NL>(1.f));  // 1 + a
  V D2, ty, cd1;                              // meridional increment in cells, dy + D2
  if (series) {
    const V z = mul_(sd, sd);
    cd1 = cosm1_small(z);
    if (!F.th_ea) {
      const V dth = asin_small(sd, z);
      D2 = fma_(dth, A.k2_hi, mul_(dth, A.k2_lo));
    }
  } else {
    const V den = fma_(st, kap, a1);
    cd1 = mul_(mul_(mul_(sd, sd), -1.f), rcp_(fma_(den, irn, bc<NL>(1.f))));
    if (!F.th_ea) {
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const float x = den[l], y = num[l];
        float dth;
        if (x > 0.f && fabsf(y) < __fmul_rn(0.03125f, x)) {
          const float t = __fmul_rn(y, rcp_(x)), t2 = __fmul_rn(t, t);
          const float q = __fmaf_rn(t2, __fmaf_rn(t2, -0.14285715f, 0.2f), -0.33333334f);
          dth = __fmaf_rn(__fmul_rn(t, t2), q, t);
        } else {
          dth = azimuth(y, x, sqrtf(__fmaf_rn(x, x, __fmul_rn(y, y))));
        }
        D2[l] = __fmaf_rn(dth, A.k2_hi, __fmul_rn(dth, A.k2_lo));
      }
    }
  }
  if (F.th_ea) {
    // nth / 2 (cos th - cos th'): r'/r - 1 - a = (b^2 + c^2) / (1 + a + r'/r), nothing cancels
    const V rr = fma_(s, irn, irn);  // r' / r
    const V T = mul_(fma_(ct, mul_(bc2, rcp_(add_(a1, rr))), mul_(b, st)), irn);
    D2 = mul_(T, A.hnth);
    ty = fma_(T, A.hnth, dy);
  } else {
    ty = add_(dy, D2);
  }
  // momentum into the new local frame, as an increment: Cartesian at phi = 0
  // (x along R), rotated back about z by -phi' (cos phi' - 1 = -kap / R',
  // sin phi' = Dp / R'), then into (r', th') at th' = th + dth:
  //   u_r' = u_r cos dth + u_th sin dth + dx st',  u_th' = -u_r sin dth + u_th cos dth + dx ct',
  //   u_ph' = u_ph + dy,  with (dx, dy) the change of (u_x, u_ph) under the azimuthal rotation
  {
    const V ux = fma_(p[0], st, mul_(p[1], ct));
    const V niRn = mul_(iRn, -1.f), cm1 = mul_(kap, niRn), nsph = mul_(c, niRn), nsd = mul_(sd, -1.f);
    const V dxr = fma_(ux, cm1, mul_(sph, p[2])), dyr = fma_(p[2], cm1, mul_(nsph, ux));
    const V stn = mul_(Rn, irn), ctn = mul_(Pz, irn);
    du[0] = add_(du[0], fma_(p[0], cd1, fma_(p[1], sd, mul_(dxr, stn))));
    du[1] = add_(du[1], fma_(p[1], cd1, fma_(p[0], nsd, mul_(dxr, ctn))));
    du[2] = add_(du[2], dyr);
  }
  const V nur = add_(u[0], du[0]), nut = add_(u[1], du[1]), nup = add_(u[2], du[2]);
  // new cell and offsets (carries are exact integers)
  int kx[NL], ky[NL];
  const V tx = add_(dx, D1);
  V kfx = floor_<NL>(tx, kx), kfy = floor_<NL>(ty, ky);
  V nx = sub_(tx, kfx), ny = sub_(ty, kfy);
  {
    const V sum = add_(add_(nx, ny), add_(add_(nur, nut), nup));  // finite when all are
    bool odd = false;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      ok[l] = on[l];
      odd |= !(fmaxf(fmaxf(fabsf(D1[l]), fabsf(D2[l])), fmaxf(nx[l], ny[l])) < 1.f) | !(fabsf(sum[l]) < 1e38f) |
             ((unsigned)(cj[l] + ky[l]) >= (unsigned)A.nth);
    }
    if (odd) {  // rounding onto a line or past the axis, or an error
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        if (nx[l] >= 1.f) { nx[l] = 0.f; ++kx[l]; }
        if (ny[l] >= 1.f) { ny[l] = 0.f; ++ky[l]; }
        if (cj[l] + ky[l] < 0) { ky[l] = -cj[l]; ny[l] = 0.f; }                                  // below the axis
        if (cj[l] + ky[l] > A.nth - 1) { ky[l] = A.nth - 1 - cj[l]; ny[l] = 1.f; }              // past the south axis
        const bool fin = isfinite(nx[l]) && isfinite(ny[l]) && isfinite(nur[l]) && isfinite(nut[l]) && isfinite(nup[l]);
        if (!fin || kx[l] < -1 || kx[l] > 1 || ky[l] < -1 || ky[l] > 1) {
          if (on[l]) atomicOr(A.err, (isfinite(nx[l]) && isfinite(nur[l])) ? ERR_COURANT : ERR_NAN);
          ok[l] = false;
          kx[l] = ky[l] = 0;
          nx[l] = dx[l];
          ny[l] = dy[l];
          phi[l] = 0.f;  // it deposits nothing
        }
        kfx[l] = (float)kx[l];
        kfy[l] = (float)ky[l];
      }
    }
  }
  // ---- Villasenor-Buneman deposit along the grid-coordinate path -----------
  const V nscale = mul_(qw, -fs);  // exact: fs is a power of two
  {
    V q1 = nx, q2 = ny;
#pragma unroll
    for (int l = 0; l < NL; ++l)
      if (kx[l] | ky[l]) {  // its path is deposited by cross(); here it has zero length
        q1[l] = dx[l];
        q2[l] = dy[l];
      }
    vb_seg<NL>(w, nscale, o, dx, dy, q1, q2);
    cross(nscale, o, dx, dy, nx, ny, kx, ky);
  }
  // azimuthal flux: charge crossing the meridional half-plane, qw dphi / 2 pi,
  // area weights at the midpoint of the grid path
  {
    int k1[NL], k2[NL];
    const V v = mul_(mul_(nscale, 0.15915494309189535f), phi);
    const V mx = mul_(add_(dx, add_(kfx, nx)), 0.5f), my = mul_(add_(dy, add_(kfy, ny)), 0.5f);
    const V wx = sub_(mx, floor_<NL>(mx, k1)), wy = sub_(my, floor_<NL>(my, k2));
    const V vx = mul_(v, wx), v0 = sub_(v, vx), v01 = mul_(v0, wy), v11 = mul_(vx, wy);
    const I S = w.stride();
    I oa[NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) oa[l] = o[l] + (I)k1[l] * S + (I)k2[l];
    deposit<NL>(w, 2, oa, 0, sub_(v0, v01));
    deposit<NL>(w, 2, oa, S, sub_(vx, v11));
    deposit<NL>(w, 2, oa, 1, v01);
    deposit<NL>(w, 2, oa, S + 1, v11);
  }
  // ---- new state; removal once the filtered shape is inside a conductor ---------
  const uint32_t lo = (uint32_t)(CELL_BIAS - (A.n_filt + 1)) << 16,
                 span = (uint32_t)(A.nr + 2 * (A.n_filt + 1)) << 16;
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    cell[l] += (uint32_t)(kx[l] * 65536 + ky[l]);
    ok[l] = ok[l] && cell[l] - lo < span;
  }
  dx = nx; dy = ny; ur = nur; ut = nut; up_ = nup;
}

// the rare path: one particle outside its tile's window (or not yet binned)
template <int SPEC>
__device__ __forceinline__ void step_global(const Args32 &A, const Parts32 &P, float fs, int64_t k, int &dead) {
  const float q = P.qw[k];
  if (q == 0.f) return;
  const GlobAcc w{&A};
  using V = Vf<1>;
  uint32_t cell[1] = {P.cell[k]};
  V dx{{P.dx[k]}}, dy{{P.dy[k]}}, ur{{P.ur[k]}}, ut{{P.ut[k]}}, up_{{P.up[k]}};
  const bool on[1] = {true};
  bool ok[1];
  step32<SPEC, 1>(A, w, fs, k, on, cell, dx, dy, ur, ut, up_, V{{q}}, ok,
                  [&](const V &nscale, const size_t *o, const V &x, const V &y, const V &nx, const V &ny, const int *kx,
                      const int *ky) {
                    if (kx[0] | ky[0]) vb_path(w, nscale[0], o[0], x[0], y[0], nx[0], ny[0], kx[0], ky[0]);
                  });
  if (!ok[0]) { P.qw[k] = 0.f; ++dead; return; }
  P.cell[k] = cell[0];
  P.dx[k] = dx[0]; P.dy[k] = dy[0];
  P.ur[k] = ur[0]; P.ut[k] = ut[0]; P.up[k] = up_[0];
}

// The two particles of a thread's next pass, loaded while it steps the present
// ones: one 8-byte load per array.
struct Pair {
  uint2 cell;
  float2 dx, dy, ur, ut, up, qw;
};
__device__ __forceinline__ Pair load_pair(const Parts32 &P, int64_t e) {
  Pair r;
  r.cell = *reinterpret_cast<const uint2 *>(P.cell + e);
  r.dx = *reinterpret_cast<const float2 *>(P.dx + e);
  r.dy = *reinterpret_cast<const float2 *>(P.dy + e);
  r.ur = *reinterpret_cast<const float2 *>(P.ur + e);
  r.ut = *reinterpret_cast<const float2 *>(P.ut + e);
  r.up = *reinterpret_cast<const float2 *>(P.up + e);
  r.qw = *reinterpret_cast<const float2 *>(P.qw + e);
  return r;
}

// One tile CTA (or one block of unbinned particles) of the FP32 step: block
// `blk` of the member whose arguments are A and P, its six field tensor maps
// at `maps` (kernel parameters, or global memory when GMAPS).
//
// Paths that cross a grid line take two or three Villasenor-Buneman segments,
// some 150 instructions; one such lane would make its whole warp run them (at
// 3 % of the particles crossing, six passes of ten).  Each warp queues them
// in shared memory instead and works the queue off 32 at a time.
template <int TI, int TJ, int SPEC, bool GMAPS>
__device__ __forceinline__ void tiles32_block(const Args32 &A, const Parts32 &P, const CUtensorMap *maps,
                                              unsigned blk) {
  using BX_ = Box<TI, TJ>;
  constexpr int WI = BX_::WI, WJ = BX_::WJ, WN = BX_::WN, WB = BX_::WB, SLOT = BX_::SLOT;
  __shared__ __align__(128) float sbuf[BX_::SF + BX_::U2];
  float2 *const sfa = reinterpret_cast<float2 *>(sbuf);        // WN each: the window, (E_r, B_th), (E_th, B_r),
  float2 *const sfb = sfa + WN;
  float *const sfc = sbuf + 4 * WN, *const sfd = sbuf + 5 * WN;  // E_ph, B_ph
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
    // the thread's first pair, on an even slot (a slot before b0 is masked)
    int64_t e = (b0 & ~(int64_t)1) + 2 * (int)threadIdx.x;
    Pair next;
    if (e < b1) next = load_pair(P, e);
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
    for (int q = threadIdx.x; q < WI; q += NTH) srn[q] = A.ir_n[wi0 + q + A.PI];
    if (SPEC != SPEC_GENERIC)
      for (int q = threadIdx.x; q < WJ; q += NTH) stn[q] = A.th_n[wj0 + q + A.PJ];
    __syncthreads();
    if (!sok) return;
    for (int q = threadIdx.x; q < WN; q += NTH) {
      const int g = q / WJ * WB + q % WJ + WOFF;
      sfa[q] = make_float2(stage[ER * SLOT + g], stage[BTH * SLOT + g]);
      sfb[q] = make_float2(stage[ETH * SLOT + g], stage[BR * SLOT + g]);
      sfc[q] = stage[EPH * SLOT + g];
      sfd[q] = stage[BPH * SLOT + g];
    }
    __syncthreads();  // the staging area becomes the accumulators
    for (int q = threadIdx.x; q < 3 * WN; q += NTH) { shi[q] = 0; slo[q] = 0; }
    __syncthreads();
    const SmemAcc<WJ, WN> w{sfa, sfb, sfc, sfd, shi, slo, srn, stn, wi0, wj0};
    const int lane = threadIdx.x & 31;
    float *const queue = sbuf + BX_::SF + 6 * WN + (threadIdx.x >> 5) * (6 * 64);  // 6 words x 64 entries
    int queued = 0;
    auto work_off = [&](int at) {  // the path of queue entry `at`
      const int code = __float_as_int(queue[5 * 64 + at]);
      vb_path(w, queue[4 * 64 + at], code & 0xffff, queue[at], queue[64 + at], queue[2 * 64 + at], queue[3 * 64 + at],
              ((code >> 16) & 3) - 1, ((code >> 18) & 3) - 1);
    };
    const int npass = (int)((b1 - (b0 & ~(int64_t)1) + NT - 1) / NT);
    for (int pass = 0; pass < npass; ++pass, e += NT) {
      if (e - 2 * lane >= b1) break;  // nothing left for this warp
      const Pair cur = next;
      if (e + NT < b1) next = load_pair(P, e + NT);
      using V = Vf<2>;
      uint32_t cell[2] = {cur.cell.x, cur.cell.y};
      V dx = up(cur.dx), dy = up(cur.dy), ur = up(cur.ur), ut = up(cur.ut), up_ = up(cur.up), qw = up(cur.qw);
      bool on[2], far[2], ok[2];
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        const bool have = e + l >= b0 && e + l < b1 && qw[l] != 0.f;
        const bool in = (cell[l] >> 16) - (uint32_t)(i0 - H + CELL_BIAS) < (uint32_t)(TI + 2 * H) &&
                        (cell[l] & 0xffffu) - (uint32_t)(j0 - H) < (uint32_t)(TJ + 2 * H);
        on[l] = have && in;
        far[l] = have && !in;
        if (!on[l]) {  // an idle lane steps a particle without charge at the tile's corner
          cell[l] = ((uint32_t)(i0 + CELL_BIAS) << 16) | (uint32_t)j0;
          dx[l] = dy[l] = 0.5f;
          ur[l] = ut[l] = up_[l] = qw[l] = 0.f;
        }
      }
      step32<SPEC, 2>(A, w, fs, e, on, cell, dx, dy, ur, ut, up_, qw, ok,
                      [&](const V &nscale, const int *o, const V &x, const V &y, const V &nx, const V &ny,
                          const int *kx, const int *ky) {
#pragma unroll
                        for (int l = 0; l < 2; ++l) {
                          const bool mine = on[l] && (kx[l] | ky[l]);
                          const unsigned m = __ballot_sync(0xffffffffu, mine);
                          if (!m) continue;
                          if (mine) {
                            const int at = queued + __popc(m & ((1u << lane) - 1u));
                            queue[at] = x[l];
                            queue[64 + at] = y[l];
                            queue[2 * 64 + at] = nx[l];
                            queue[3 * 64 + at] = ny[l];
                            queue[4 * 64 + at] = nscale[l];
                            queue[5 * 64 + at] = __int_as_float(o[l] | (kx[l] + 1) << 16 | (ky[l] + 1) << 18);
                          }
                          queued += __popc(m);
                          if (queued >= 32) {
                            __syncwarp();
                            queued -= 32;
                            work_off(queued + lane);
                            __syncwarp();
                          }
                        }
                      });
      if (ok[0] && ok[1]) {
        *reinterpret_cast<uint2 *>(P.cell + e) = make_uint2(cell[0], cell[1]);
        *reinterpret_cast<float2 *>(P.dx + e) = pk(dx);
        *reinterpret_cast<float2 *>(P.dy + e) = pk(dy);
        *reinterpret_cast<float2 *>(P.ur + e) = pk(ur);
        *reinterpret_cast<float2 *>(P.ut + e) = pk(ut);
        *reinterpret_cast<float2 *>(P.up + e) = pk(up_);
      } else {
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          const int64_t k = e + l;
          if (ok[l]) {
            P.cell[k] = cell[l];
            P.dx[k] = dx[l]; P.dy[k] = dy[l];
            P.ur[k] = ur[l]; P.ut[k] = ut[l]; P.up[k] = up_[l];
          } else if (on[l]) {
            P.qw[k] = 0.f;
            ++dead;
          } else if (far[l]) {  // drifted out of the window since the last sort
            step_global<SPEC>(A, P, fs, k, dead);
          }
        }
      }
    }
    __syncwarp();
    if (lane < queued) work_off(lane);
    if (dead) atomicAdd(&sdead, dead);
    __syncthreads();
    for (int q = threadIdx.x; q < WN; q += NTH) {
      const size_t o = pidx(A, wi0 + q / WJ, wj0 + q % WJ);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int hsum = shi[c * WN + q], lsum = slo[c * WN + q];
        if (sums_full(hsum, lsum, b1 - b0)) atomicOr(A.err, ERR_CAPACITY);
        const long long v = ((long long)hsum << SPLIT) + (long long)lsum;
        if (v) atomicAdd(reinterpret_cast<unsigned long long *>(A.acc[c] + o), (unsigned long long)v);
      }
    }
    if (threadIdx.x == 0 && sdead) add_ll(A.cnt + CNT_DELETED, sdead);
  } else {  // particles outside any bin (injected since the last sort)
    for (int r = 0; r < NT; r += NTH) {
      const int64_t k = A.sorted_end + (int64_t)(blk - A.nunits) * NT + r + threadIdx.x;
      if (k < A.n_used) step_global<SPEC>(A, P, fs, k, dead);
    }
    if (dead) add_ll(A.cnt + CNT_DELETED, dead);
  }
}

template <int TI, int TJ, int SPEC>
__global__ void __launch_bounds__(NTH, 4) k_tiles32(Args32 A, Parts32 P, const __grid_constant__ TileMaps maps) {
  follow();
  tiles32_block<TI, TJ, SPEC, false>(A, P, maps.m, blockIdx.x);
}

// the tile kernel over several members of an ensemble in one grid; see
// ens_tiles32 for what its launches do to each other
template <int TI, int TJ, int SPEC>
__global__ void __launch_bounds__(NTH, 4) k_ens_tiles32(const __grid_constant__ EnsTileBatch B) {
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
  if (shape == 1) launch_on(s, overlap, k_tiles32<8, 32, SPEC>, blocks, NTH, A, P, M);
  else if (shape == 2) launch_on(s, overlap, k_tiles32<32, 8, SPEC>, blocks, NTH, A, P, M);
  else launch_on(s, overlap, k_tiles32<16, 16, SPEC>, blocks, NTH, A, P, M);
}

template <int SPEC>
void launch_ens(int shape, unsigned blocks, cudaStream_t s, bool beside, const EnsTileBatch &B) {
  if (shape == 1) launch_on(s, beside, k_ens_tiles32<8, 32, SPEC>, blocks, NTH, B);
  else if (shape == 2) launch_on(s, beside, k_ens_tiles32<32, 8, SPEC>, blocks, NTH, B);
  else launch_on(s, beside, k_ens_tiles32<16, 16, SPEC>, blocks, NTH, B);
}

}  // namespace

void launch_two(int spec, int shape, unsigned blocks, cudaStream_t s, bool overlap, const Args32 &A, const Parts32 &P,
                const TileMaps &M) {
  if (spec == SPEC_MONOPOLE) launch<SPEC_MONOPOLE>(shape, blocks, s, overlap, A, P, M);
  else if (spec == SPEC_ROTATOR) launch<SPEC_ROTATOR>(shape, blocks, s, overlap, A, P, M);
  else launch<SPEC_GENERIC>(shape, blocks, s, overlap, A, P, M);
}

void launch_ens_two(int spec, int shape, unsigned blocks, cudaStream_t s, bool beside,
                    const EnsTileBatch &B) {
  if (spec == SPEC_MONOPOLE) launch_ens<SPEC_MONOPOLE>(shape, blocks, s, beside, B);
  else if (spec == SPEC_ROTATOR) launch_ens<SPEC_ROTATOR>(shape, blocks, s, beside, B);
  else launch_ens<SPEC_GENERIC>(shape, blocks, s, beside, B);
}

}  // namespace t32
}  // namespace pic
