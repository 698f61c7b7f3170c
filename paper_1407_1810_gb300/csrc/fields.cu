// fields.cu -- grid-sized kernels beside the particle hot path (FP64):
//   Yee leapfrog in integral form (App. A, Eqs. discreteeq, erpolarupdate) with
//   conducting radial boundaries (Sec. 3.4.1), the lossy layer (Eq. EBcond),
//   the 1-2-1 current filter with the polar remap (App. B), axis ghost
//   columns and FP32 gather copies, surface pair injection (Sec. 5.3,
//   Eq. volinjeq) and the Gauss-law / energy diagnostics.
// All metric factors are precomputed per row and per column (pic::Metric), so
// the kernels are pure streaming stencils over the padded arrays.
#include <algorithm>
#include <cstdio>
#include <cstring>

#include "pic_internal.h"

namespace pic {

namespace {

constexpr int BX = 32, BY = 8;

inline dim3 grid2(int ni, int nj) { return dim3((nj + BX - 1) / BX, (ni + BY - 1) / BY); }

// ---- the leapfrog of a step ---------------------------------------------------
// A step takes B forward by a half step, E by a full one and B by a half
// again (App. A).  The second half of one step and the first half of the next
// add the same curl of the same E, so the B update below forms it once, adds
// it to B^{n+1/2} for the B at integer time that the gather and every reader
// use (f[BR..BPH]), and adds it again for the half-step B of the next step
// (bh).  bh is always B + dB(E) of the stored fields: fields_b_start forms it
// after the fields were replaced.  Only the lossy rows take the curl twice
// (the layer scales E and B between the two halves).
//
// The FP64 pipe bounds these kernels (2 lanes a clock and SM): their cost is
// the number of FP64 operations a node, 31 here against 46 for three passes
// and FP64 -> FP32 conversion instructions.  The operations are explicitly
// rounded: single-context, batched and slab kernels give the same bits.

// h c curl E at node (i, j) for the three components of B (h = dt / 2)
__device__ __forceinline__ void curl_e(const Metric &m, int ri, int cj, double er, double er_j, double et,
                                       double et_i, double ep, double ep_j, double ep_i, double d[3]) {
  const double t0 = m.bT0[ri], t1 = m.bT1[ri];
  d[0] = __dmul_rn(m.bR[ri], __fma_rn(ep, m.cB1[cj], -__dmul_rn(ep_j, m.cB2[cj])));
  d[1] = __fma_rn(t1, ep_i, -__dmul_rn(t0, ep));
  d[2] = __fma_rn(-__dmul_rn(m.bP[ri], m.inv_dth_t[cj]), __dsub_rn(er, er_j), __fma_rn(t0, et, -__dmul_rn(t1, et_i)));
}

// E <- E + dt c curl B - F / dA over the faces of the dual grid (last three
// lines of Eq. discreteeq; E_r on the axis by Eq. erpolarupdate, obtained here
// from the same formula with sin(tb_{-1}) = sin(tb_{nth}) = 0 and the cap
// areas in inv_dcos_tb), then the lossy layer (Eq. EBcond: times 1 - sigma*
// at the component's own radial stagger), whose rows keep the E before it in
// epre for the second half step of B.  E_th, E_ph on the conductors (i = 0, nr)
// and E_ph on the axis are not updated: 0, or what pic_set_fields left there,
// which the layer scales like the rest.
__device__ __forceinline__ void e_node(const EnsFieldArg &S, int i, int j, double Fr, double Ft, double Fp) {
  const Grid &G = S.G;
  const Metric &m = G.m;
  const int ri = i + G.PI, cj = j + G.PJ;
  const size_t o = gidx(G, i, j);
  const double *Br = S.bh[0], *Bt = S.bh[1], *Bp = S.bh[2];
  const bool lossy = S.lossy_i0 >= 0 && i >= S.lossy_i0;
  const size_t l = lossy ? (size_t)(i - S.lossy_i0) * G.LD + cj : 0;
  if (i < G.nr) {  // E_r at (i+1/2, j)
    const double c = __fma_rn(Bp[o], m.cE1[cj], -__dmul_rn(Bp[o - 1], m.cE2[cj]));
    double e = __fma_rn(m.eR[ri], c, S.f[ER][o]);
    e = __fma_rn(-Fr, __dmul_rn(m.inv_area_h[ri], m.inv_dcos_tb[cj]), e);
    if (lossy) { S.epre[0][l] = e; e = __dmul_rn(e, m.keep_h[ri]); }
    S.f[ER][o] = e;
  }
  // (a slab's open side is an interior row)
  const bool in = (i >= 1 || G.open_lo) && (i < G.nr || G.open_hi);
  const double w0 = m.w0[ri], w1 = m.w1[ri], id2 = m.inv_dr2_h[ri];
  if ((in || lossy) && j < G.nth) {  // E_th at (i, j+1/2)
    double e = S.f[ETH][o];
    if (in) {
      const double c = __fma_rn(-m.cF[cj], Ft, __fma_rn(w0, Bp[o - G.LD], -__dmul_rn(w1, Bp[o])));
      e = __fma_rn(id2, c, e);
    }
    if (lossy) { S.epre[1][l] = e; e = __dmul_rn(e, m.keep_n[ri]); }
    S.f[ETH][o] = e;
  }
  const bool ph = in && j >= 1 && j < G.nth;
  if (ph || lossy) {  // E_ph at (i, j)
    double e = S.f[EPH][o];
    if (ph) {
      const double c = __fma_rn(m.wd[ri], __dsub_rn(Br[o], Br[o - 1]), Fp);
      const double k = __fma_rn(-m.inv_dtb[cj], c, __fma_rn(w1, Bt[o], -__dmul_rn(w0, Bt[o - G.LD])));
      e = __fma_rn(id2, k, e);
    }
    if (lossy) { S.epre[2][l] = e; e = __dmul_rn(e, m.keep_n[ri]); }
    S.f[EPH][o] = e;
  }
}

// B at integer time and at the next half step of node (i, j), the axis
// continuation of the half-integer-j components into columns -1 and nth (B_r
// even; E_th, B_ph odd) and the FP32 gather copies of the six components.
template <bool FP32>
__device__ __forceinline__ void b_node(const EnsFieldArg &S, int i, int j) {
  const Grid &G = S.G;
  const Metric &m = G.m;
  const int ri = i + G.PI, cj = j + G.PJ;
  const size_t o = gidx(G, i, j);
  const double er = S.f[ER][o], er_j = S.f[ER][o + 1], et = S.f[ETH][o], et_i = S.f[ETH][o + G.LD];
  const double ep = S.f[EPH][o], ep_j = S.f[EPH][o + 1], ep_i = S.f[EPH][o + G.LD];
  // B_th on the axis is not updated: 0, or what pic_set_fields left there, with
  // its FP32 copy; only the lossy layer changes them
  const bool lossy = S.lossy_i0 >= 0 && i >= S.lossy_i0;
  const bool axis = (j == 0 || j == G.nth) && lossy && i < G.nr;
  const double axis_bt = axis ? S.f[BTH][o] : 0.0;
  double d[3], d2[3], b[3];
  curl_e(m, ri, cj, er, er_j, et, et_i, ep, ep_j, ep_i, d2);
  if (lossy) {  // the half step before the layer: E as it was then
    const size_t l = (size_t)(i - S.lossy_i0) * G.LD + cj;
    const bool up = i < G.nr;
    curl_e(m, ri, cj, S.epre[0][l], S.epre[0][l + 1], S.epre[1][l], up ? S.epre[1][l + G.LD] : 0.0, S.epre[2][l],
           S.epre[2][l + 1], up ? S.epre[2][l + G.LD] : 0.0, d);
  } else {
    d[0] = d2[0]; d[1] = d2[1]; d[2] = d2[2];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) b[k] = __dadd_rn(S.bh[k][o], d[k]);
  if (lossy) {
    b[0] = __dmul_rn(b[0], m.keep_n[ri]);
    b[1] = __dmul_rn(b[1], m.keep_h[ri]);
    b[2] = __dmul_rn(b[2], m.keep_h[ri]);
  }
  const bool hj = j < G.nth, hi = i < G.nr;  // half-integer columns / rows of the grid
  if (hj) {  // B_r at (i, j+1/2)
    S.f[BR][o] = b[0];
    S.bh[0][o] = __dadd_rn(b[0], d2[0]);
  }
  if (hi && j >= 1 && hj) {  // B_th at (i+1/2, j)
    S.f[BTH][o] = b[1];
    S.bh[1][o] = __dadd_rn(b[1], d2[1]);
  } else if (axis) {
    S.f[BTH][o] = b[1] = __dmul_rn(axis_bt, m.keep_h[ri]);
  }
  if (hi && hj) {  // B_ph at (i+1/2, j+1/2)
    S.f[BPH][o] = b[2];
    S.bh[2][o] = __dadd_rn(b[2], d2[2]);
  } else {
    b[2] = 0.0;
  }
  float q[6];
  if (FP32) {
    q[0] = f64_to_f32(er); q[1] = f64_to_f32(et); q[2] = f64_to_f32(ep);
    q[3] = f64_to_f32(b[0]); q[4] = f64_to_f32(b[1]); q[5] = f64_to_f32(b[2]);
    S.f32[ER][o] = q[0]; S.f32[EPH][o] = q[2];
    if ((hi && j >= 1 && hj) || axis) S.f32[BTH][o] = q[4];
    if (hj) { S.f32[ETH][o] = q[1]; S.f32[BR][o] = q[3]; S.f32[BPH][o] = q[5]; }
  }
  if (j == 0 || j == G.nth - 1) {
    const size_t a = j == 0 ? o - 1 : o + 1;
    S.f[ETH][a] = -et; S.f[BR][a] = b[0]; S.f[BPH][a] = -b[2];
    if (FP32) { S.f32[ETH][a] = -q[1]; S.f32[BR][a] = q[3]; S.f32[BPH][a] = -q[5]; }
  }
}

// bh = B + dB(E) of the stored fields at node (i, j)
__device__ __forceinline__ void b_start_node(const EnsFieldArg &S, int i, int j) {
  const Grid &G = S.G;
  const size_t o = gidx(G, i, j);
  double d[3];
  curl_e(G.m, i + G.PI, j + G.PJ, S.f[ER][o], S.f[ER][o + 1], S.f[ETH][o], S.f[ETH][o + G.LD], S.f[EPH][o],
         S.f[EPH][o + 1], S.f[EPH][o + G.LD], d);
  const bool hj = j < G.nth, hi = i < G.nr;
  if (hj) S.bh[0][o] = __dadd_rn(S.f[BR][o], d[0]);
  if (hi && j >= 1 && hj) S.bh[1][o] = __dadd_rn(S.f[BTH][o], d[1]);
  if (hi && hj) S.bh[2][o] = __dadd_rn(S.f[BPH][o], d[2]);
}

__global__ void k_b_start(const __grid_constant__ EnsFieldArg S) {
  const int i = blockIdx.y * BY + threadIdx.y, j = blockIdx.x * BX + threadIdx.x;
  if (i <= S.G.nr && j <= S.G.nth) b_start_node(S, i, j);
}

// Axisymmetric continuation of the half-integer-j components into columns -1
// and nth (B_r even; E_th, B_ph odd).
__device__ __forceinline__ void ghost_row(const Grid &G, int i, double *Et, double *Br, double *Bp) {
  if (i > G.nr) return;
  const size_t n0 = gidx(G, i, -1), s0 = gidx(G, i, G.nth);
  Et[n0] = -Et[n0 + 1]; Br[n0] = Br[n0 + 1]; Bp[n0] = -Bp[n0 + 1];
  Et[s0] = -Et[s0 - 1]; Br[s0] = Br[s0 - 1]; Bp[s0] = -Bp[s0 - 1];
}

__global__ void k_axis_ghosts(Grid G, double *Et, double *Br, double *Bp) {
  ghost_row(G, blockIdx.x * blockDim.x + threadIdx.x, Et, Br, Bp);
}

// FP32 gather copies of the six components (the gather-prep step of the FP32
// path) over rows -g..nr+g and columns -1..nth: every node the gather can
// read.  The FP64 fields are zero outside rows 0..nr and columns -1..nth (no
// kernel writes there), and so are the FP32 copies from their allocation, so
// the padding beyond needs no copy.
__device__ __forceinline__ void copy32_node(const Grid &G, int i, int j, const double *__restrict__ a0,
                                            const double *__restrict__ a1, const double *__restrict__ a2,
                                            const double *__restrict__ a3, const double *__restrict__ a4,
                                            const double *__restrict__ a5, float *b0, float *b1, float *b2,
                                            float *b3, float *b4, float *b5) {
  if (i > G.nr + G.g || j > G.nth) return;
  const size_t k = gidx(G, i, j);
  b0[k] = f64_to_f32(a0[k]); b1[k] = f64_to_f32(a1[k]); b2[k] = f64_to_f32(a2[k]);
  b3[k] = f64_to_f32(a3[k]); b4[k] = f64_to_f32(a4[k]); b5[k] = f64_to_f32(a5[k]);
}

__global__ void k_copy32(Grid G, const double *__restrict__ a0, const double *__restrict__ a1,
                         const double *__restrict__ a2, const double *__restrict__ a3,
                         const double *__restrict__ a4, const double *__restrict__ a5, float *b0, float *b1,
                         float *b2, float *b3, float *b4, float *b5) {
  copy32_node(G, -G.g + (int)(blockIdx.y * BY + threadIdx.y), (int)(blockIdx.x * BX + threadIdx.x) - 1, a0, a1, a2,
              a3, a4, a5, b0, b1, b2, b3, b4, b5);
}

// One 1-2-1 pass (Eq. filtereq) with the polar remap of App. B: weights V_l(j)
// fold the part that would leave through the axis back onto the mirror point,
// + for integer-j arrays (F_r, F_ph, charge) and - for the half-integer-j F_th.
// Rows outside the ghost band -g..nr+g are not kept.
__device__ __forceinline__ void filter_node(const Grid &G, int i, int j, const double *__restrict__ in,
                                            double *__restrict__ out, int half_j) {
  const int nj = half_j ? G.nth : G.nth + 1;
  if (i > G.nr + G.g || j >= nj) return;
  double vm, v0 = 0.5, vp;
  if (half_j) {
    vm = j == 0 ? 0.0 : 0.25;
    vp = j == G.nth - 1 ? 0.0 : 0.25;
    if (j == 0) v0 -= 0.25;
    if (j == G.nth - 1) v0 -= 0.25;
  } else {
    vm = j == 0 ? 0.0 : (j == 1 ? 0.5 : 0.25);
    vp = j == G.nth ? 0.0 : (j == G.nth - 1 ? 0.5 : 0.25);
  }
  const size_t o = gidx(G, i, j);
  double s = 0.0;
#pragma unroll
  for (int k = -1; k <= 1; ++k) {
    const int ii = i + k;
    if (ii < -G.g || ii > G.nr + G.g) continue;
    const size_t q = o + (ptrdiff_t)k * G.LD;
    double row = vm * in[q - 1] + v0 * in[q] + vp * in[q + 1];
    s += (k == 0 ? 0.5 : 0.25) * row;
  }
  out[o] = s;
}

__global__ void k_filter(Grid G, const double *__restrict__ in, double *__restrict__ out, int half_j) {
  follow();
  filter_node(G, -G.g + (int)(blockIdx.y * BY + threadIdx.y), blockIdx.x * BX + threadIdx.x, in, out, half_j);
}

// Surface charge per meridional cell: the jump of E_r across the conductor,
// total E_r at (1/2, j) minus the analytic inside field's E_r at (r0, theta_j)
// (zero for the monopole fields), averaged over the cell's two nodes.  The
// analytic fields' part is a quadratic in cos theta (sigma_jump).
__device__ __forceinline__ void sigma_cell(const Grid &G, int j, const double *__restrict__ Er, const SigmaJump &K,
                                           double *sig, long long *smax) {
  if (j >= G.nth) return;
  double e[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double ct = G.m.cos_t[j + h + G.PJ];
    e[h] = Er[gidx(G, 0, j + h)] + fma(ct, fma(ct, K.k2, K.k1), K.k0);
  }
  const double s = 0.5 * (e[0] + e[1]);
  sig[j] = s;
  if (smax) atomicMax(smax, __double_as_longlong(fabs(s)));
}

// ---- deposit -> filtered flux, in one pass ----------------------------------
// The N passes of the 1-2-1 filter act along rows and columns independently,
// so they are one convolution with the 2N + 1 binomial weights along each,
// taken from a shared-memory tile with a halo of N nodes:
//  - the polar fold of App. B (a pass's share that lands beyond the axis comes
//    back to its mirror point) equals the plain convolution of the deposit
//    continued past the pole as its mirror image -- even, with the pole node
//    doubled and its result halved, for integer j; odd for half-integer j;
//  - rows that leave the ghost band are dropped after every pass: the
//    convolution of the deposit continued as an odd image past row -g - 1 and
//    nr + g + 1.
// The weights are integers over 4^N a direction, so the FP32 path's fixed-point
// sums are filtered exactly in 64-bit integers, on the pipes that have the
// room, and rounded once (a nine-launch FP64 filter took 255 us of a 1024^2
// rotator step, the FP64 pipe 86 % busy).  A tile whose sums leave no room for
// the 16^N of the weights takes 128-bit integers: the same exact result.
constexpr int FUSE_FILT = 4;  // passes the tile's halo holds; more run pass by pass
constexpr int TW = BX + 2 * FUSE_FILT, TH = BY + 2 * FUSE_FILT;
__constant__ int FILT_W[FUSE_FILT + 1][FUSE_FILT + 1] = {  // C(2N, N + k)
    {1, 0, 0, 0, 0}, {2, 1, 0, 0, 0}, {6, 4, 1, 0, 0}, {20, 15, 6, 1, 0}, {70, 56, 28, 8, 1}};

// FP64 tiles take the weights over 4^N a direction from a table of doubles (an
// integer-to-double conversion or a product costs as much of the FP64 pipe as
// an addition of the convolution), so that no weighted sum is larger than what
// it averages (only two neighbours of one sign beyond 2^1023 still overflow).
// Where a tile holds a pole, its other nodes are halved instead of the pole's
// doubled, so that a value of the last binade stays finite; the halving goes
// through the exponent bits, and infinities and NaN pass as they are.  All of
// it is exact above the subnormal numbers.
__constant__ double FILT_WD[FUSE_FILT + 1][FUSE_FILT + 1] = {
    {1, 0, 0, 0, 0},
    {2 / 4., 1 / 4., 0, 0, 0},
    {6 / 16., 4 / 16., 1 / 16., 0, 0},
    {20 / 64., 15 / 64., 6 / 64., 1 / 64., 0},
    {70 / 256., 56 / 256., 28 / 256., 8 / 256., 1 / 256.}};
template <class T>
__device__ __forceinline__ T filt_weight(int N, int k) { return T(FILT_W[N][k]); }
template <>
__device__ __forceinline__ double filt_weight<double>(int N, int k) { return FILT_WD[N][k]; }
// a loaded value with the factor c of its image; FP64: its sign, and half of
// it where c stands for 1 against the 2 of a pole in the same tile
template <class T>
__device__ __forceinline__ T filt_scaled(int c, bool, T v) { return T(c) * v; }
template <>
__device__ __forceinline__ double filt_scaled<double>(int c, bool halve, double v) {
  int hi = __double2hiint(v);
  const int lo = __double2loint(v);
  if (halve && (c == 1 || c == -1)) {
    const unsigned e = (unsigned)hi >> 20 & 0x7ffu;
    if (e - 2u < 0x7fdu) {  // its half is normal
      hi -= 0x00100000;
    } else if (e < 2u && ((hi & 0x7fffffff) | lo)) {
      v *= 0.5;
      return c < 0 ? -v : v;
    }
  }
  return __hiloint2double(c < 0 ? hi ^ 0x80000000 : hi, lo);
}

// Images of the rows and columns that this thread loads of a tile: array
// offset (or -1: zero) and factor (+-1, +-2) of rows i0 - N + ty (+ 8) and, for
// integer and half-integer j, of columns j0 - N + tx (+ 32) of the continued
// deposit.  In registers: a phase of the block that forms them in shared
// memory costs another barrier (a 72 x 56 step 43.2 -> 42.4 us, 192 x 160
// 79.5 -> 76.6 us with both these and the unrolled passes).
struct FiltImages {
  int row[2], row_c[2], col[2][2], col_c[2][2];
};

// whether a pole is among the columns a tile reads
__device__ __forceinline__ bool filt_poles(const Grid &G, int j0, int N) {
  return j0 - N <= 0 || j0 + BX - 1 + N >= G.nth;
}

__device__ __forceinline__ FiltImages filt_images(const Grid &G, int i0, int j0, int N) {
  FiltImages im;
  const int lo = -G.g - 1, hi = G.nr + G.g + 1, n = G.nth;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    int ii = i0 - N + (int)threadIdx.y + a * BY, c = 1;
    if (ii <= lo) { ii = 2 * lo - ii; c = -1; }
    else if (ii >= hi) { ii = 2 * hi - ii; c = -1; }
    im.row[a] = ii <= lo || ii >= hi ? -1 : ii + G.PI;  // -1: the dropped row itself
    im.row_c[a] = c;
    const int j = j0 - N + (int)threadIdx.x + a * BX;
    // right of every column that a node of the tile reads: any
    int jj = j > n + 2 * FUSE_FILT ? n : j, jh = j > n + 2 * FUSE_FILT ? n - 1 : j, d = 1;
    while (jj < 0 || jj > n) jj = jj < 0 ? -jj : 2 * n - jj;
    while (jh < 0 || jh >= n) { jh = jh < 0 ? -1 - jh : 2 * n - 1 - jh; d = -d; }
    im.col[0][a] = jj + G.PJ;
    im.col_c[0][a] = jj == 0 || jj == n ? 2 : 1;
    im.col[1][a] = jh + G.PJ;
    im.col_c[1][a] = d;
  }
  return im;
}

template <class T, int NC>
struct FiltTile {
  T in[NC][TH][TW + 1];
  T mid[NC][TH][BX + 1];
};

// NC components (the first of them component c0) of the tile with N passes at
// this thread's node; every thread of the block calls it.  halve (FP64): the
// tile holds a pole; the integer-j sums of its other nodes are half of theirs
template <int N, class T, int NC, class L>
__device__ __forceinline__ void filt_conv(FiltTile<T, NC> &t, const FiltImages &im, const Grid &G, int c0, bool halve,
                                          T out[NC], const L &load) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  constexpr int w = BX + 2 * N, h = BY + 2 * N;
#pragma unroll
  for (int k = 0; k < NC; ++k)
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int r = ty + a * BY, q = tx + b * BX, half = c0 + k == 1;
        if (r < h && q < w) {
          const int ro = im.row[a];
          t.in[k][r][q] = ro < 0 ? T(0)
                                 : filt_scaled<T>(im.row_c[a] * im.col_c[half][b], halve && !half,
                                                  load(c0 + k, (size_t)ro * G.LD + im.col[half][b]));
        }
      }
  __syncthreads();
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int r = ty + a * BY;
    if (r < h)
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const T *x = &t.in[k][r][tx + N];
        T s = filt_weight<T>(N, 0) * x[0];
#pragma unroll
        for (int m = 1; m <= N; ++m) s += filt_weight<T>(N, m) * (x[-m] + x[m]);
        t.mid[k][r][tx] = s;
      }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    T s = filt_weight<T>(N, 0) * t.mid[k][ty + N][tx];
#pragma unroll
    for (int m = 1; m <= N; ++m) s += filt_weight<T>(N, m) * (t.mid[k][ty + N - m][tx] + t.mid[k][ty + N + m][tx]);
    out[k] = s;
  }
}

union FiltSmem {
  FiltTile<long long, 3> q;
  FiltTile<__int128, 1> w;
  FiltTile<double, 3> d;
  __device__ FiltSmem() {}
};

// the three filtered components at this thread's node, N passes
template <bool FP32, int N>
__device__ __forceinline__ void filtered_flux(const EnsFieldArg &S, FiltSmem &sm, int i0, int j0, bool pole,
                                              double F[3]) {
  const Grid &G = S.G;
  const FiltImages im = filt_images(G, i0, j0, N);
  if (FP32) {
    const int s = qexp_value(S.qexp) - KFIX;  // one flux unit is 2^s of charge
    const long long lim = 1ll << (60 - 4 * N);
    bool big = false;
    long long v[3];
    filt_conv<N>(sm.q, im, G, 0, false, v, [&](int k, size_t x) {
      const long long y = S.acc[k][x];
      big |= y >= lim || y <= -lim;
      return y;
    });
#pragma unroll
    for (int k = 0; k < 3; ++k) F[k] = fixed_to_f64(k != 1 && pole ? v[k] / 2 : v[k], s - 4 * N);
    if (__syncthreads_or(big)) {
      for (int k = 0; k < 3; ++k) {
        __int128 z[1];
        filt_conv<N>(sm.w, im, G, k, false, z, [&](int c, size_t x) { return (__int128)S.acc[c][x]; });
        F[k] = fixed_to_f64(k != 1 && pole ? z[0] / 2 : z[0], s - 4 * N);
        __syncthreads();
      }
    }
  } else {
    double v[3];
    const bool poles = filt_poles(G, j0, N);
    filt_conv<N>(sm.d, im, G, 0, poles, v, [&](int k, size_t x) { return S.Fin[k][x]; });
#pragma unroll
    for (int k = 0; k < 3; ++k) F[k] = k != 1 && poles && !pole ? v[k] + v[k] : v[k];
  }
}

// One block (32 x 8 nodes of the ghost band -g..nr+g, 0..nth) of the E update:
// the flux of the deposit filtered and stored (the step's fluxes), then E.
template <bool FP32>
__device__ __forceinline__ void e_block(const EnsFieldArg &S, unsigned b, FiltSmem &sm) {
  const Grid &G = S.G;
  const unsigned gx = (unsigned)(G.nth + 1 + BX - 1) / BX;
  const int i0 = -G.g + (int)(b / gx) * BY, j0 = (int)(b % gx) * BX;
  const int i = i0 + (int)threadIdx.y, j = j0 + (int)threadIdx.x;
  const bool in = i <= G.nr + G.g && j <= G.nth;
  const size_t o = in ? gidx(G, i, j) : 0;
  const int N = S.n_filt;
  const bool pole = j == 0 || j == G.nth;
  double F[3] = {0.0, 0.0, 0.0};
  switch (N) {
    case 0:
      if (in) {
        const int s = FP32 ? qexp_value(S.qexp) - KFIX : 0;  // one flux unit is 2^s of charge
#pragma unroll
        for (int k = 0; k < 3; ++k) F[k] = FP32 ? fixed_to_f64(S.acc[k][o], s) : S.Fin[k][o];
      }
      break;
    case 1: filtered_flux<FP32, 1>(S, sm, i0, j0, pole, F); break;
    case 2: filtered_flux<FP32, 2>(S, sm, i0, j0, pole, F); break;
    case 3: filtered_flux<FP32, 3>(S, sm, i0, j0, pole, F); break;
    case 4: filtered_flux<FP32, 4>(S, sm, i0, j0, pole, F); break;
    default:  // filtered pass by pass before this launch
      if (in)
        for (int k = 0; k < 3; ++k) F[k] = S.Fout[k][o];
  }
  if (b == 0 && threadIdx.x == 0 && threadIdx.y == 0 && S.inject) S.cnt[CNT_SMAX] = 0;  // raised by the B update
  if (!in) return;
  if (N <= FUSE_FILT) {
    S.Fout[0][o] = F[0];
    if (j < G.nth) S.Fout[1][o] = F[1];
    S.Fout[2][o] = F[2];
  }
  if (i >= 0 && i <= G.nr) e_node(S, i, j, F[0], F[1], F[2]);
}

// One block of the B update over the same nodes; it also clears the deposit
// of the step, and with `sigma` forms the surface charge of the injection
// from the new E_r (its maximum too, when no smoothing pass follows).
template <bool FP32>
__device__ __forceinline__ void b_block(const EnsFieldArg &S, unsigned b, bool sigma) {
  const Grid &G = S.G;
  const unsigned gx = (unsigned)(G.nth + 1 + BX - 1) / BX;
  const int i = -G.g + (int)((b / gx) * BY + threadIdx.y), j = (int)((b % gx) * BX + threadIdx.x);
  if (i > G.nr + G.g || j > G.nth) return;
  const size_t o = gidx(G, i, j);
  if (FP32)
    for (int k = 0; k < 3; ++k) S.acc[k][o] = 0;
  else  // (an even number of separate passes leaves the filtered flux in Fin)
    for (int k = 0; k < 3; ++k) (S.Fout[k] == S.Fin[k] ? S.Ftmp : S.Fin)[k][o] = 0.0;
  if (i < 0 || i > G.nr) return;
  b_node<FP32>(S, i, j);
  if (sigma && i == 0) sigma_cell(G, j, S.f[ER], S.jump, S.sig, S.inject_smooth ? nullptr : S.cnt + CNT_SMAX);
}

// the passes of an integer-j FP64 array (the node charge) in one
template <int N>
__device__ __forceinline__ double filtered_charge(FiltTile<double, 1> &t, const Grid &G, int i0, int j0, bool pole,
                                                  const double *__restrict__ a) {
  double v[1];
  const bool poles = filt_poles(G, j0, N);
  filt_conv<N>(t, filt_images(G, i0, j0, N), G, 0, poles, v, [&](int, size_t x) { return a[x]; });
  return poles && !pole ? v[0] + v[0] : v[0];
}
__global__ void __launch_bounds__(BX *BY) k_filter_tile(Grid G, const double *__restrict__ a, double *__restrict__ out,
                                                       int N) {
  __shared__ FiltTile<double, 1> t;
  const int i0 = -G.g + (int)blockIdx.y * BY, j0 = (int)blockIdx.x * BX;
  const int i = i0 + (int)threadIdx.y, j = j0 + (int)threadIdx.x;
  const bool pole = j == 0 || j == G.nth;
  const double v = N == 1 ? filtered_charge<1>(t, G, i0, j0, pole, a) : N == 2 ? filtered_charge<2>(t, G, i0, j0, pole, a)
                 : N == 3 ? filtered_charge<3>(t, G, i0, j0, pole, a) : filtered_charge<4>(t, G, i0, j0, pole, a);
  if (i <= G.nr + G.g && j <= G.nth) out[gidx(G, i, j)] = v;
}

template <bool FP32>
__global__ void __launch_bounds__(BX *BY) k_e_step(const __grid_constant__ EnsFieldArg S) {
  __shared__ FiltSmem sm;
  follow();
  e_block<FP32>(S, blockIdx.x, sm);
}
template <bool FP32>
__global__ void __launch_bounds__(BX *BY) k_b_step(const __grid_constant__ EnsFieldArg S, int sigma) {
  follow();
  b_block<FP32>(S, blockIdx.x, sigma != 0);
}

// fixed point -> FP64 fluxes over the ghost band, for the pass-by-pass filter
__global__ void k_flux_from_acc(const __grid_constant__ EnsFieldArg S) {
  follow();
  const Grid &G = S.G;
  const int i = -G.g + (int)(blockIdx.y * BY + threadIdx.y), j = blockIdx.x * BX + threadIdx.x;
  if (i > G.nr + G.g || j > G.nth) return;
  const int s = qexp_value(S.qexp) - KFIX;
  const size_t o = gidx(G, i, j);
  for (int k = 0; k < 3; ++k) S.Fin[k][o] = fixed_to_f64(S.acc[k][o], s);
}

__global__ void k_inject_sigma(Grid G, const double *__restrict__ Er, SigmaJump K, double *sig, long long *smax) {
  sigma_cell(G, blockIdx.x * blockDim.x + threadIdx.x, Er, K, sig, smax);
}

// One 1-2-1 pass over sigma along theta; each polar cell is its own mirror
// image across the axis.
__device__ __forceinline__ void smooth_cell(int j, int nth, const double *__restrict__ in, double *out,
                                            long long *smax) {
  if (j >= nth) return;
  const double a = in[j > 0 ? j - 1 : 0], c = in[j < nth - 1 ? j + 1 : nth - 1];
  const double s = ((a + 2.0 * in[j]) + c) * 0.25;
  out[j] = s;
  if (smax) atomicMax(smax, __double_as_longlong(fabs(s)));
}

__global__ void k_inject_smooth(int nth, const double *__restrict__ in, double *out, long long *smax) {
  follow();
  smooth_cell(blockIdx.x * blockDim.x + threadIdx.x, nth, in, out, smax);
}

// SplitMix64 (Steele, Lea and Flood 2014) as a counter-based generator:
// output n + 1 of the stream seeded with `seed` is the variant-13 mix of
// seed + (n + 1) times the golden-ratio increment.
__device__ inline uint64_t splitmix64_out(uint64_t seed, uint64_t n) {
  uint64_t z = seed + (n + 1u) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

struct InjectRule {
  int mode, npp;
  double finj, q;       // q: VARIABLE, |charge| per particle
  uint64_t seed, step;  // VARIABLE: generator key (seed, step * nth + j)
};

// Pairs injected into cell j and the |charge| of each (Eq. volinjeq).
__device__ inline int inject_count(const Grid &G, const InjectRule &R, int j, double sg, double sm, double dA,
                                   double &w, bool &capped) {
  capped = false;
  if (R.mode == PIC_INJECT_VARIABLE) {
    const double x = R.finj * fabs(sg) * dA / R.q;
    w = R.q;
    if (!(fabs(sg) > 1e-12 * sm && x > 0.0)) return 0;
    int m;
    if (x >= R.npp + 1.0) {
      m = R.npp + 1;
    } else {
      const double fl = floor(x);
      const double u = (double)(splitmix64_out(R.seed, R.step * (uint64_t)G.nth + (uint64_t)j) >> 11) *
                       (1.0 / 9007199254740992.0);
      m = (int)fl + (u < x - fl ? 1 : 0);
    }
    if (m > R.npp) { m = R.npp; capped = true; }
    return m;
  }
  w = R.finj * fabs(sg) * dA / R.npp;
  return (fabs(sg) > 1e-12 * sm && w > 0.0) ? R.npp : 0;
}

// One thread per slot (j, k, sign) of the 2 npp nth reserved this step; slots
// past a cell's count keep zero charge (free).
// (every lane of a warp calls it: the exponent is raised warp-wide)
template <bool FP32>
__device__ __forceinline__ void inject_slot(int64_t idx, const Grid &G, const double *__restrict__ sig,
                                            const long long *smax, const Parts64 &P, const Parts32 &Q, int64_t base,
                                            int64_t id0, const InjectRule &R, long long *cnt, long long *capped_cnt,
                                            long long *qexp) {
  const int npp = R.npp;
  int qe = (int)QEXP_NONE;
  if (idx < (int64_t)G.nth * npp * 2) {
    const int j = (int)(idx / (2 * npp)), k = (int)((idx / 2) % npp), s = (int)(idx % 2);
    const double sm = __longlong_as_double(*smax), sg = sig[j];
    const double r0 = G.r_min;
    const double dA = 2.0 * PI_D * r0 * r0 * (G.m.cos_t[j + G.PJ] - G.m.cos_t[j + 1 + G.PJ]);
    double w;
    bool capped;
    const int m = inject_count(G, R, j, sg, sm, dA, w, capped);
    if (capped && k == 0 && s == 0) add_ll(capped_cnt, 1LL);
    const bool on = k < m;
    const int64_t slot = base + idx;
    const double qv = on ? (s == 0 ? w : -w) : 0.0;
    const double oy = (k + 0.5) / (on ? m : npp);
    if (FP32) {
      Q.cell[slot] = ((uint32_t)(0 + CELL_BIAS) << 16) | (uint32_t)j;
      Q.dx[slot] = 0.5f;
      Q.dy[slot] = (float)oy;
      Q.ur[slot] = Q.ut[slot] = Q.up[slot] = 0.0f;
      Q.qw[slot] = (float)qv;
      Q.id[slot] = id0 + idx;
      if (on) qe = charge_exp(fabsf((float)qv));
    } else {
      P.x1[slot] = 0.5;
      P.x2[slot] = j + oy;
      P.ur[slot] = P.ut[slot] = P.up[slot] = 0.0;
      P.qw[slot] = qv;
      P.id[slot] = id0 + idx;
    }
    if (on) add_ll(cnt, 1LL);
  }
  if (FP32) raise_qexp(qexp, qe);  // every lane of the warp reaches this
}

template <bool FP32>
__global__ void k_inject_write(Grid G, const double *__restrict__ sig, const long long *smax, Parts64 P,
                               Parts32 Q, int64_t base, int64_t id0, InjectRule R, long long *cnt,
                               long long *capped_cnt, long long *qexp) {
  follow();
  inject_slot<FP32>(blockIdx.x * (int64_t)blockDim.x + threadIdx.x, G, sig, smax, P, Q, base, id0, R, cnt,
                    capped_cnt, qexp);
}

__device__ inline double warp_max(double v) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ inline double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Integral Gauss law per dual cell: G = flux of E out of the dual cell of node
// (i, j) (caps close at the axis); d = G - Qbar.  snapshot: store d; else
// reduce max |d - d_0| and max |Q| over interior nodes 1 <= i <= imax.
__global__ void k_gauss(Grid G, const double *__restrict__ Er, const double *__restrict__ Et,
                        const double *__restrict__ Qf, const double *__restrict__ Qa, double *snap, int ilo, int imax,
                        int snapshot, long long *gmax, long long *qmax) {
  const int j = blockIdx.x * BX + threadIdx.x, i = ilo + blockIdx.y * BY + threadIdx.y;
  double v = 0.0, qa = 0.0;
  if (i <= imax && j <= G.nth) {
    const Metric &m = G.m;
    const int ri = i + G.PI, cj = j + G.PJ;
    const size_t o = gidx(G, i, j);
    const double dc = 1.0 / m.inv_dcos_tb[cj];
    const double ar = 2.0 * PI_D * m.r_h[ri] * m.r_h[ri], al = 2.0 * PI_D * m.r_h[ri - 1] * m.r_h[ri - 1];
    const double side = PI_D * (m.r_h[ri] * m.r_h[ri] - m.r_h[ri - 1] * m.r_h[ri - 1]);
    double g = Er[o] * ar * dc - Er[o - G.LD] * al * dc + (Et[o] * m.sin_tb[cj] - Et[o - 1] * m.sin_tb[cj - 1]) * side;
    double d = g - Qf[o];
    if (snapshot) snap[o] = d;
    else v = fabs(d - snap[o]);
    qa = Qa[o];
  }
  v = warp_max(v);
  qa = warp_max(qa);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(gmax, __double_as_longlong(v));
    atomicMax(qmax, __double_as_longlong(qa));
  }
}

// rows 0..imax (a slab leaves its open outer interface row to the neighbour)
__global__ void k_field_energy(Grid G, const double *f0, const double *f1, const double *f2, const double *f3,
                               const double *f4, const double *f5, int imax, double *acc) {
  const int j = blockIdx.x * BX + threadIdx.x, i = blockIdx.y * BY + threadIdx.y;
  double e = 0.0;
  if (i <= imax && j <= G.nth) {
    const Metric &m = G.m;
    const int ri = i + G.PI, cj = j + G.PJ;
    const size_t o = gidx(G, i, j);
    const double *fs[6] = {f0, f1, f2, f3, f4, f5};
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int si = stag_i(c), sj = stag_j(c);
      if ((si && i >= G.nr) || (sj && j >= G.nth)) continue;
      const double vr = si ? m.vol_r_h[ri] : m.vol_r_n[ri];
      const double vt = sj ? m.vol_t_h[cj] : m.vol_t_n[cj];
      const double v = fs[c][o];
      e += 0.5 * v * v * vr * vt;
    }
  }
  e = warp_sum(e);
  if ((threadIdx.x & 31) == 0) atomicAdd(acc, e);
}

// ---- the same kernels over the members of an ensemble ----------------------
// 256-thread blocks; a member's 2-D node blocks (32 x 8, as the kernels above
// take them) are numbered row-major across its grid.
struct Node2 {
  int i, j;
};
__device__ inline Node2 node_of(unsigned b, int nj, int i_first) {
  const unsigned gx = (unsigned)(nj + BX - 1) / BX;
  return Node2{i_first + (int)((b / gx) * BY + (threadIdx.x >> 5)), (int)((b % gx) * BX + (threadIdx.x & 31))};
}

// pass `pass` of the filter on all three flux components: even passes read
// the deposit's buffers and write the scratch, odd passes the reverse
__global__ void k_ens_filter(const EnsFieldArg *__restrict__ tab, EnsList L, int pass) {
  const int2 e = L.blk[blockIdx.x];
  const EnsFieldArg &E = tab[e.x];
  const Grid &G = E.G;
  const unsigned per = (unsigned)((G.nth + 1 + BX - 1) / BX) * (unsigned)((G.nr + 2 * G.g + 1 + BY - 1) / BY);
  const unsigned b = (unsigned)e.y;
  const int comp = (int)(b / per);
  const Node2 n = node_of(b % per, G.nth + 1, -G.g);
  const double *in = (pass & 1) ? E.Ftmp[comp] : E.Fin[comp];
  double *out = (pass & 1) ? E.Fin[comp] : E.Ftmp[comp];
  filter_node(G, n.i, n.j, in, out, comp == 1);
}

__global__ void k_ens_flux(const EnsFieldArg *__restrict__ tab, EnsList L) {
  const int2 e = L.blk[blockIdx.x];
  const EnsFieldArg &E = tab[e.x];
  const Node2 n = node_of((unsigned)e.y, E.G.nth + 1, -E.G.g);
  if (n.i > E.G.nr + E.G.g || n.j > E.G.nth) return;
  const int s = qexp_value(E.qexp) - KFIX;
  const size_t o = gidx(E.G, n.i, n.j);
  for (int k = 0; k < 3; ++k) E.Fin[k][o] = fixed_to_f64(E.acc[k][o], s);
}

// the member of this block, its argument copied to shared memory (one
// coalesced load instead of a dependent load for every array and table)
__device__ __forceinline__ unsigned ens_member(const EnsFieldArg *__restrict__ tab, const EnsList &L,
                                               EnsFieldArg &S) {
  static_assert(sizeof(EnsFieldArg) % 8 == 0 && sizeof(EnsFieldArg) <= 8 * BX * BY, "copied by one block");
  const int2 e = L.blk[blockIdx.x];
  const int t = threadIdx.y * BX + threadIdx.x;
  if (t < (int)(sizeof(EnsFieldArg) / 8))
    reinterpret_cast<unsigned long long *>(&S)[t] = reinterpret_cast<const unsigned long long *>(tab + e.x)[t];
  __syncthreads();
  return (unsigned)e.y;
}
struct EnsMember {
  EnsFieldArg S;
  __device__ EnsMember() {}
};

__global__ void __launch_bounds__(BX *BY) k_ens_e_step(const EnsFieldArg *__restrict__ tab, EnsList L) {
  __shared__ FiltSmem sm;
  __shared__ EnsMember M;
  const unsigned b = ens_member(tab, L, M.S);
  e_block<true>(M.S, b, sm);
}

__global__ void __launch_bounds__(BX *BY) k_ens_b_step(const EnsFieldArg *__restrict__ tab, EnsList L) {
  __shared__ EnsMember M;
  const unsigned b = ens_member(tab, L, M.S);
  b_block<true>(M.S, b, M.S.inject != 0);
}

__device__ inline InjectRule ens_rule(const EnsFieldArg &E) {
  return InjectRule{E.inject, E.npp, E.f_inj, E.inject_q, E.inject_seed, E.inj_step};
}

__global__ void k_ens_smooth(const EnsFieldArg *__restrict__ tab, EnsList L, int pass) {
  const int2 e = L.blk[blockIdx.x];
  const EnsFieldArg &E = tab[e.x];
  const int j = (int)(((unsigned)e.y) * blockDim.x + threadIdx.x), nth = E.G.nth;
  const double *in = (pass & 1) ? E.sig + (nth + 1) : E.sig;
  double *out = (pass & 1) ? E.sig : E.sig + (nth + 1);
  smooth_cell(j, nth, in, out, pass == E.inject_smooth - 1 ? E.cnt + CNT_SMAX : nullptr);
}

__global__ void k_ens_write(const EnsFieldArg *__restrict__ tab, EnsList L) {
  const int2 e = L.blk[blockIdx.x];
  const EnsFieldArg &E = tab[e.x];
  const int64_t idx = (int64_t)((unsigned)e.y) * blockDim.x + threadIdx.x;
  const double *sig = (E.inject_smooth & 1) ? E.sig + (E.G.nth + 1) : E.sig;
  const Parts64 none;
  inject_slot<true>(idx, E.G, sig, E.cnt + CNT_SMAX, none, E.p32, E.inj_base, E.inj_id0, ens_rule(E),
                    E.cnt + CNT_INJECTED, E.cnt + CNT_CAPPED, E.qexp);
}

inline int div_up(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

}  // namespace

int lossy_first_row(const pic_ctx *c) {
  return c->d.absorb_profile != PIC_ABSORB_NONE && c->d.absorb_cells > 0
             ? std::max(0, c->G.nr - c->G.absorb_cells - 1) : -1;
}

int ens_blocks(const pic_ctx *c, int kind) {
  const Grid &G = c->G;
  const int band = div_up(G.nth + 1, BX) * div_up(G.nr + 2 * G.g + 1, BY);  // nodes -g..nr+g, 0..nth
  switch (kind) {
    case ENS_FLUX: return c->d.n_filt > FUSE_FILT ? band : 0;
    case ENS_FILTER: return c->d.n_filt > FUSE_FILT ? 3 * band : 0;
    case ENS_BAND: return band;
    case ENS_SMOOTH: return c->d.inject ? div_up(G.nth, 256) : 0;
    case ENS_WRITE: return c->d.inject ? div_up((int64_t)G.nth * c->d.pairs_per_cell * 2, 256) : 0;
    default: return 0;
  }
}

// The analytic fields' jump of E_r at the star, E_r outside at (1/2, j) minus
// E_r inside at r0, as k0 + k1 cos th + k2 cos^2 th at time t (vacuum_field's
// terms in E_r)
SigmaJump sigma_jump(const pic_ctx *c, double t) {
  const Grid &G = c->G;
  const double W = omega_at(G.omega, G.t_spin, t), r0 = G.r_min;
  const double rb = c->d.r_map == PIC_R_LOG ? r0 * std::exp(0.5 * G.dxi) : r0 + 0.5 * G.dxi, q = r0 / rb;
  const double in = G.b0 * r0 * W;  // mu W / r0^2
  SigmaJump K{0.0, 0.0, 0.0};
  if (G.vacuum == PIC_VAC_MONOPOLE_ROTATOR) {
    K.k1 = -2.0 * G.b0 * q * q * q * r0 * W;
  } else if (G.vacuum == PIC_VAC_DIPOLE_COROT) {  // sin^2 th (mu W / rb^2 - mu W / r0^2)
    K.k0 = in * (q * q - 1.0);
    K.k2 = -K.k0;
  } else if (G.vacuum == PIC_VAC_DIPOLE_ROTATOR) {  // -a (3 cos^2 th - 1) - in sin^2 th
    const double a = in * q * q * q * q;
    K.k0 = a - in;
    K.k2 = in - 3.0 * a;
  }
  return K;
}

// launches of the grid phases of one step (as pic_step_body makes them)
int grid_launches(const pic_ctx *c) {
  return (c->d.n_filt > FUSE_FILT ? 1 + 3 * c->d.n_filt : 0) + 2 + (c->d.inject ? 1 + c->d.inject_smooth : 0);
}

// whether the step's filter passes end in the scratch planes (pass by pass,
// an odd number): F and Ft then change places
bool filter_swaps(const pic_ctx *c) { return c->d.n_filt > FUSE_FILT && (c->d.n_filt & 1); }

void ens_fill_field_arg(const pic_ctx *c, EnsFieldArg *a) {
  memset(a, 0, sizeof *a);
  const bool fp32 = c->d.precision == PIC_FP32, fused = c->d.n_filt <= FUSE_FILT;
  a->G = c->G;
  for (int k = 0; k < 6; ++k) { a->f[k] = c->f[k]; a->f32[k] = c->f32[k]; }
  for (int k = 0; k < 3; ++k) {
    a->bh[k] = c->bh[k];
    a->epre[k] = c->epre[k];
    // FP64: the deposit is in Ft and the filtered flux goes to F.  FP32: pass
    // by pass the converted deposit goes to F, and Ft is the scratch.
    a->Fin[k] = fp32 ? c->F[k] : c->Ft[k];
    a->Ftmp[k] = fp32 ? c->Ft[k] : c->F[k];
    a->Fout[k] = fused ? c->F[k] : ((c->d.n_filt & 1) ? a->Ftmp[k] : a->Fin[k]);
    a->acc[k] = c->acc[k];
  }
  a->cnt = c->d_cnt;
  a->qexp = c->qexp;
  a->sig = c->sig;
  a->p32 = c->p32;
  a->f_inj = c->d.f_inj;
  a->inject_q = c->d.inject_q;
  a->inject_seed = c->d.inject_seed;
  a->inject = c->d.inject;
  a->npp = c->d.pairs_per_cell;
  a->inject_smooth = c->d.inject_smooth;
  a->n_filt = c->d.n_filt;
  a->lossy_i0 = lossy_first_row(c);
}

void ens_filter(const EnsFieldArg *tab, const EnsList &L, int blocks, int pass, cudaStream_t s) {
  k_ens_filter<<<(unsigned)blocks, 256, 0, s>>>(tab, L, pass);
}
void ens_flux(const EnsFieldArg *tab, const EnsList &L, int blocks, cudaStream_t s) {
  k_ens_flux<<<(unsigned)blocks, 256, 0, s>>>(tab, L);
}
void ens_e_step(const EnsFieldArg *tab, const EnsList &L, int blocks, cudaStream_t s) {
  k_ens_e_step<<<(unsigned)blocks, dim3(BX, BY), 0, s>>>(tab, L);
}
void ens_b_step(const EnsFieldArg *tab, const EnsList &L, int blocks, cudaStream_t s) {
  k_ens_b_step<<<(unsigned)blocks, dim3(BX, BY), 0, s>>>(tab, L);
}
void ens_inject_smooth(const EnsFieldArg *tab, const EnsList &L, int blocks, int pass, cudaStream_t s) {
  k_ens_smooth<<<(unsigned)blocks, 256, 0, s>>>(tab, L, pass);
}
void ens_inject_write(const EnsFieldArg *tab, const EnsList &L, int blocks, cudaStream_t s) {
  k_ens_write<<<(unsigned)blocks, 256, 0, s>>>(tab, L);
}

void fields_b_start(pic_ctx *c) {
  if (c->bh_ok) return;
  EnsFieldArg a;
  ens_fill_field_arg(c, &a);
  ++c->launches, k_b_start<<<grid2(c->G.nr + 1, c->G.nth + 1), dim3(BX, BY), 0, c->stream>>>(a);
  c->bh_ok = true;
}

bool filter_apart(const pic_ctx *c) { return c->d.n_filt > FUSE_FILT; }

void fields_flux(pic_ctx *c) {
  EnsFieldArg a;
  ens_fill_field_arg(c, &a);
  const Grid &G = c->G;
  ++c->launches, launch_on(c->stream, c->overlap, k_flux_from_acc, grid2(G.nr + 2 * G.g + 1, G.nth + 1), dim3(BX, BY), a);
}

void fields_filter(pic_ctx *c) {
  EnsFieldArg a;
  ens_fill_field_arg(c, &a);
  const Grid &G = c->G;
  const dim3 gr = grid2(G.nr + 2 * G.g + 1, G.nth + 1);
  for (int p = 0; p < c->d.n_filt; ++p)
    for (int k = 0; k < 3; ++k)
      ++c->launches, launch_on(c->stream, c->overlap, k_filter, gr, dim3(BX, BY), G, (p & 1) ? a.Ftmp[k] : a.Fin[k],
                               (p & 1) ? a.Fin[k] : a.Ftmp[k], k == 1);
}

void fields_e_step(pic_ctx *c) {
  EnsFieldArg a;
  ens_fill_field_arg(c, &a);
  const unsigned nb = (unsigned)ens_blocks(c, ENS_BAND);
  if (c->d.precision == PIC_FP32) ++c->launches, launch_on(c->stream, c->overlap, k_e_step<true>, nb, dim3(BX, BY), a);
  else ++c->launches, launch_on(c->stream, c->overlap, k_e_step<false>, nb, dim3(BX, BY), a);
}

void fields_b_step(pic_ctx *c, bool sigma) {
  EnsFieldArg a;
  ens_fill_field_arg(c, &a);
  a.jump = sigma_jump(c, (c->step + 1) * c->G.dt);
  const int sg = sigma && c->d.inject ? 1 : 0;
  const unsigned nb = (unsigned)ens_blocks(c, ENS_BAND);
  if (c->d.precision == PIC_FP32) ++c->launches, launch_on(c->stream, c->overlap, k_b_step<true>, nb, dim3(BX, BY), a, sg);
  else ++c->launches, launch_on(c->stream, c->overlap, k_b_step<false>, nb, dim3(BX, BY), a, sg);
  // the filtered flux stays in F (pic_get_flux), the cleared deposit in Ft
  if (a.Fout[0] != c->F[0])
    for (int k = 0; k < 3; ++k) std::swap(c->F[k], c->Ft[k]);
}

void fields_copy32(pic_ctx *c) {
  const Grid &G = c->G;
  ++c->launches, k_copy32<<<grid2(G.nr + 2 * G.g + 1, G.nth + 2), dim3(BX, BY), 0, c->stream>>>(
      G, c->f[0], c->f[1], c->f[2], c->f[3], c->f[4], c->f[5], c->f32[0], c->f32[1], c->f32[2], c->f32[3], c->f32[4],
      c->f32[5]);
}

void fields_fill_ghosts(pic_ctx *c) {
  const Grid &G = c->G;
  ++c->launches, k_axis_ghosts<<<(G.nr + 1 + 127) / 128, 128, 0, c->stream>>>(G, c->f[ETH], c->f[BR], c->f[BPH]);
  if (c->d.precision == PIC_FP32) fields_copy32(c);
}

void filter_charge(pic_ctx *c) {
  const Grid &G = c->G;
  const int n = c->d.n_filt;
  const dim3 gr = grid2(G.nr + 2 * G.g + 1, G.nth + 1);
  if (n == 0) return;
  if (n <= FUSE_FILT) {
    ++c->launches, k_filter_tile<<<gr, dim3(BX, BY), 0, c->stream>>>(G, c->Q, c->Qt, n);
    std::swap(c->Q, c->Qt);
  }
  for (int p = 0; n > FUSE_FILT && p < n; ++p) {
    ++c->launches, k_filter<<<gr, dim3(BX, BY), 0, c->stream>>>(G, c->Q, c->Qt, 0);
    std::swap(c->Q, c->Qt);
  }
}

void inject(pic_ctx *c, double t, bool have_sigma) {
  const Grid &G = c->G;
  const int npp = c->d.pairs_per_cell, ns = c->d.inject_smooth;
  long long *smax = c->d_cnt + CNT_SMAX;
  double *a = c->sig, *b = c->sig + (G.nth + 1);
  const int tb = (G.nth + 127) / 128;
  if (!have_sigma) {  // a radial slab: after the exchange of the step's fields
    cudaMemsetAsync(smax, 0, sizeof(long long), c->stream);
    ++c->launches, k_inject_sigma<<<tb, 128, 0, c->stream>>>(G, c->f[ER], sigma_jump(c, t), a, ns ? nullptr : smax);
  }
  for (int p = 0; p < ns; ++p) {
    ++c->launches, launch_on(c->stream, c->overlap, k_inject_smooth, tb, 128, G.nth, a, b, p == ns - 1 ? smax : nullptr);
    double *x = a; a = b; b = x;
  }
  const InjectRule R{c->d.inject, npp, c->d.f_inj, c->d.inject_q, c->d.inject_seed, (uint64_t)c->step};
  const int64_t nslots = (int64_t)G.nth * npp * 2;
  const int blocks = (int)((nslots + 255) / 256);
  if (c->d.precision == PIC_FP32)
    ++c->launches, launch_on(c->stream, c->overlap, k_inject_write<true>, blocks, 256, G, a, smax, c->p64, c->p32, c->n_used, c->next_id, R,
                                                        c->d_cnt + CNT_INJECTED, c->d_cnt + CNT_CAPPED, c->qexp);
  else
    ++c->launches, launch_on(c->stream, c->overlap, k_inject_write<false>, blocks, 256, G, a, smax, c->p64, c->p32, c->n_used, c->next_id, R,
                                                         c->d_cnt + CNT_INJECTED, c->d_cnt + CNT_CAPPED, c->qexp);
  c->n_used += nslots;
  c->next_id += nslots;
}

// Spin-down luminosity (Sec. 5.3, Fig. 7d): the radial Poynting flux
// (E x B)_r of the total field, plasma plus analytic at time t, through the
// sphere of node radius r_i, one block per interior row.  On the sphere the
// meridional cell j carries E_th(i, j+1/2); B_ph (at i -+ 1/2), E_ph (at the
// nodes j, j+1) and B_th (at i -+ 1/2 and j, j+1) are averaged to the cell's
// centre; each cell adds (E_th B_ph - E_ph B_th) 2 pi r_i^2 (cos th_j -
// cos th_{j+1}).  L[0] and L[nr] are 0.
__global__ void k_luminosity(Grid G, const double *__restrict__ Et, const double *__restrict__ Ep,
                             const double *__restrict__ Bt, const double *__restrict__ Bp, double t, double *L) {
  __shared__ double sm[32];
  const Metric &m = G.m;
  const int i = blockIdx.x;
  double s = 0.0;
  if (i >= 1 && i < G.nr) {
    const double r = m.r_n[i + G.PI], ring = 2.0 * PI_D * r * r;
    const Vac<double> V{G.vacuum, G.b0, G.r_min, omega_at(G.omega, G.t_spin, t)};
    for (int j = threadIdx.x; j < G.nth; j += blockDim.x) {
      const int cj = j + G.PJ;
      double E[3], B[3];
      vacuum_field<double>(V, r, m.sin_tb[cj], m.cos_tb[cj], false, E, B);
      const size_t o = gidx(G, i, j);
      const double et = Et[o] + E[1];
      const double bp = 0.5 * (Bp[o - G.LD] + Bp[o]) + B[2];
      const double ep = 0.5 * (Ep[o] + Ep[o + 1]) + E[2];
      const double bt = 0.25 * (Bt[o - G.LD] + Bt[o] + Bt[o - G.LD + 1] + Bt[o + 1]) + B[1];
      s += (et * bp - ep * bt) * ring * m.vol_t_h[cj];
    }
  }
  for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += sm[w];
    L[i] = tot;
  }
}

void luminosity(pic_ctx *c, double t, double *L) {
  const Grid &G = c->G;
  ++c->launches, k_luminosity<<<G.nr + 1, 256, 0, c->stream>>>(G, c->f[ETH], c->f[EPH], c->f[BTH], c->f[BPH], t, L);
}

void gauss_rows(pic_ctx *c, int ilo, int imax, bool snapshot) {
  const Grid &G = c->G;
  if (imax < ilo) return;
  ++c->launches, k_gauss<<<grid2(imax - ilo + 1, G.nth + 1), dim3(BX, BY), 0, c->stream>>>(
      G, c->f[ER], c->f[ETH], c->Q, c->Qa, c->gsnap, ilo, imax, snapshot ? 1 : 0, c->d_cnt + CNT_GMAX,
      c->d_cnt + CNT_QMAX);
}

void field_energy_rows(pic_ctx *c, int imax) {
  const Grid &G = c->G;
  ++c->launches, k_field_energy<<<grid2(G.nr + 1, G.nth + 1), dim3(BX, BY), 0, c->stream>>>(
      G, c->f[0], c->f[1], c->f[2], c->f[3], c->f[4], c->f[5], imax, c->d_acc + ACC_FIELD);
}

void moments(pic_ctx *c, bool snapshot, pic_moments *out) {
  const Grid &G = c->G;
  if (c->d.precision == PIC_FP32) charge32(c);
  else charge64(c);
  filter_charge(c);
  int L = c->d.absorb_profile == PIC_ABSORB_NONE ? 0 : c->d.absorb_cells;
  int imax = G.nr - L - 1;
  cudaMemsetAsync(c->d_cnt + CNT_GMAX, 0, 2 * sizeof(long long), c->stream);
  if (imax >= 1)
    ++c->launches, k_gauss<<<grid2(imax, G.nth + 1), dim3(BX, BY), 0, c->stream>>>(G, c->f[ER], c->f[ETH], c->Q, c->Qa, c->gsnap,
                                                                    1, imax, snapshot ? 1 : 0, c->d_cnt + CNT_GMAX,
                                                                    c->d_cnt + CNT_QMAX);
  if (snapshot) { c->have_snap = true; return; }
  cudaMemsetAsync(c->d_acc, 0, ACC_N * sizeof(double), c->stream);
  cudaMemsetAsync(c->d_cnt + CNT_LIVE, 0, sizeof(long long), c->stream);
  ++c->launches, k_field_energy<<<grid2(G.nr + 1, G.nth + 1), dim3(BX, BY), 0, c->stream>>>(
      G, c->f[0], c->f[1], c->f[2], c->f[3], c->f[4], c->f[5], G.nr, c->d_acc + ACC_FIELD);
  if (c->d.precision == PIC_FP32) reduce_particles32(c);
  else reduce_particles64(c);
  long long cnt[CNT_N];
  double acc[ACC_N];
  cudaMemcpyAsync(cnt, c->d_cnt, sizeof cnt, cudaMemcpyDeviceToHost, c->stream);
  cudaMemcpyAsync(acc, c->d_acc, sizeof acc, cudaMemcpyDeviceToHost, c->stream);
  cudaStreamSynchronize(c->stream);
  double gmax, qmax;
  memcpy(&gmax, &cnt[CNT_GMAX], sizeof(double));
  memcpy(&qmax, &cnt[CNT_QMAX], sizeof(double));
  out->live = cnt[CNT_LIVE];
  out->deleted = cnt[CNT_DELETED];
  out->injected = cnt[CNT_INJECTED];
  out->inject_capped = cnt[CNT_CAPPED];
  out->axis_ties = cnt[CNT_TIES];
  out->step = c->step;
  out->dt = G.dt;
  out->time = c->step * G.dt;
  out->kinetic_energy = acc[ACC_KIN];
  out->field_energy = acc[ACC_FIELD];
  out->total_charge = acc[ACC_CHARGE];
  out->gauss_residual = (!c->have_snap) ? -1.0 : (qmax > 0 ? gmax / qmax : gmax);
}

}  // namespace pic
