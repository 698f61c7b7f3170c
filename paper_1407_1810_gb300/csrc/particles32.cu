// particles32.cu -- the FP32 cell+offset particle path (the hot path) around its
// tile kernel (tiles_one.cu, tiles_two.cu): the particles are kept binned by tiles
// of TI x TJ cells (counting sort every sort_interval steps, which drops the
// deleted ones), each tile's bin is cut into work units, one CTA each, and a step
// launches the tile kernel's form for the grid over them.  Also: the node charge
// and the particle sums of the diagnostics, the batched launches and the batched
// sort of ensemble members.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "tiles32.cuh"

namespace pic {

using namespace t32;

namespace {

// Self-test of the bounded wait above: thread 0 of a one-warp block arms an
// mbarrier for 16 bytes that no copy will deliver (arrive_first = 0) or
// completes its phase itself first (arrive_first = 1), then waits at most
// `limit` polls; on giving up it sets ERR_TIMEOUT, as the tile kernel does.
// Nothing is in flight, so the block can leave after a timeout.
__global__ void k_wait_selftest(long long limit, int arrive_first, int *err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar)));
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (arrive_first) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar)) : "memory");
  } else {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&bar)), "r"(16u) : "memory");
  }
  if (!window_wait(&bar, limit)) atomicOr(err, ERR_TIMEOUT);
}

// ---- counting sort into tile bins (drops removed particles) ---------------
// Bins are numbered cell by cell, tile-major: key = tile * tc + cell index
// inside the tile; removed particles go to the last bin, ntiles * tc.  Keys
// fit in 32 bits: at most (nr + 2g + TI) (nth + TJ) cells with nr, nth <= 32000.
// Two kinds of sort share the bins:
//  - mixing (after particles are loaded or the tile shape changes): by cell,
//    each tile's bin stored transposed (transposed_slot below), so the lanes
//    of a warp step particles of different cells;
//  - keeping (every later sort): by tile only (all of a tile's particles in
//    bin tile * tc), each tile's particles in their previous relative order,
//    which keeps them mixed: particles move a few cells between sorts.
__device__ inline int cell_key(const Args32 &A, uint32_t cell, float qw) {
  if (qw == 0.f) return A.ntiles * A.tc;
  const int ci = (int)(cell >> 16) - CELL_BIAS - A.row0, cj = (int)(cell & 0xffffu);
  const int tile = ((ci / A.ti) * A.ntj + cj / A.tj) * A.tc;
  return A.mix ? tile + (ci % A.ti) * A.tj + cj % A.tj : tile;
}

__device__ __forceinline__ void hist_block(const Args32 &A, const Parts32 &P, int64_t n, int64_t *count,
                                           unsigned blk) {
  const int64_t k = blk * (int64_t)blockDim.x + threadIdx.x;
  const int key = k < n ? cell_key(A, P.cell[k], P.qw[k]) : -1;
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  const int lane = threadIdx.x & 31;
  if (key >= 0 && lane == __ffs(peers) - 1)
    atomicAdd(reinterpret_cast<unsigned long long *>(count + key), (unsigned long long)__popc(peers));
}

__global__ void k_hist(Args32 A, Parts32 P, int64_t n, int64_t *count) { hist_block(A, P, n, count, blockIdx.x); }

// exclusive scan of nb counts by one block of 1024 threads (the top level of
// the scan below); count becomes the cursor and start[nb] the total
__device__ __forceinline__ void scan_bins_block(int64_t *count, int64_t *start, int nb) {
  __shared__ int64_t part[1024];
  const int t = threadIdx.x;
  const int per = (nb + 1023) / 1024, a = t * per, b = min(nb, a + per);
  int64_t s = 0;
  for (int k = a; k < b; ++k) s += count[k];
  part[t] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    int64_t v = t >= off ? part[t - off] : 0;
    __syncthreads();
    part[t] += v;
    __syncthreads();
  }
  int64_t run = part[t] - s;
  for (int k = a; k < b; ++k) {
    const int64_t c = count[k];
    start[k] = run;
    count[k] = run;
    run += c;
  }
  if (t == 1023) start[nb] = part[1023];
}

__global__ void k_scan_bins(int64_t *count, int64_t *start, int nb) {
  follow();
  scan_bins_block(count, start, nb);
}

// block sum of 256 values (all threads get it)
__device__ inline int64_t block_sum256(int64_t v, int64_t *sm) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  int64_t t = 0;
  for (int w = 0; w < 8; ++w) t += sm[w];
  __syncthreads();
  return t;
}

// multi-block exclusive scan over nb bins, SCAN_CHUNK bins per block of 256
// threads: sums of each chunk, a one-block scan of the sums, then each chunk
// scanned from its offset (16 consecutive bins per thread)
__device__ __forceinline__ void scan_sums_block(const int64_t *count, int64_t nb, int64_t *sums, unsigned blk) {
  __shared__ int64_t sm[8];
  const int64_t a = blk * (int64_t)SCAN_CHUNK;
  int64_t s = 0;
  for (int k = threadIdx.x; k < SCAN_CHUNK; k += 256)
    if (a + k < nb) s += count[a + k];
  s = block_sum256(s, sm);
  if (threadIdx.x == 0) sums[blk] = s;
}

__global__ void k_scan_sums(const int64_t *count, int64_t nb, int64_t *sums) {
  follow();
  scan_sums_block(count, nb, sums, blockIdx.x);
}

__device__ __forceinline__ void scan_apply_block(int64_t *count, int64_t *start, int64_t nb, const int64_t *offs,
                                                 int nblk, unsigned blk) {
  __shared__ int64_t sm[8];
  const int64_t a = blk * (int64_t)SCAN_CHUNK + threadIdx.x * 16;
  int64_t v[16], s = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) { v[i] = a + i < nb ? count[a + i] : 0; s += v[i]; }
  // exclusive scan of the 256 thread sums
  int64_t x = s;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sm[w] = x;
  __syncthreads();
  int64_t base = offs[blk];
  for (int k = 0; k < w; ++k) base += sm[k];
  int64_t run = base + x - s;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    if (a + i < nb) { start[a + i] = run; count[a + i] = run; }
    run += v[i];
  }
  if (blk == 0 && threadIdx.x == 0) start[nb] = offs[nblk];
}

__global__ void k_scan_apply(int64_t *count, int64_t *start, int64_t nb, const int64_t *offs, int nblk) {
  follow();
  scan_apply_block(count, start, nb, offs, nblk, blockIdx.x);
}

// work units of each tile: ceil(n_t / unit) of even size, none for an empty tile
__device__ __forceinline__ void unit_count_at(int t, const int64_t *start, int tc, int ntiles, int64_t unit,
                                              int64_t *ucount) {
  if (t >= ntiles) return;
  const int64_t n = start[(int64_t)(t + 1) * tc] - start[(int64_t)t * tc];
  ucount[t] = (n + unit - 1) / unit;
}

__global__ void k_unit_count(const int64_t *start, int tc, int ntiles, int64_t unit, int64_t *ucount) {
  follow();
  unit_count_at(blockIdx.x * blockDim.x + threadIdx.x, start, tc, ntiles, unit, ucount);
}

// the unit list from the exclusive scan of the counts (uoff[ntiles] = total)
__device__ __forceinline__ void unit_fill_at(int t, const int64_t *uoff, int ntiles, long long *units) {
  if (t >= ntiles) return;
  for (int64_t u = uoff[t]; u < uoff[t + 1]; ++u) units[u] = ((long long)t << 32) | (long long)(u - uoff[t]);
}

__global__ void k_unit_fill(const int64_t *uoff, int ntiles, long long *units) {
  follow();
  unit_fill_at(blockIdx.x * blockDim.x + threadIdx.x, uoff, ntiles, units);
}

// Order inside a tile's bin.  The counting sort yields the tile's particles
// cell by cell; they are stored transposed: the cell-ordered sequence fills
// the columns of a matrix with trw columns, and the bin holds its rows.  The
// lanes of a warp, which step consecutive slots, then hold particles about
// n / trw apart in cell order: different cells, so their deposits rarely hit
// the same shared-memory address in one instruction.  64 columns where a warp
// steps 64 particles at once, 16 (the rows of a tile) where it steps 32.  (The
// results do not depend on the order: the deposit sums are exact.)  q:
// position in cell order, n: particles in the bin; returns the slot.
__device__ inline int64_t transposed_slot(int64_t q, int64_t n, int trw) {
  const int64_t R = (n + trw - 1) / trw;  // rows
  const int64_t L = n - (R - 1) * trw;    // columns of R elements; the others hold R - 1
  int64_t c, r;
  if (q < L * R) { c = q / R; r = q - c * R; }
  else { const int64_t u = q - L * R; c = L + u / (R - 1); r = u - (c - L) * (R - 1); }
  return r * trw + c;
}

__device__ __forceinline__ void scatter_block(const Args32 &A, const Parts32 &S, const Parts32 &D, int64_t n,
                                              int64_t *cursor, unsigned blk) {
  const int64_t k = blk * (int64_t)blockDim.x + threadIdx.x;
  const int trash = A.ntiles * A.tc;
  // every load issued before the cursor atomic, whose round trip they overlap
  const int64_t kk = k < n ? k : 0;
  const uint32_t cell = S.cell[kk];
  const float dx = S.dx[kk], dy = S.dy[kk], ur = S.ur[kk], ut = S.ut[kk], up = S.up[kk], qw = S.qw[kk];
  const int64_t id = S.id[kk];
  const int key = k < n ? cell_key(A, cell, qw) : -1;
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
  unsigned long long base = 0;
  if (key >= 0 && key < trash && lane == leader)
    base = atomicAdd(reinterpret_cast<unsigned long long *>(cursor + key), (unsigned long long)__popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (key < 0 || key >= trash) return;
  int64_t d = (int64_t)base + __popc(peers & ((1u << lane) - 1u));
  if (A.mix) {
    const int t = key / A.tc;
    const int64_t t0 = A.start[(int64_t)t * A.tc], t1 = A.start[(int64_t)(t + 1) * A.tc];
    d = t0 + transposed_slot(d - t0, t1 - t0, A.trw);
  }
  D.cell[d] = cell; D.dx[d] = dx; D.dy[d] = dy;
  D.ur[d] = ur; D.ut[d] = ut; D.up[d] = up;
  D.qw[d] = qw; D.id[d] = id;
}

__global__ void k_scatter_cells(Args32 A, Parts32 S, Parts32 D, int64_t n, int64_t *cursor) {
  follow();
  scatter_block(A, S, D, n, cursor, blockIdx.x);
}

// ---- the tile sort of several ensemble members at once ---------------------
// One member's sort as the batched kernels read it (device table): the same
// arrays and the same kernel bodies as sort32, every phase one launch for all
// members due, and one read-back of their live counts, unit counts and error
// words.
struct EnsSortArg {
  Args32 A;                   // keys and tile geometry; A.mix: this sort's order
  Parts32 S, D;               // particles before and after the sort
  int64_t n;                  // particles before the sort
  int64_t *count, *start, *bsum;
  int64_t nbins;
  int nblk, ublk, ntiles, tc;
  int64_t *ucount, *usum;
  long long *units;
  int64_t unit;
  const int *err;
  int64_t *out;               // live, units, error bits (for the host)
};

__global__ void k_ens_sort_zero(const EnsSortArg *__restrict__ tab, EnsList L) {
  const int2 e = L.blk[blockIdx.x];
  const EnsSortArg &E = tab[e.x];
  const int64_t q = (int64_t)e.y * blockDim.x + threadIdx.x;
  if (q <= E.nbins) E.count[q] = 0;
}
__global__ void k_ens_hist(const EnsSortArg *__restrict__ tab, EnsList L) {
  const int2 e = L.blk[blockIdx.x];
  const EnsSortArg &E = tab[e.x];
  hist_block(E.A, E.S, E.n, E.count, (unsigned)e.y);
}
// units = 0: the scan of the bin counts; 1: of the per-tile unit counts
__global__ void k_ens_scan_sums(const EnsSortArg *__restrict__ tab, EnsList L, int units) {
  const int2 e = L.blk[blockIdx.x];
  const EnsSortArg &E = tab[e.x];
  if (units) scan_sums_block(E.ucount, E.ntiles, E.usum, (unsigned)e.y);
  else scan_sums_block(E.count, E.nbins, E.bsum, (unsigned)e.y);
}
__global__ void k_ens_scan_bins(const EnsSortArg *__restrict__ tab, EnsList L, int units) {
  const EnsSortArg &E = tab[L.blk[blockIdx.x].x];
  if (units) scan_bins_block(E.usum, E.usum + E.ublk + 1, E.ublk);
  else scan_bins_block(E.bsum, E.bsum + E.nblk + 1, E.nblk);
}
__global__ void k_ens_scan_apply(const EnsSortArg *__restrict__ tab, EnsList L, int units) {
  const int2 e = L.blk[blockIdx.x];
  const EnsSortArg &E = tab[e.x];
  if (units) scan_apply_block(E.ucount, E.ucount, E.ntiles, E.usum + E.ublk + 1, E.ublk, (unsigned)e.y);
  else scan_apply_block(E.count, E.start, E.nbins, E.bsum + E.nblk + 1, E.nblk, (unsigned)e.y);
}
__global__ void k_ens_scatter(const EnsSortArg *__restrict__ tab, EnsList L) {
  const int2 e = L.blk[blockIdx.x];
  const EnsSortArg &E = tab[e.x];
  scatter_block(E.A, E.S, E.D, E.n, E.count, (unsigned)e.y);
}
__global__ void k_ens_unit_count(const EnsSortArg *__restrict__ tab, EnsList L) {
  const int2 e = L.blk[blockIdx.x];
  const EnsSortArg &E = tab[e.x];
  unit_count_at(e.y * blockDim.x + threadIdx.x, E.start, E.tc, E.ntiles, E.unit, E.ucount);
}
__global__ void k_ens_unit_fill(const EnsSortArg *__restrict__ tab, EnsList L) {
  const int2 e = L.blk[blockIdx.x];
  const EnsSortArg &E = tab[e.x];
  unit_fill_at(e.y * blockDim.x + threadIdx.x, E.ucount, E.ntiles, E.units);
}
__global__ void k_ens_sort_out(const EnsSortArg *__restrict__ tab, int m) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  const EnsSortArg &E = tab[k];
  E.out[0] = E.start[(int64_t)E.ntiles * E.tc];
  E.out[1] = E.ucount[E.ntiles];
  E.out[2] = *E.err;
}

// ---- node charge (diagnostics) ----------------------------------------------
// Positive and negative charge at every node.  A particle's |qw| in units of
// 2^(e - QFIX) (e: the context's charge exponent) is an integer, its offsets are
// 64-bit fractions, and the four area weights' shares are 64-bit products rounded
// down that add up to the whole charge: sums of integers, in any order the same.
// A share is off by up to 3 units, 3 2^-54 of the particle's charge while that is
// at least 2^(e - QRANGE).  Smaller charges (other species, pairs injected where
// the surface charge is small, an exponent that flux_quantum raised) take FP64
// products and FP64 atomics, in a kernel of their own that leaves at once where
// there are none.  Q is the difference of the signs' sums and sum |qw| their sum,
// rounded once to FP64; the small charges are added to that.
//
// A block takes a work unit of the tile kernel (one tile's particles, which are
// mixed across its cells) and sums three 20-bit limbs a node in shared memory with
// native 32-bit atomics, flushed before they can overflow; particles outside the
// window add to global memory.  5e7 particles of a 1024^2 rotator: 4.6 ms with
// FP64 global atomics for all, bound by the atomics and the FP64 pipe; 0.54 ms so,
// and 0.66 ms with charges that vary as |cos theta|, 3 % of them small.  (18-bit
// limbs, half the flushes and no small charges told apart: 0.52.  19-bit, QRANGE 3:
// 0.52, and 0.89 with 12 % small; 21-bit, QRANGE 8: 0.57 and 0.66.  The small
// charges' atomics in the tile kernel: 0.04 more for all.)
constexpr int QFIX = 59, QLIMB = 20, QSPLIT = 30;  // fraction bits; limb; low part of a global sum
constexpr int QRANGE = 5;
constexpr int QFLUSH = (1 << 12) / NT;               // passes of NT particles: 2^12 terms of less than 2^20
struct ChargePlanes {
  unsigned long long *hi[2], *lo[2];  // sums of the high and the low QSPLIT bits, of positive and negative charge
  long long *list, cap;               // the slots of the first cap charges below 2^(e - QRANGE)
  long long *small, *next;            // all of them counted; the next call's counter, which this call clears
};

// w in [0, 1) as a fraction of 2^64 (exact from 2^-40 on)
__device__ __forceinline__ unsigned long long frac64(float w) {
  const unsigned b = __float_as_uint(w), ex = b >> 23;
  const unsigned long long m = (b & 0x7fffffu) | (ex ? 0x800000u : 0u);
  return ex >= 86 ? m << (ex - 86) : (ex + 64 > 86 ? m >> (86 - ex) : 0ull);
}

// whether a charge lies in [2^(e - QRANGE), 2^e], and it in units of 2^(e - QFIX) if so
__device__ __forceinline__ bool charge_fits(float q, int e) {
  return (unsigned)((int)(__float_as_uint(q) >> 23 & 0xffu) - 127 - (e - QRANGE)) <= (unsigned)QRANGE;
}
__device__ __forceinline__ unsigned long long charge_units(float q, int e) {
  const unsigned b = __float_as_uint(q) & 0x7fffffffu;
  return (unsigned long long)((b & 0x7fffffu) | 0x800000u) << ((int)(b >> 23) - 150 + QFIX - e);  // q = m 2^(exponent - 150)
}

// particle k into the list of small charges (a list that has run over needs no
// more of them)
__device__ __forceinline__ void charge_list(const ChargePlanes &C, int64_t k) {
  if (*(volatile long long *)C.small > C.cap) return;
  const long long at = (long long)atomicAdd((unsigned long long *)C.small, 1ull);
  if (at < C.cap) C.list[at] = k;
}

struct ChargeShare {
  unsigned long long t[4];  // nodes (i, j), (i + 1, j), (i, j + 1), (i + 1, j + 1)
};
__device__ __forceinline__ ChargeShare charge_share(unsigned long long U, float dx, float dy) {
  const unsigned long long W1 = frac64(dx), W2 = frac64(dy);
  const unsigned long long a = __umul64hi(U, W1), b = __umul64hi(U, W2), ab = __umul64hi(a, W2);
  return ChargeShare{{U - a - b + ab, a - ab, b - ab, ab}};
}

template <int TI, int TJ>
__global__ void __launch_bounds__(NT) k_charge_tiles(Args32 A, Parts32 P, ChargePlanes C) {
  constexpr int WJ = Win<TI, TJ>::WJ, WN = Win<TI, TJ>::WN;
  __shared__ unsigned lim[2][3][WN];
  const int e = qexp_value(A.qexp);
  const unsigned blk = blockIdx.x;
  const bool binned = blk < (uint64_t)A.nunits;
  int64_t b0, b1;
  int i0 = 0, j0 = 0;
  if (binned) {
    int t;
    unit_range(A, A.units[blk], t, b0, b1);
    if (b1 <= b0) return;
    i0 = A.row0 + (t / A.ntj) * TI;
    j0 = (t % A.ntj) * TJ;
    for (int k = threadIdx.x; k < 6 * WN; k += NT) (&lim[0][0][0])[k] = 0;
    __syncthreads();
  } else {
    b0 = A.sorted_end + (int64_t)(blk - A.nunits) * NT;
    b1 = min(A.n_used, b0 + NT);
  }
  const int wi0 = i0 - H - 1, wj0 = j0 - H - 1;
  int pass = 0;
  for (int64_t base = b0; base < b1; base += NT) {
    const int64_t k = base + threadIdx.x;
    const float q = k < b1 ? P.qw[k] : 0.f;
    if (q != 0.f) {
      const uint32_t c = P.cell[k];
      int ci = (int)(c >> 16) - CELL_BIAS, cj = (int)(c & 0xffffu);
      const float dx = P.dx[k];
      float dy = P.dy[k];
      if (dy >= 1.f) { dy = 0.f; ++cj; }  // on the south axis
      const int sg = q < 0.f;
      const bool fits = charge_fits(q, e);
      if (!fits) charge_list(C, k);
      const ChargeShare s = charge_share(fits ? charge_units(q, e) : 0ull, dx, dy);
      if (binned && ci >= i0 - H && ci < i0 + TI + H && cj >= j0 - H && cj < j0 + TJ + H + 1) {
        const int o = (ci - wi0) * WJ + (cj - wj0);
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const int w = o + (n & 1) * WJ + (n >> 1);
          atomicAdd(&lim[sg][0][w], (unsigned)(s.t[n] & ((1u << QLIMB) - 1)));
          atomicAdd(&lim[sg][1][w], (unsigned)(s.t[n] >> QLIMB) & ((1u << QLIMB) - 1));
          atomicAdd(&lim[sg][2][w], (unsigned)(s.t[n] >> (2 * QLIMB)));
        }
      } else {
        const size_t o = pidx(A, ci, cj);
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const size_t w = o + (n & 1) * (size_t)A.LD + (n >> 1);
          if (!s.t[n]) continue;
          atomicAdd(C.hi[sg] + w, s.t[n] >> QSPLIT);
          atomicAdd(C.lo[sg] + w, s.t[n] & ((1ull << QSPLIT) - 1));
        }
      }
    }
    if (binned && (++pass == QFLUSH || base + NT >= b1)) {
      pass = 0;
      __syncthreads();
      for (int w = threadIdx.x; w < 2 * WN; w += NT) {
        const int sgn = w >= WN, n = sgn ? w - WN : w;
        const unsigned long long l0 = lim[sgn][0][n], l1 = lim[sgn][1][n], l2 = lim[sgn][2][n];
        if (l0 | l1 | l2) {  // l2 2^40 + l1 2^20 + l0 at QSPLIT = 30 bits
          const size_t o = pidx(A, wi0 + n / WJ, wj0 + n % WJ);
          constexpr int R = QSPLIT - QLIMB;
          atomicAdd(C.hi[sgn] + o, (l2 << (QLIMB - R)) + (l1 >> R));
          atomicAdd(C.lo[sgn] + o, ((l1 & ((1ull << R) - 1)) << QLIMB) + l0);
          lim[sgn][0][n] = lim[sgn][1][n] = lim[sgn][2][n] = 0;
        }
      }
      __syncthreads();
    }
  }
}

// the planes of a context's ghost band to FP64: Q and sum |qw|.  Q and Qa may
// be two of the planes (each node is read before it is written); the plane
// borrowed from the flux accumulators is cleared again.
__global__ void k_charge_finish(Grid G, const long long *qexp, ChargePlanes C, unsigned long long *borrowed,
                                double *Q, double *Qa) {
  follow();
  if ((blockIdx.x | blockIdx.y | threadIdx.x | threadIdx.y) == 0) *C.next = 0;
  const int i = -G.g + (int)(blockIdx.y * 8 + threadIdx.y), j = blockIdx.x * 32 + threadIdx.x;
  if (i > G.nr + G.g || j > G.nth) return;
  const size_t o = gidx(G, i, j);
  const __int128 p = ((__int128)C.hi[0][o] << QSPLIT) + C.lo[0][o], n = ((__int128)C.hi[1][o] << QSPLIT) + C.lo[1][o];
  const int s = qexp_value(qexp) - QFIX;
  borrowed[o] = 0;
  Q[o] = fixed_to_f64(p - n, s);
  Qa[o] = fixed_to_f64(p + n, s);
}

// the charges that k_charge_tiles left out, onto its results: those listed, or, of more than the
// list holds, all that a pass over the charges finds
__device__ __forceinline__ void charge_small(const Args32 &A, const Parts32 &P, double *Q, double *Qa, int64_t k) {
  const uint32_t c = P.cell[k];
  const size_t o = pidx(A, (int)(c >> 16) - CELL_BIAS, (int)(c & 0xffffu)), LD = A.LD;
  const double q = P.qw[k], w1 = P.dx[k], w2 = P.dy[k], a = fabs(q);
  const double w[4] = {(1 - w1) * (1 - w2), w1 * (1 - w2), (1 - w1) * w2, w1 * w2};
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const size_t x = o + (n & 1) * LD + (n >> 1);
    atomicAdd(Q + x, q * w[n]);
    atomicAdd(Qa + x, a * w[n]);
  }
}

__global__ void k_charge_small(Args32 A, Parts32 P, ChargePlanes C, double *Q, double *Qa) {
  follow();
  const int64_t n = *C.small, step = (int64_t)gridDim.x * blockDim.x;
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n <= C.cap) {
    for (; k < n; k += step) charge_small(A, P, Q, Qa, C.list[k]);
    return;
  }
  const int e = qexp_value(A.qexp);
  for (; k < A.n_used; k += 8 * step) {
    float q[8];  // the loads of eight before the first is looked at
#pragma unroll
    for (int r = 0; r < 8; ++r) q[r] = k + r * step < A.n_used ? P.qw[k + r * step] : 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (q[r] != 0.f && !charge_fits(q[r], e)) charge_small(A, P, Q, Qa, k + r * step);
  }
}

// h + l = a running FP32 sum and its exact rounding errors (Knuth's two-sum)
__device__ __forceinline__ void two_sum(float v, float &h, float &l) {
  const float s = __fadd_rn(h, v), z = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(v, z)));
  h = s;
}

// whether the largest of eight magnitudes leaves the error-carrying sum of the
// eight its range: no overflow, and what falls below the normal numbers is below
// 2^-53 of it
__device__ __forceinline__ bool sums_in_range(float m) {
  const unsigned b = __float_as_uint(m), lo = (127 - 70) << 23, hi = (127 + 120) << 23;
  return b == 0 || b - lo <= hi - lo;
}

// Kinetic energy, charge and live count.  Each particle's (gamma - 1) |qw| is
// formed in FP32 (gamma - 1 = u^2 / (1 + gamma): no cancellation) and summed
// in FP64 eight at a time, the eight through an error-carrying FP32 sum: a
// conversion and an addition on the FP64 pipe per particle and sum kept this
// pass FP64-bound (5e7 particles, 0.8 GB: 0.40 ms; 0.26 four, 0.24 eight at a
// time, 0.18 with the eight's loads issued together).  Eight next to an end of
// FP32's range (charges up to 2^100 are accepted) are added in FP64.
__global__ void k_reduce32(Parts32 P, int64_t n, double qm, double *acc, long long *live) {
  double kin = 0.0, ch = 0.0;
  long long l = 0;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += 8 * step) {
    // every load before the first sum; a free slot (charge 0) adds zeros
    // whatever its momentum holds
    float q[8], a[8], b[8], c[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int64_t x = k + r * step, y = x < n ? x : k;
      q[r] = P.qw[y]; a[r] = P.ur[y]; b[r] = P.ut[y]; c[r] = P.up[y];
      if (x >= n) q[r] = 0.f;
    }
    float e[8], em = 0.f, qm8 = 0.f;
    int m = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const float u2 = a[r] * a[r] + b[r] * b[r] + c[r] * c[r], w = fabsf(q[r]) * (u2 / (1.f + sqrtf(1.f + u2)));
      e[r] = q[r] != 0.f ? w : 0.f;
      em = fmaxf(em, e[r]);
      qm8 = fmaxf(qm8, fabsf(q[r]));
      m += q[r] != 0.f;
    }
    if (sums_in_range(em) && sums_in_range(qm8)) {
      float kh = 0.f, kl = 0.f, qh = 0.f, ql = 0.f;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        two_sum(e[r], kh, kl);
        two_sum(q[r], qh, ql);
      }
      kin += (double)kh + (double)kl;
      ch += (double)qh + (double)ql;
    } else {
      for (int r = 0; r < 8; ++r) {
        kin += e[r];
        ch += q[r];
      }
    }
    l += m;
  }
  block_sum3(kin / qm, ch, l, acc + ACC_KIN, acc + ACC_CHARGE, live);
}

constexpr int TRW_WARP = 32;

// The form of the tile kernel a context takes.  Two particles a thread are the
// faster form once there are tiles enough to fill the chip (1024 x 1024, 20
// steps: monopole of 6.3e7 particles 29.5 ms with one, 24.1 with two; rotator of
// 1e8 49.6 and 36.9; a whole run of 448 x 416: 8.05 and 7.38); on a small grid,
// bound by latency and by the grid phase, the two are closer (72 x 56 rotator
// 0.65 and 0.67 ms, 192 x 160 dipole 1.35 and 1.27, 250 x 231 monopole 1.51 and
// 1.41; 64-member ensemble, 40 steps: 49.1 and 46.8).  They round differently and
// neither is the less exact: against the FP64 path, over 78 runs of sparse plasmas
// (2000 to 60000 particles, grids on both sides of the line, six seeds each, 1 to
// 80 steps), the two-particle form's momenta are off by 0.5 to 1.07 times as
// much as the other's, its positions by 0.69 to 1.03, its fields by as much one
// way as the other.  The line is the largest grid of an ensemble's members (256 x
// 512): up to it results keep the bits of the one-particle form.  The grid alone
// decides, so that a member, a slab and a run of its own agree.
constexpr int64_t PACK_CELLS = 1 << 17;
bool use_packed(const pic_ctx *c) { return (int64_t)c->G.nr_glob * c->G.nth > PACK_CELLS; }

Args32 make_args(pic_ctx *c, double t) {
  const Grid &G = c->G;
  Args32 A;
  A.nr = G.nr; A.nth = G.nth; A.n_filt = G.n_filt; A.PI = G.PI; A.PJ = G.PJ; A.LD = G.LD;
  A.r_log = G.r_map == PIC_R_LOG; A.th_ea = G.th_map == PIC_TH_EQUAL_AREA;
  A.vacuum = G.vacuum; A.pusher = G.pusher;
  A.dxi = (float)G.dxi; A.inv_dxi = (float)(1.0 / G.dxi); A.dt = (float)G.dt; A.qm = (float)G.qm;
  A.dt_lo = (float)(G.dt - (double)A.dt);
  A.inv_dxi_lo = (float)(1.0 / G.dxi - (double)A.inv_dxi);
  A.hinv_dxi = 0.5f * A.inv_dxi; A.hinv_dxi_lo = 0.5f * A.inv_dxi_lo;
  A.hnth = 0.5f * (float)G.nth;
  A.k2_hi = (float)(G.nth / M_PI);
  A.k2_lo = (float)(G.nth / M_PI - (double)A.k2_hi);
  A.inv_nth = (float)(1.0 / G.nth); A.nth_f = (float)G.nth;
  A.qexp = c->qexp;
  A.ids = c->p32.id;
  A.ties = axis_ties(c);
  A.r_n = c->r_n32;
  A.ir_n = c->ir_n32;
  A.trw = use_packed(c) ? 2 * TRW_WARP : TRW_WARP / 2;
  A.th_n = c->th_n32;
  A.pi_nth = (float)(M_PI / G.nth);
  for (int k = 0; k < 6; ++k) A.f[k] = c->f32[k];
  for (int k = 0; k < 3; ++k) A.acc[k] = c->acc[k];
  A.err = c->d_err;
  A.cnt = c->d_cnt;
  A.row0 = c->tiles.row0; A.ntj = c->tiles.ntj; A.ntiles = c->tiles.ntiles;
  // Particles keep whole-grid rows in their packed cell.  A radial slab
  // (rows i0.. of a grid of nr_glob rows) indexes its arrays through a
  // padding offset shifted by i0, tests the conductors and removal against
  // the whole grid and places its tiles at its own rows; a whole grid has
  // i0 = 0 and nr_glob = nr, i.e. these are its own values.
  A.nr = G.nr_glob;
  A.PI = G.PI - G.i0;
  A.row0 = c->tiles.row0 + G.i0;
  A.ti = c->tiles.TI; A.tj = c->tiles.TJ; A.tc = c->tiles.tc;
  A.mix = 0;
  A.start = c->tiles.start;
  A.units = c->tiles.units;
  A.nunits = c->tiles.nunits;
  A.unit = c->tiles.unit;
  A.sorted_end = c->tiles.sorted_end;
  A.n_used = c->n_used;
  A.b0 = (float)G.b0; A.r_min = (float)G.r_min;
  A.b0_lo = (float)(G.b0 - (double)A.b0);
  A.qmdt = (float)(G.qm * G.dt);
  A.omega_t = (float)omega_at(G.omega, G.t_spin, t);
  A.nbrw = -(A.b0 * A.r_min * A.omega_t);
  return A;
}

}  // namespace

// The six field tensors of every tile shape (at context creation; the arrays
// do not move afterwards).  0 or -1 when the encoder is unavailable or
// rejects a map.
template <int TI, int TJ>
static int encode_maps(pic_ctx *c, void *fn, unsigned char *out) {
  using Enc = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                           const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                           CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  const Grid &G = c->G;
  const cuuint64_t dims[2] = {(cuuint64_t)G.LD, (cuuint64_t)(c->grid_elems / G.LD)};
  const cuuint64_t strides[1] = {(cuuint64_t)G.LD * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)Box<TI, TJ>::WB, (cuuint32_t)Box<TI, TJ>::WI};
  const cuuint32_t estr[2] = {1, 1};
  TileMaps *M = reinterpret_cast<TileMaps *>(out);
  for (int k = 0; k < 6; ++k) {
    const CUresult r = reinterpret_cast<Enc>(fn)(&M->m[k], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, c->f32[k], dims, strides,
                                                 box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return -1;
  }
  return 0;
}

int tiles32_setup(pic_ctx *c) {
  static_assert(sizeof(TileMaps) <= sizeof(c->tile_maps[0]), "tensor-map storage");
  void *fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !fn)
    return -1;
  // the grid arrays' pitch must be a whole number of 16-byte units
  if ((c->G.LD * sizeof(float)) % 16 != 0 || (c->G.PJ - H - 1 - WOFF) % 4 != 0) return -1;
  if (encode_maps<16, 16>(c, fn, c->tile_maps[0]) || encode_maps<8, 32>(c, fn, c->tile_maps[1]) ||
      encode_maps<32, 8>(c, fn, c->tile_maps[2]))
    return -1;
  // a device copy for the batched ensemble kernel (the arrays never move)
  if (cudaMemcpy(c->d_tile_maps, c->tile_maps, sizeof c->tile_maps, cudaMemcpyHostToDevice) != cudaSuccess) return -1;
  return 0;
}

// the compile-time specialisation of the tile kernel a context takes (the
// monopole one turns each column's node angle by the offset with a short
// series: nth >= 32 keeps that angle below pi / 32)
static int tile_spec(const pic_ctx *c) {
  const pic_desc &d = c->d;
  return c->small_steps && d.r_map == PIC_R_LOG && d.pusher == PIC_VAY
             ? (d.th_map == PIC_TH_LINEAR && d.vacuum == PIC_VAC_MONOPOLE && d.nth >= 32 ? SPEC_MONOPOLE
                : d.th_map == PIC_TH_EQUAL_AREA && d.vacuum == PIC_VAC_MONOPOLE_ROTATOR ? SPEC_ROTATOR
                                                                                         : SPEC_GENERIC)
             : SPEC_GENERIC;
}

int64_t ens_tile_blocks(const pic_ctx *c) {
  if (c->n_used == 0) return 0;
  return c->tiles.nunits + (c->n_used - c->tiles.sorted_end + NT - 1) / NT;
}

void particles32(pic_ctx *c, double t) {
  if (c->n_used == 0) return;
  Args32 A = make_args(c, t);
  const int64_t blocks = ens_tile_blocks(c);
  const TileMaps &M = *reinterpret_cast<const TileMaps *>(c->tile_maps[c->d.tile_shape]);
  const int shape = c->tiles.TI == 8 ? 1 : (c->tiles.TI == 32 ? 2 : 0);
  ++c->launches;
  (use_packed(c) ? launch_two : launch_one)(tile_spec(c), shape, (unsigned)blocks, c->stream, c->overlap, A, c->p32, M);
}

}  // namespace pic

// The bounded device-side wait of the tile kernel, exercised on its own (see
// include/picsar.h): PIC_ETIMEOUT when the wait gave up, PIC_OK when it saw
// its phase complete.
extern "C" int pic_wait_selftest(int64_t polls, int32_t arrive_first, void *stream) {
  if (polls < 1) return pic_fail(PIC_EINVAL, "polls must be >= 1");
  cudaStream_t st = (cudaStream_t)stream;
  int *d = nullptr;
  PIC_CUDA(cudaMalloc((void **)&d, sizeof(int)));
  int h = 0;
  cudaError_t e = cudaMemsetAsync(d, 0, sizeof(int), st);
  if (e == cudaSuccess) {
    pic::k_wait_selftest<<<1, 32, 0, st>>>((long long)polls, arrive_first ? 1 : 0, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(d);
  if (e != cudaSuccess) return pic_cuda_check(e, "wait self-test");
  if (h & pic::ERR_TIMEOUT) return pic_fail(PIC_ETIMEOUT, "the bounded wait gave up (as intended when nothing arrives)");
  return PIC_OK;
}

namespace pic {

size_t ens_tile_arg_bytes() { return sizeof(EnsTileArg); }

// kind = 9 x packed + 3 x specialisation + tile shape (0: 16 x 16, 1: 8 x 32, 2: 32 x 8)
int ens_tile_kind(const pic_ctx *c) {
  const int shape = c->tiles.TI == 8 ? 1 : (c->tiles.TI == 32 ? 2 : 0);
  return 9 * (use_packed(c) ? 1 : 0) + 3 * tile_spec(c) + shape;
}

void ens_tile_arg(pic_ctx *c, double t, void *out) {
  EnsTileArg a;
  a.A = make_args(c, t);
  a.P = c->p32;
  const int shape = c->tiles.TI == 8 ? 1 : (c->tiles.TI == 32 ? 2 : 0);
  a.maps = reinterpret_cast<const CUtensorMap *>(c->d_tile_maps + (size_t)shape * sizeof(TileMaps));
  memcpy(out, &a, sizeof a);
}

// The tile launches of one step of an ensemble (members in batches of
// ENS_TILE_SLOTS, one kind after the other) touch different members: each but
// the first starts as soon as the one before it has its last blocks on the
// chip, and ends after it, so what follows waits for all of them.  Only the
// first waits for the step before it, by plain stream order; the later ones
// start after the first's blocks, hence after that wait too.
// 64 members, two launches a step: 50.2 -> 49.3 ms for 40 steps (the first's
// last, partly filled round of the chip is shared with the second).
int ens_tiles32(int kind, const void *args, const int64_t *blocks, int n, cudaStream_t s, bool first_of_step) {
  const EnsTileArg *T = static_cast<const EnsTileArg *>(args);
  const bool pack = kind >= 9;
  const int spec = kind % 9 / 3, shape = kind % 3;
  int launches = 0;
  static thread_local EnsTileBatch B;  // 20 KB: kept off the stack
  for (int first = 0; first < n; first += ENS_TILE_SLOTS) {
    const int m = std::min(ENS_TILE_SLOTS, n - first);
    B.n = m;
    B.off[0] = 0;
    for (int k = 0; k < m; ++k) {
      B.a[k] = T[first + k];
      B.off[k + 1] = B.off[k] + (int)blocks[first + k];
    }
    const unsigned g = (unsigned)B.off[m];
    (pack ? launch_ens_two : launch_ens_one)(spec, shape, g, s, !first_of_step || launches > 0, B);
    ++launches;
  }
  return launches;
}

// Particles per work unit of a context on its own.  The 152 SMs hold 608 CTAs
// at a time, so the kernel runs in rounds of 608 units: cutting each tile's
// bin into m even units takes about ceil(m tiles / 608) rounds of the passes a
// unit needs and its window and flush, worth 1.5 passes.  The m with the least
// is taken; the bound is a tenth above the even share, so that a tile a little
// fuller than the average is not cut once more.  At least 1 / 2432 of the
// particles: where they crowd in few tiles, four rounds are cut fine enough.
// (Steps alone, units of 1 / 1216 of the
// particles -> so: 20 steps of monopole 250 x 231 1.70 -> 1.65 ms, of dipole
// 192 x 160 1.31 -> 1.20, of rotator 72 x 56 0.84 either way; 19 of monopole
// 448 x 416 3.56 -> 3.47.)
// Members of an ensemble share the chip: their units follow the particles of
// all of them (64 members, 2.4e7 particles: 62 ms for 40 steps with units of
// 4096, 64 with 2048, 71 with 1024, 78 with 512).
// A unit is also what one CTA's 32-bit sums must hold: it never exceeds
// UNIT_ROOM particles (which no crowding can overflow), or 1 / 1216 of a larger
// run's.  On grids of one or a few tiles the cut goes beyond 64 pieces a tile, to
// four rounds of the chip (20 steps of 16 x 16 cells and 1e6 particles 2.67 ms
// with at most 64 pieces, 1.06 so; 4e6 10.0 and 3.0; 32 x 32 and 1e7 7.5 and 5.3).
constexpr int SLOTS = 4 * 152;
static int64_t unit_size(const pic_ctx *c) {
  const int64_t n = c->n_used;
  const int64_t room = std::max<int64_t>(UNIT_ROOM, (n + 2 * SLOTS - 1) / (2 * SLOTS));
  if (c->ens_particles > 0) {
    const int64_t u = (c->ens_particles + 8 * SLOTS - 1) / (8 * SLOTS);
    return std::min(room, std::max<int64_t>(2 * NT, (u + NT - 1) / NT * NT));
  }
  const Tiles &T = c->tiles;
  const int64_t tiles = (int64_t)((c->G.nr + T.TI - 1) / T.TI) * T.ntj;  // those of the grid proper
  const double avg = (double)n / (double)tiles;
  double best = 1e300;
  int64_t unit = NT;
  for (int64_t m = 1; m <= 64 || m * tiles <= 4 * SLOTS; ++m) {
    const double share = avg / m;
    const int64_t u = std::max<int64_t>(NT, (int64_t)(1.1 * share) + 1);
    const double cost = std::ceil((double)m * tiles / SLOTS) * (std::ceil(share / NT) + 1.5);
    if (u <= room && cost < best) {
      best = cost;
      unit = u;
    }
    if (share <= NT) break;
  }
  return std::min(room, std::max(unit, (n + 4 * SLOTS - 1) / (4 * SLOTS)));
}

int64_t sort32(pic_ctx *c) {
  Tiles &T = c->tiles;
  const int64_t n = c->n_used;
  T.nunits = 0;
  if (n == 0) {
    T.sorted_end = 0;
    cudaMemsetAsync(T.start, 0, (T.nbins + 1) * sizeof(int64_t), c->stream);
    return 0;
  }
  // room for the work units first: on failure no particle has moved, every
  // particle takes the unbinned path until a sort succeeds, and the context
  // reports the error
  T.unit = unit_size(c);
  const int64_t ucap = T.ntiles + n / T.unit + 1;
  if (ucap > T.units_cap) {
    cudaStreamSynchronize(c->stream);
    cudaFree(T.units);
    T.units = nullptr;
    T.units_cap = 0;
    T.sorted_end = 0;
    if (cudaMalloc((void **)&T.units, (size_t)ucap * sizeof(long long)) != cudaSuccess) {
      cudaGetLastError();
      c->host_err |= ERR_CAPACITY;
      return -1;
    }
    T.units_cap = ucap;
  }
  Args32 A = make_args(c, 0.0);
  A.mix = c->mix_sort ? 1 : 0;
  c->mix_sort = false;
  int64_t *count = T.cursor;
  cudaMemsetAsync(count, 0, (T.nbins + 1) * sizeof(int64_t), c->stream);
  const unsigned blocks = (unsigned)((n + 255) / 256);
  const int nblk = (int)((T.nbins + SCAN_CHUNK - 1) / SCAN_CHUNK);
  ++c->launches, k_hist<<<blocks, 256, 0, c->stream>>>(A, c->p32, n, count);
  ++c->launches, launch_on(c->stream, c->overlap, k_scan_sums, nblk, 256, count, T.nbins, T.bsum);
  ++c->launches, launch_on(c->stream, c->overlap, k_scan_bins, 1, 1024, T.bsum, T.bsum + nblk + 1, nblk);
  ++c->launches, launch_on(c->stream, c->overlap, k_scan_apply, nblk, 256, count, T.start, T.nbins, T.bsum + nblk + 1, nblk);
  ++c->launches, launch_on(c->stream, c->overlap, k_scatter_cells, blocks, 256, A, c->p32, c->q32, n, count);
  // the work units of the tile kernel (n bounds the live count from above)
  const unsigned tb = (unsigned)((T.ntiles + 255) / 256);
  const int ublk = (int)((T.ntiles + SCAN_CHUNK - 1) / SCAN_CHUNK);
  ++c->launches, launch_on(c->stream, c->overlap, k_unit_count, tb, 256, T.start, T.tc, T.ntiles, T.unit, T.ucount);
  ++c->launches, launch_on(c->stream, c->overlap, k_scan_sums, ublk, 256, T.ucount, T.ntiles, T.usum);
  ++c->launches, launch_on(c->stream, c->overlap, k_scan_bins, 1, 1024, T.usum, T.usum + ublk + 1, ublk);
  ++c->launches, launch_on(c->stream, c->overlap, k_scan_apply, ublk, 256, T.ucount, T.ucount, T.ntiles, T.usum + ublk + 1, ublk);
  ++c->launches, launch_on(c->stream, c->overlap, k_unit_fill, tb, 256, T.ucount, T.ntiles, T.units);
  // particles in cell bins: everything before the bin of removed ones; units
  cudaMemcpyAsync(c->h_pinned, T.start + (int64_t)T.ntiles * T.tc, sizeof(int64_t), cudaMemcpyDeviceToHost, c->stream);
  cudaMemcpyAsync(c->h_pinned + 1, T.ucount + T.ntiles, sizeof(int64_t), cudaMemcpyDeviceToHost, c->stream);
  cudaStreamSynchronize(c->stream);
  const int64_t live = c->h_pinned[0];
  T.nunits = c->h_pinned[1];
  Parts32 tmp = c->p32;
  c->p32 = c->q32;
  c->q32 = tmp;
  c->n_used = live;
  T.sorted_end = live;
  return live;
}

void ens_sort_scratch_free(EnsSortScratch &sc) {
  if (sc.h) cudaFreeHost(sc.h);
  if (sc.d) cudaFree(sc.d);
  sc = EnsSortScratch{};
}

int ens_sort32(pic_ctx *const *cs, int m, cudaStream_t st, EnsSortScratch &sc, int64_t *kernels) {
  *kernels = 0;
  std::vector<pic_ctx *> due;
  for (int k = 0; k < m; ++k) {
    pic_ctx *c = cs[k];
    if (c->n_used == 0) {  // nothing to order: as sort32
      sort32(c);
      c->steps_since_sort = 0;
      continue;
    }
    due.push_back(c);
  }
  const int nd = (int)due.size();
  if (nd == 0) return PIC_OK;
  // room for each member's work units (reallocated after the device is idle
  // on the stream: a previous graph may still read the old list).  A member's
  // unit size goes with its list: until every call has succeeded it keeps both.
  bool synced = false;
  std::vector<int64_t> unit(nd);
  for (int k = 0; k < nd; ++k) {
    pic_ctx *c = due[k];
    Tiles &T = c->tiles;
    unit[k] = unit_size(c);
    const int64_t ucap = T.ntiles + c->n_used / unit[k] + 1;
    if (ucap <= T.units_cap) continue;
    if (!synced) { PIC_CUDA(cudaStreamSynchronize(st)); synced = true; }
    cudaFree(T.units);
    T.units = nullptr;
    T.units_cap = 0;
    T.sorted_end = 0;
    T.nunits = 0;
    PIC_CUDA(cudaMalloc((void **)&T.units, (size_t)ucap * sizeof(long long)));
    T.units_cap = ucap;
  }
  // phase maps: {member, block} per block of each launch
  enum { M_ZERO, M_PART, M_BINS, M_TOP, M_TILE, M_UBINS, M_UTOP, M_N };
  std::vector<int2> mp[M_N];
  auto add = [&](int q, int k, int64_t blocks) {
    for (int64_t b = 0; b < blocks; ++b) mp[q].push_back(make_int2(k, (int)b));
  };
  std::vector<EnsSortArg> tab(nd);
  const size_t tab_bytes = (size_t)nd * sizeof(EnsSortArg);
  for (int k = 0; k < nd; ++k) {
    pic_ctx *c = due[k];
    Tiles &T = c->tiles;
    EnsSortArg &E = tab[k];
    E.A = make_args(c, 0.0);
    E.A.mix = c->mix_sort ? 1 : 0;
    E.S = c->p32;
    E.D = c->q32;
    E.n = c->n_used;
    E.count = T.cursor;
    E.start = T.start;
    E.bsum = T.bsum;
    E.nbins = T.nbins;
    E.nblk = (int)((T.nbins + SCAN_CHUNK - 1) / SCAN_CHUNK);
    E.ublk = (int)((T.ntiles + SCAN_CHUNK - 1) / SCAN_CHUNK);
    E.ntiles = T.ntiles;
    E.tc = T.tc;
    E.ucount = T.ucount;
    E.usum = T.usum;
    E.units = T.units;
    E.unit = unit[k];
    E.err = c->d_err;
    add(M_ZERO, k, (T.nbins + 1 + 255) / 256);
    add(M_PART, k, (E.n + 255) / 256);
    add(M_BINS, k, E.nblk);
    add(M_TOP, k, 1);
    add(M_TILE, k, (T.ntiles + 255) / 256);
    add(M_UBINS, k, E.ublk);
    add(M_UTOP, k, 1);
  }
  // one buffer: the table, the maps and the read-back values
  size_t at[M_N + 1];
  at[0] = (tab_bytes + 255) / 256 * 256;
  for (int q = 0; q < M_N; ++q) at[q + 1] = at[q] + (mp[q].size() * sizeof(int2) + 255) / 256 * 256;
  const size_t out_at = at[M_N], bytes = out_at + (size_t)nd * 3 * sizeof(int64_t);
  if (bytes > sc.cap) {
    PIC_CUDA(cudaStreamSynchronize(st));
    ens_sort_scratch_free(sc);
    PIC_CUDA(cudaMallocHost((void **)&sc.h, bytes));
    PIC_CUDA(cudaMalloc((void **)&sc.d, bytes));
    sc.cap = bytes;
  }
  for (int k = 0; k < nd; ++k) tab[k].out = reinterpret_cast<int64_t *>(sc.d + out_at) + 3 * k;
  memcpy(sc.h, tab.data(), tab_bytes);
  for (int q = 0; q < M_N; ++q) memcpy(sc.h + at[q], mp[q].data(), mp[q].size() * sizeof(int2));
  PIC_CUDA(cudaMemcpyAsync(sc.d, sc.h, out_at, cudaMemcpyHostToDevice, st));
  const EnsSortArg *dt = reinterpret_cast<const EnsSortArg *>(sc.d);
  auto L = [&](int q) {
    EnsList x;
    x.blk = reinterpret_cast<const int2 *>(sc.d + at[q]);
    return x;
  };
  auto nb = [&](int q) { return (unsigned)mp[q].size(); };
  k_ens_sort_zero<<<nb(M_ZERO), 256, 0, st>>>(dt, L(M_ZERO));
  k_ens_hist<<<nb(M_PART), 256, 0, st>>>(dt, L(M_PART));
  k_ens_scan_sums<<<nb(M_BINS), 256, 0, st>>>(dt, L(M_BINS), 0);
  k_ens_scan_bins<<<nb(M_TOP), 1024, 0, st>>>(dt, L(M_TOP), 0);
  k_ens_scan_apply<<<nb(M_BINS), 256, 0, st>>>(dt, L(M_BINS), 0);
  k_ens_scatter<<<nb(M_PART), 256, 0, st>>>(dt, L(M_PART));
  k_ens_unit_count<<<nb(M_TILE), 256, 0, st>>>(dt, L(M_TILE));
  k_ens_scan_sums<<<nb(M_UBINS), 256, 0, st>>>(dt, L(M_UBINS), 1);
  k_ens_scan_bins<<<nb(M_UTOP), 1024, 0, st>>>(dt, L(M_UTOP), 1);
  k_ens_scan_apply<<<nb(M_UBINS), 256, 0, st>>>(dt, L(M_UBINS), 1);
  k_ens_unit_fill<<<nb(M_TILE), 256, 0, st>>>(dt, L(M_TILE));
  k_ens_sort_out<<<(unsigned)((nd + 255) / 256), 256, 0, st>>>(dt, nd);
  PIC_CUDA(cudaGetLastError());
  PIC_CUDA(cudaMemcpyAsync(sc.h + out_at, sc.d + out_at, (size_t)nd * 3 * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  PIC_CUDA(cudaStreamSynchronize(st));
  *kernels = 12;
  const int64_t *out = reinterpret_cast<const int64_t *>(sc.h + out_at);
  for (int k = 0; k < nd; ++k) {
    pic_ctx *c = due[k];
    Tiles &T = c->tiles;
    std::swap(c->p32, c->q32);
    c->n_used = out[3 * k];
    T.sorted_end = out[3 * k];
    T.unit = unit[k];
    T.nunits = out[3 * k + 1];
    c->mix_sort = false;
    c->host_err |= (int)out[3 * k + 2];
    c->steps_since_sort = 0;
    c->launches += 10;  // the kernels of its own sort (sort32)
  }
  return PIC_OK;
}

void charge32(pic_ctx *c) {
  for (double *p : {c->Q, c->Qa, c->Qt}) cudaMemsetAsync(p, 0, c->grid_elems * sizeof(double), c->stream);
  if (c->n_used == 0) return;
  using U = unsigned long long;
  // the flux accumulators are clear between steps: the first lends a plane
  const ChargePlanes C{{(U *)c->Q, (U *)c->Qt}, {(U *)c->Qa, (U *)c->acc[0]},
                       (long long *)c->scratch, (long long)(c->scratch_bytes / sizeof(long long)),
                       c->d_cnt + CNT_SMALL + c->charge_slot, c->d_cnt + CNT_SMALL + 1 - c->charge_slot};
  c->charge_slot ^= 1;
  const Args32 A = make_args(c, 0.0);
  const unsigned blocks = (unsigned)ens_tile_blocks(c);
  if (c->tiles.TI == 8) ++c->launches, k_charge_tiles<8, 32><<<blocks, NT, 0, c->stream>>>(A, c->p32, C);
  else if (c->tiles.TI == 32) ++c->launches, k_charge_tiles<32, 8><<<blocks, NT, 0, c->stream>>>(A, c->p32, C);
  else ++c->launches, k_charge_tiles<16, 16><<<blocks, NT, 0, c->stream>>>(A, c->p32, C);
  const Grid &G = c->G;
  const dim3 gr((G.nth + 1 + 31) / 32, (G.nr + 2 * G.g + 1 + 7) / 8);
  // (never captured: its callers wait for the result)
  ++c->launches, launch_on(c->stream, true, k_charge_finish, gr, dim3(32, 8), G, c->qexp, C, (U *)c->acc[0], c->Q, c->Qa);
  ++c->launches, launch_on(c->stream, true, k_charge_small, 4 * 152, 256, A, c->p32, C, c->Q, c->Qa);
}

void reduce_particles32(pic_ctx *c) {
  if (c->n_used == 0) return;
  // a fixed grid (4 blocks per SM) keeps the same-address atomics few
  ++c->launches, k_reduce32<<<4 * 152, 256, 0, c->stream>>>(c->p32, c->n_used, c->G.qm, c->d_acc,
                                                                        c->d_cnt + CNT_LIVE);
}

}  // namespace pic
