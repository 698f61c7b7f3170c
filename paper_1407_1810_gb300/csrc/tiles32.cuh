// tiles32.cuh -- what the FP32 tile kernel's translation units share: its
// arguments, the tile and window geometry, the field window through the tensor
// memory accelerator, and the launchers of its two forms (tiles_one.cu: one
// particle a thread; tiles_two.cu: two).
#pragma once
#include <cuda.h>  // CUtensorMap

#include "pic_internal.h"

namespace pic {
namespace t32 {

// halo cells around a tile served from shared memory.  A particle that
// drifts beyond it between sorts takes the global-memory path, and one such
// lane makes its whole warp run that path: with 4 cells (0.003 % of
// particle-steps at 20 steps per sort, against 0.14 % with 2) the window of
// 27 x 27 nodes still leaves room for 4 CTAs per SM.
constexpr int H = 4;
// the last tile of a row or column reaches up to its side + H + 1 nodes past
// the grid's ghost band: the padding of the grid arrays must hold it for the
// longest tile side (32 cells), so the window stays inside the allocation
static_assert(32 + H + 1 <= PAD, "grid padding must cover every tile window");
// window nodes of a TI x TJ tile: the tile, the halo and the stencil reach
template <int TI, int TJ>
struct Win {
  static constexpr int WI = TI + 2 * H + 3, WJ = TJ + 2 * H + 3, WN = WI * WJ;
};
constexpr int NT = 256;                                  // particles per pass of a tile CTA, and its threads
constexpr int NTH = NT / 2;                              // its threads with two particles each
// Shared-memory accumulation splits each term v (|v| <= 2^36 quanta) into
// v = h 2^SPLIT + l with |h| <= 2^18, |l| <= 2^17 and sums h and l with
// native 32-bit shared atomics.  A particle's terms on one node of a component
// add up to at most 2^36, so the sums of a work unit of up to UNIT_ROOM
// particles stay below 2^31 whatever they do; in a larger unit a node whose sums
// come near that limit is reported as ERR_CAPACITY.
constexpr int SPLIT = 18;
constexpr int UNIT_ROOM = 8000;

struct Args32 {
  int nr, nth, n_filt, PI, PJ, LD;
  int r_log, th_ea, vacuum, pusher;
  float dxi, inv_dxi, dt, qm, inv_nth, nth_f;
  // constants carried as FP32 hi + lo pairs: a constant rounded once to FP32
  // would bias every particle's step the same way (a systematic error that
  // grows linearly with the step count)
  float dt_lo, inv_dxi_lo, k2_hi, k2_lo;  // k2 = nth / pi (linear theta map)
  float b0_lo, qmdt;     // qmdt = (q/m) dt rounded once
  float pi_nth;          // pi / nth (linear theta map: angle per column)
  float hinv_dxi, hinv_dxi_lo, hnth;  // 1 / (2 dxi) as a pair; nth / 2
  float nbrw;                         // -b0 r_min Omega
  const long long *qexp;    // fixed-point exponent e: one flux unit is 2^(e - KFIX)
  const int64_t *ids;       // particle ids (read only for an axis-crossing tie)
  AxisTies ties;
  const float *r_n;         // f_r(i) per padded row (FP32)
  const float *ir_n;        // per padded row: 1 / f_r(i) (log r), f_r(i) (linear r)
  int trw;                  // sort: columns of the transposed bins
  const float2 *th_n;       // (sin, cos) of the node angle per padded column (FP32, linear theta map)
  const float *f[6];        // FP32 field copies (padded)
  long long *acc[3];        // global fixed-point flux accumulators (padded)
  int *err;
  long long *cnt;
  // tiles
  int row0, ntj, ntiles, ti, tj, tc;
  int mix;                  // sort: 1 = by cell, bins stored transposed; 0 = by tile, order kept
  const int64_t *start;
  const long long *units;   // work units: tile << 32 | index of the unit within its tile
  int64_t nunits, unit;     // units of the binned particles; particles per unit
  int64_t sorted_end, n_used;
  // vacuum
  float b0, r_min, omega_t;
};

// the particles [b0, b1) of a work unit (tile << 32 | index in the tile): its
// even share of the tile's bin
__device__ __forceinline__ void unit_range(const Args32 &A, long long u, int &tile, int64_t &b0, int64_t &b1) {
  tile = (int)(u >> 32);
  const int64_t s = A.start[(int64_t)tile * A.tc], n = A.start[(int64_t)(tile + 1) * A.tc] - s;
  const int64_t m = (n + A.unit - 1) / A.unit, q = u & 0xffffffffll;
  if (n < (1ll << 31) / 4096 && m < 4096) {  // 32-bit quotients
    b0 = s + (int64_t)((uint32_t)n * (uint32_t)q / (uint32_t)m);
    b1 = s + (int64_t)((uint32_t)n * (uint32_t)(q + 1) / (uint32_t)m);
  } else {
    b0 = s + n * q / m;
    b1 = s + n * (q + 1) / m;
  }
}

// whether a node's sums in a unit of n particles may have left 32 bits
__device__ __forceinline__ bool sums_full(int hsum, int lsum, int64_t n) {
  return (abs(hsum) >= (1 << 30) || abs(lsum) >= (1 << 30)) && n > UNIT_ROOM;
}

__device__ inline size_t pidx(const Args32 &A, int i, int j) {
  return (size_t)(i + A.PI) * (size_t)A.LD + (size_t)(j + A.PJ);
}

// Specialisations of the step: the grid maps, pusher and analytic field kind
// fixed at compile time for the two common configurations, so their branches
// fold away (8 % faster than reading them from the arguments), on grids fine
// enough that the radial and meridional series need no general fallback
// (pic_ctx::small_steps); SPEC_GENERIC reads them at run time.
enum Spec { SPEC_GENERIC = 0, SPEC_MONOPOLE = 1, SPEC_ROTATOR = 2 };
template <int SPEC>
struct Flags {
  bool r_log, th_ea;
  int pusher, vacuum;
  __device__ explicit Flags(const Args32 &A)
      : r_log(SPEC == SPEC_GENERIC ? A.r_log != 0 : true),
        th_ea(SPEC == SPEC_GENERIC ? A.th_ea != 0 : SPEC == SPEC_ROTATOR),
        pusher(SPEC == SPEC_GENERIC ? A.pusher : PIC_VAY),
        vacuum(SPEC == SPEC_GENERIC ? A.vacuum : (SPEC == SPEC_ROTATOR ? PIC_VAC_MONOPOLE_ROTATOR : PIC_VAC_MONOPOLE)) {}
};

// ---- the field window through the tensor memory accelerator ---------------
// Each FP32 field is a 2-D tensor (LD columns x rows of the padded grid).  A
// tile's window (WI rows x WJ columns from (wi0, wj0)) is fetched as one box
// per field whose first column is wj0 - WOFF: with the padding PJ a multiple of
// 8 and every tile's j0 a multiple of 8, that column is a multiple of 4 floats
// (16 bytes), as a tiled copy requires; the box is WB columns wide, a whole
// number of 16-byte units.  The boxes land in a staging area, are laid out at
// the window's own pitch WJ (odd, so lanes in different rows fall in different
// banks) and the staging area then becomes the deposit accumulators.
constexpr int WOFF = 3;
static_assert((PAD - H - 1 - WOFF) % 8 == 0, "window box column must stay 16-byte aligned");
template <int TI, int TJ>
struct Box {
  static constexpr int WI = Win<TI, TJ>::WI, WJ = Win<TI, TJ>::WJ, WN = Win<TI, TJ>::WN;
  static constexpr int WB = (WOFF + WJ + 3) / 4 * 4;        // box width (floats)
  static constexpr int SLOT = (WI * WB + 31) / 32 * 32;     // one field's box, 128-byte multiple
  static constexpr int SF = (6 * WN + 31) / 32 * 32;        // laid-out window (floats)
  static constexpr int QUEUE = NTH / 32 * 6 * 64;           // the warps' queues of crossing paths
  // staging, then accumulators (one particle a thread); and the queues (two)
  static constexpr int U1 = 6 * SLOT > 6 * WN ? 6 * SLOT : 6 * WN;
  static constexpr int U2 = 6 * SLOT > 6 * WN + QUEUE ? 6 * SLOT : 6 * WN + QUEUE;
};

struct TileMaps {  // the six field tensors for the current tile shape (kernel parameter)
  CUtensorMap m[6];
};

__device__ inline uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ inline void tma_window(float *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// wait for phase 0 of the window barrier, at most `limit` polls
__device__ inline bool window_wait(uint64_t *bar, long long limit) {
  for (long long k = 0; k < limit; ++k) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_u32(bar))
        : "memory");
    if (done) return true;
  }
  return false;
}

// Tensor maps read by the TMA unit from global memory (the batched ensemble
// kernel's per-member maps, written by a host copy before any launch) are
// ordered after those writes by an acquire fence of the tensor-map proxy.
__device__ inline void tensormap_acquire(const CUtensorMap *map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(map) : "memory");
}

// One member of a batched launch: its step's arguments and its six field
// tensor maps (device memory) for its tile shape.
struct EnsTileArg {
  Args32 A;
  Parts32 P;
  const CUtensorMap *maps;
};

// Up to ENS_TILE_SLOTS members in one launch, passed as kernel parameters:
// the arguments sit in the same immutable parameter memory as those of
// k_tiles32, so the compiler treats them alike (loads it may hoist out of the
// particle loop), which keeps every member's arithmetic bit-identical to its
// own k_tiles32 launch.  Member k owns blocks [off[k], off[k + 1]).
constexpr int ENS_TILE_SLOTS = 48;
struct EnsTileBatch {
  EnsTileArg a[ENS_TILE_SLOTS];
  int off[ENS_TILE_SLOTS + 1];
  int n;
};
static_assert(sizeof(EnsTileBatch) <= 32000, "kernel parameters are limited to 32 KB");

// launches a form's tile kernel: the shape (0: 16 x 16, 1: 8 x 32, 2: 32 x 8)
// and specialisation of one context, or of the members of a batch
void launch_one(int spec, int shape, unsigned blocks, cudaStream_t s, bool overlap, const Args32 &A, const Parts32 &P,
                const TileMaps &M);
void launch_two(int spec, int shape, unsigned blocks, cudaStream_t s, bool overlap, const Args32 &A, const Parts32 &P,
                const TileMaps &M);
void launch_ens_one(int spec, int shape, unsigned blocks, cudaStream_t s, bool beside, const EnsTileBatch &B);
void launch_ens_two(int spec, int shape, unsigned blocks, cudaStream_t s, bool beside, const EnsTileBatch &B);

}  // namespace t32
}  // namespace pic
