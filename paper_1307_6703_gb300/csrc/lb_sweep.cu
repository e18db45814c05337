// lb_sweep.cu -- strip-sweep kernel: one fused time step of the vdW lattice
// Boltzmann scheme (arXiv:1307.6703, Sec. II) streamed through shared memory
// by TMA, for FP32 storage and for 16-bit deviation storage.
//
// Work decomposition.  The lattice is cut into tiles: column strips of at
// most 56 columns (origins on 16-byte TMA coordinates) by row segments.  One
// warp (a CTA of 32 threads) computes one tile.  Its window is the 64 columns
// x0-4 .. x0+59 (strip plus 4-column halos), two adjacent columns per lane,
// and it sweeps the segment upwards, two rows per iteration.  Every row of
// the previous state is read from HBM once by the TMA engine: tensor copies
// bring a pair of rows of all nine population planes into the warp's own
// ring in shared memory (one mbarrier per slot, waits bounded).  With tau = 1
// the ring has 3 slots and pair k+3 is requested as soon as iteration k has
// read pair k; otherwise 5 slots, pair k+3 requested at the end of iteration
// k; either way it is first read in iteration k+2.
//
// Iteration k (a = ya - 3 + 2k) runs four stages, each on two rows:
//   A  rows a, a+1     : propagated populations (pull), density n (n-hat on
//                        walls), raw momentum sum_i f_i c_i
//   B  rows a-1, a     : P = p^i - p^w (Eq. eqstate), L = lap n, grad n
//   C  rows a-2, a-1   : F = dP + kappa n dL + F_ext (Eq. force2), n u*
//                        (Eq. newvel), wall rule on wall rows
//   D  rows a-3, a-2   : div(n u*), equilibrium (Eq. eqfunc), forcing
//                        (Eqs. forceterm, coeff), BGK collision; store f*.
// A lane keeps the rows of n, P, L and n u* that a stencil still needs in
// registers; the values of the two columns beside its own come from the
// neighbouring lanes by shuffles, once per row and quantity.  So no stage
// waits for another warp, nothing but the populations goes through shared
// memory, and the two columns of a lane are the two halves of the packed
// FP32 instructions in every stage.  Column halos (3, 2, 1 sites for n, P/L,
// F/J) are computed by the outer lanes; row halos come from the sweep itself,
// so apart from the 7-row warm-up of each segment (stages A, A-B, A-C only)
// nothing is recomputed.
//
// Why this split.  One warp per tile needs no barrier, and two columns per lane
// take fewer instructions: 187 a site and thread (FP32, warm-ups and waits
// included) against 320 in the form before (a CTA of 124 threads, one column each,
// all stages exchanging through shared memory between four CTA barriers an
// iteration).
// What bounds it now is memory for FP32 (72 algorithmic bytes a site) and, for
// 16-bit storage, the issue rate and the latency of 12 warps an SM.  Measured
// per step of 4096 x 1024, tau = 1, 20 steps a launch: FP32 58.7 -> 51.9 us
// (5,820 GB/s; 49.3 us in 200-step launches), bf16 59.4 -> 49.2 us; 512 x 256
// FP32, 100 steps: 35.8 -> 8.8 us.
//
// Walls: rows -1 and ny of n, P, L and n u* are the mirror images of rows 1
// and ny-2 (even reflection; y part of n u* odd): the stages of a wall row
// take the row inside for the one outside.  Periodic directions: the state buffers
// carry 4 ghost columns (and, without walls, 4 ghost rows) on each side,
// refreshed by the kernel when it stores boundary sites, so every TMA box is
// one plain copy.
//
// The collision uses the algebraically equivalent "moment" form
//   f*_i = (1 - omega) f_i + w_i E_i,
//   E_i = omega n [A_i + 3 c.u + 9/2 (c.u)^2 - 3/2 u^2] + 3 c.B + 9/2 C:cc - 3/2 tr C,
// with A_i the rest factor 1 + (T - T0)(c.c - 2 T0) / (2 T0^2), T0 = 1/3;
// the rest population is taken as n minus the other eight, which is the same
// value in exact arithmetic and keeps the site mass exact in FP32.
//
// Storage formats.  FP32: the nine populations as floats.  16-bit deviation
// storage (bfloat16 or IEEE half): for i = 1..8 the deviation d_i = f_i - r_i
// from a reference population (r = rho_ref/9 on axis links, rho_ref/36 on
// diagonal links, rounded to FP32) is stored rounded to nearest even; the
// rest population stays a float and takes the remainder n - sum_{i>=1} f_i
// of the ROUNDED values, so each site keeps its density to FP32 round-off.
// Arithmetic is FP32 in both formats; with 16-bit storage it runs on the
// deviations themselves: the references cancel in the momentum, add one
// constant to the density, and enter the collision as one constant per link
// class, so decoding and encoding are a conversion each.
//
// On the last step of a call (or every step while a monitoring ring is set)
// every CTA also writes FP64 partial sums of mass and momentum of the state
// it stored, and a flag for non-finite or out-of-range sites.  In a multi-step
// launch, and while monitoring, the CTA that finishes last adds them up, so the
// global sums of the new state need no further kernel; after a single step a
// block does when they are asked for (one warp takes 34 us for 2368 records).
//
// Initial state, single steps and moments are programmatic dependent launches
// (pdl.cuh): a step's successor may be scheduled once every CTA of the step has
// left its main loop, and waits (griddepcontrol.wait) for the step to complete
// before it touches global memory, which hides the launch gap between the two
// grids.
#include <cmath>
#include <cstddef>
#include <type_traits>
#include <vector>
#include <algorithm>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lb_device.cuh"
#include "lb_internal.h"
#include "pdl.cuh"

namespace lbk {

namespace {

constexpr int kCols = 64;                   // window columns of a tile: two per lane
static_assert(kCols == kSweepWindow, "the dependency lists cover the window");
constexpr int kTileW = kCols - 8;           // widest tile
constexpr int kThreads = 32;
constexpr unsigned kAll = 0xffffffffu;
constexpr uint32_t kWaitLimit = 1u << 22;
static_assert(kWaitLimit == kSweepWaitLimit, "what lb_set_wait_limit starts from");
// Rows of a tile where the tiling's segments would leave warps idle: about
// kTilesPerWarp tiles of a step per resident warp, so that a tile's neighbours
// have finished the previous step by the time its ticket is drawn; a multiple
// of 4 rows (the steady loop's turn; 31 rows instead of 32 cost 10 %), or 2
// where the lattice is too small for that anyway.  Measured per step: 4096 x
// 1024 FP32 52.3 us at 32 rows (54.1 at 24, 52.9 at 40, 59.9 at 64), 512 x 256
// 10.0 at 2 (10.9 at 4, 16.1 at 16), 2048 x 512 20.4 at 8 (24.9 at 4, 25.6 at
// 32).
constexpr int kSegMax = 64;
constexpr double kTilesPerWarp = 1.3;
// Fewer in a batch: its lattices do not wait for one another.  Per step at 1.3 /
// 1.1, tau 1: 512 lattices of 64 x 32 FP32 37.2 / 31.7 us, bf16 45.6 / 41.5, 256 of
// 128 x 64 48.7 / 45.3 and 61.6 / 57.5, 300 of 96 x 48 33.8 / 31.1 and 43.2 / 42.0, 64
// uneven ones of up to 1024 x 256 85.4 / 85.8 and 88.0 / 87.0, 16 of 1024 x 256 53.9 /
// 54.9 and 58.5 / 59.4.
constexpr double kTilesPerWarpBatch = 1.1;

// A storage policy describes one slot of the ring (two rows of the window)
// and how a lane reads its two columns 2t, 2t + 1 of plane q: mid() is those
// two, left() the columns 2t - 1, 2t and right() 2t + 1, 2t + 2 (the sources
// of links with c_x = 1 and -1).  Lanes 0 and 31 read one column beyond the
// window there: inside the slot, and only for halo values nobody uses.
//
// FP32 storage: one 3D box {64, 2, 9} (columns, rows, planes) per pair.
struct StoreF32 {
  static constexpr bool kDev = false;
  static constexpr bool kOdd = false;         // nx not a multiple of the quantum
  static constexpr int kQuantum = 4;          // 16-byte x coordinates of float boxes
  static constexpr int kMaxW = 116;           // widest strip a tiling may name (split into tiles)
  static constexpr unsigned kTxBytes = 9 * 2 * kCols * sizeof(float);
  static constexpr int kSlotBytes = kTxBytes;
  struct Row {
    const unsigned char *p;  // column 2t of plane 0; planes 2 rows apart
  };
  static constexpr int kPlane = 2 * kCols * 4;
  __device__ __forceinline__ static Row row(const unsigned char *slot, int r, int t) {
    return {slot + r * (kCols * 4) + 8 * t};
  }
  __device__ __forceinline__ static float2 mid(const Row &r, int q) {
    return *reinterpret_cast<const float2 *>(r.p + q * kPlane);
  }
  __device__ __forceinline__ static float2 left(const Row &r, int q) {
    const float *c = reinterpret_cast<const float *>(r.p + q * kPlane);
    return make_float2(c[-1], c[0]);
  }
  __device__ __forceinline__ static float2 right(const Row &r, int q) {
    const float *c = reinterpret_cast<const float *>(r.p + q * kPlane);
    return make_float2(c[1], c[2]);
  }
};

// The same for lattices whose number of columns is not a multiple of 4: the last
// column of tiles is narrower, its last pair of columns may be half outside,
// and periodic images are stored one column at a time (nx odd shifts them by
// half a pair).  (These lattices used the tile kernel, whose tiles of 32 x 16
// sites pull every population three times from L1/L2: 20 steps of 1021 x 509
// 990 us a pass, now 394.)
struct StoreF32Odd : StoreF32 {
  static constexpr bool kOdd = true;
};

// 16-bit deviation storage: a float box {64, 2, 1} of the rest plane and a
// 16-bit box {64, 2, 8} of the deviation planes (128-byte rows) per pair.  A
// lane's two columns are one 32-bit word of a deviation plane.  mid(0) is the
// rest population, mid/left/right(q >= 1) deviations d_q = f_q - r_q.
template <class H>
struct StoreDev {
  using Half = H;
  static constexpr bool kDev = true;
  static constexpr bool kOdd = false;
  static constexpr int kQuantum = 8;          // 16-byte x coordinates of 16-bit boxes
  static constexpr int kMaxW = 120;
  static constexpr int kRestBytes = 2 * kCols * sizeof(float);
  static constexpr int kDevOffset = kRestBytes;
  static constexpr int kDevBytes = 8 * 2 * kCols * 2;
  static constexpr unsigned kTxBytes = kRestBytes + kDevBytes;
  static constexpr int kSlotBytes = kDevOffset + kDevBytes;
  struct Row {
    const unsigned char *f0;  // rest plane, column 2t
    const unsigned char *d;   // deviation plane of link 1, column 2t
  };
  static constexpr int kPlane = 2 * kCols * 2;
  __device__ __forceinline__ static Row row(const unsigned char *slot, int r, int t) {
    return {slot + r * (kCols * 4) + 8 * t, slot + kDevOffset + r * (kCols * 2) + 4 * t};
  }
  __device__ static float lo(unsigned w);  // first (even) column of a word
  __device__ static float hi(unsigned w);
  __device__ static unsigned enc2(float2 v);
  __device__ __forceinline__ static float2 dec2(unsigned w) { return make_float2(lo(w), hi(w)); }
  __device__ __forceinline__ static const unsigned *words(const Row &r, int q) {
    return reinterpret_cast<const unsigned *>(r.d + (q - 1) * kPlane);
  }
  __device__ __forceinline__ static float2 mid(const Row &r, int q) {
    if (q == 0) return *reinterpret_cast<const float2 *>(r.f0);
    return dec2(words(r, q)[0]);
  }
  __device__ __forceinline__ static float2 left(const Row &r, int q) {
    const unsigned *w = words(r, q);
    return make_float2(hi(w[-1]), lo(w[0]));
  }
  __device__ __forceinline__ static float2 right(const Row &r, int q) {
    const unsigned *w = words(r, q);
    return make_float2(hi(w[0]), lo(w[1]));
  }
  __device__ static float dec(H v);  // one element
};
template <>
__device__ __forceinline__ float StoreDev<__nv_bfloat16>::lo(unsigned w) { return __uint_as_float(w << 16); }
template <>
__device__ __forceinline__ float StoreDev<__nv_bfloat16>::hi(unsigned w) { return __uint_as_float(w & 0xffff0000u); }
template <>
__device__ __forceinline__ unsigned StoreDev<__nv_bfloat16>::enc2(float2 v) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const unsigned *>(&h);
}
template <>
__device__ __forceinline__ float StoreDev<__nv_bfloat16>::dec(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ float StoreDev<__half>::lo(unsigned w) {
  return __low2float(*reinterpret_cast<const __half2 *>(&w));
}
template <>
__device__ __forceinline__ float StoreDev<__half>::hi(unsigned w) {
  return __high2float(*reinterpret_cast<const __half2 *>(&w));
}
template <>
__device__ __forceinline__ unsigned StoreDev<__half>::enc2(float2 v) {
  const __half2 h = __floats2half2_rn(v.x, v.y);
  return *reinterpret_cast<const unsigned *>(&h);
}
template <>
__device__ __forceinline__ float StoreDev<__half>::dec(__half v) { return __half2float(v); }

using StoreBF16 = StoreDev<__nv_bfloat16>;
using StoreFP16 = StoreDev<__half>;

// The two forms of the kernel.  With tau = 1 (omega = 1) the collision has no
// (1 - omega) f term: f* depends on the moments alone, so stage D reads no
// populations and a row pair is done with once stage A has read it (half the
// shared-memory loads, 3 slots instead of 5, so 12 warps an SM instead of 9:
// 51.9 us a step against 57.0 for tau = 2, 4096 x 1024 FP32).  Same bits: the
// term it leaves out is an exact zero.
template <class St, bool kTau1>
struct Form {
  // slots of the ring: pairs k, k+1 in use and one coming (tau = 1), or pairs
  // k-2 .. k+1 and one coming
  static constexpr int kPairs = kTau1 ? 3 : 5;
  // resident warps per SM: 12 by registers (168 a thread), 9 by shared memory
  static constexpr int kMinBlocks = kTau1 || St::kDev ? 12 : 9;
};

// A warp's population ring.  Rows ya - 4 + 2p and ya - 3 + 2p are pair p, in
// slot p % kPairs.
template <int SlotBytes, int kPairs>
struct __align__(128) SweepSmem {
  unsigned char pops[kPairs][SlotBytes];  // one row pair of every plane per slot
  unsigned long long full[kPairs];
  static_assert(SlotBytes % 128 == 0, "TMA destinations must be 128-byte aligned");
};
template <class St, bool kTau1>
using SmemOf = SweepSmem<St::kSlotBytes, Form<St, kTau1>::kPairs>;
static_assert(StoreBF16::kDevOffset % 128 == 0, "16-bit boxes must land on 128-byte boundaries");

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}

// One poll of phase `parity` of an mbarrier.
__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
// Wait for it, at most `limit` polls; false on give-up (the data are then
// meaningless but every address the kernel touches stays in bounds; the
// caller waits no more, stops the tile at its end and drains the copies still
// in flight).  One loop with one exit: the warp is whole afterwards.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t limit) {
  uint32_t it = 0;
  while (!mbar_poll(bar, parity) && it < limit) ++it;
  return it < limit;
}

__device__ __forceinline__ void tma_box(const CUtensorMap *map, uint32_t dst, uint32_t bar, int xpad, int ypad,
                                        uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(xpad), "r"(ypad), "r"(0), "r"(bar), "l"(policy)
      : "memory");
}

// L2 policies for the population boxes.  A tile's first four pairs (its
// 4-row warm-up and first 4 rows) are the rows the segment below reads last,
// about one tile-duration later: they are kept (evict-last) so that read
// comes from L2; the tile's other rows get the normal policy.
__device__ __forceinline__ uint64_t l2_policy(bool keep) {
  uint64_t p;
  if (keep)
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  else
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}
constexpr int kKeepPairs = 4;

// Two rows (all nine planes, the window's columns) of the padded state into
// a ring slot, completing on the slot's mbarrier.
template <class St>
__device__ __forceinline__ void tma_pair(const CUtensorMap *m0, const CUtensorMap *m1, uint32_t dst, uint32_t bar,
                                         int xpad, int ypad, uint64_t policy) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(St::kTxBytes)
               : "memory");
  tma_box(m0, dst, bar, xpad, ypad, policy);
  if constexpr (St::kDev) tma_box(m1, dst + St::kDevOffset, bar, xpad, ypad, policy);
}
// 1/v by the PTX approximate reciprocal (v > 0 and finite here: densities
// and 1 - b n on the liquid-vapour branch).
__device__ __forceinline__ float rcp(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// Arithmetic on one site (V = float) or on the two columns of a lane (V =
// float2, executed as the packed FP32 pair instructions of sm_100 and later).
// Each operation is rounded once, as written, so the result of a site does
// not depend on which half of a pair (and so which tiling) computed it --
// with one rule for the callers: no product feeds an
// addition or subtraction.  The code generator fuses a pair multiply into
// the pair add that consumes it (one rounding instead of two; measured on
// GB300, and unlike the scalar forms, which stay as written), so every such
// combination is written as an explicit fma in both forms.
struct V2 {
  __device__ static float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
  __device__ static float2 sub(float2 a, float2 b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&d);
  }
  __device__ static float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
  __device__ static float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
  __device__ static float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
  __device__ static float2 inv(float2 v) { return make_float2(rcp(v.x), rcp(v.y)); }
  // a/b to half a unit in the last place and a little (values well inside the
  // normal range): the approximate quotient, corrected by its exact remainder
  // (Markstein, IBM J. Res. Dev. 34 (1990) 111).
  __device__ static float2 div(float2 a, float2 b) {
    const float2 r = inv(b), q = mul(a, r);
    return fma(fma(neg(b), q, a), r, q);
  }
};

// Density and raw momentum sum_i f_i c_i of the pulled populations (16-bit
// storage: deviations, n gets the references' sum r_sum):
// E = f1 + f5 + f8 and W = f3 + f6 + f7 serve n and the x momentum.
//
// kFine, here and below: the form of lb_moments, which memory bounds.  Opposite
// links nearly cancel, so their differences come first; the pressure's quotient,
// the Laplacian and the gradients round where the terms are small.  A step's
// forms take fewer instructions, but as a reading of the state they leave the
// velocity 1.2 to 1.4 times further from FP64 (root mean square, 120 lattices of
// all kinds) than these.  Moments of 4096 x 1024: FP32 45.6 us with a step's
// forms, 45.9 with these, bf16 28.3 and 29.3.
template <bool kDev, bool kFine>
__device__ __forceinline__ void site_sums(const SweepConsts &K, const float2 *f, float2 &n, float2 &sx, float2 &sy) {
  using O = V2;
  const float2 E = O::add(O::add(f[1], f[5]), f[8]), W = O::add(O::add(f[3], f[6]), f[7]);
  n = O::add(O::add(f[0], O::add(f[2], f[4])), O::add(E, W));
  if constexpr (kDev) n = O::add(n, K.r_sum);
  if constexpr (kFine) {
    sx = O::add(O::add(O::sub(f[1], f[3]), O::sub(f[5], f[6])), O::sub(f[8], f[7]));
    sy = O::add(O::add(O::sub(f[2], f[4]), O::sub(f[5], f[8])), O::sub(f[6], f[7]));
  } else {
    sx = O::sub(E, W);
    sy = O::sub(O::add(O::add(f[2], f[5]), f[6]), O::add(O::add(f[4], f[7]), f[8]));
  }
}

// P = p^i - p^w = nT - nT/(1 - bn) + a n^2 (Eq. eqstate).
template <bool kFine>
__device__ __forceinline__ float2 pressure_diff(const SweepConsts &K, float2 c) {
  using O = V2;
  const float2 nT = O::mul(c, K.T), d = O::fma(c, K.nb, K.one), an = O::mul(c, K.a);
  if constexpr (kFine) return O::fma(c, K.T, O::fma(an, c, O::neg(O::div(nT, d))));
  else return O::fma(an, c, O::fma(O::neg(nT), O::inv(d), nT));  // nT - nT r in one rounding
}

// Where one step's results go: the new state (fout; the deviation planes of
// 16-bit storage at fdev) and, when arrivals is set, the fused global sums:
// the CTA that finishes last adds the nrec records at recs into total (if
// set) and monitor (if set, with mon_step) and resets *arrivals.
struct StepIO {
  const float *fin;  // the input state (and its deviation planes)
  const void *fdin;
  float *fout;
  void *fdev;
  const double *recs;
  unsigned nrec;
  unsigned *arrivals;
  double *total;
  double *monitor;
  double mon_step;
};
// One row of a quantity as a lane sees it: its two columns c and the columns
// on their left and right.
struct Nbr {
  float2 c;
  float l, r;
};
__device__ __forceinline__ Nbr spread(float2 c) {
  return {c, __shfl_up_sync(kAll, c.y, 1), __shfl_down_sync(kAll, c.x, 1)};
}
// x-derivative, y-derivative and Laplacian stencils of Eqs. (xstencil,
// laplstencil).  Every operation is rounded as written (explicit intrinsics,
// no contraction), so a site's value does not depend on the tile that
// computed it.
//
// right - left neighbour, right + left neighbour
__device__ __forceinline__ float2 xdiff(const Nbr &v) {
  return make_float2(__fsub_rn(v.c.y, v.l), __fsub_rn(v.r, v.c.x));
}
__device__ __forceinline__ float2 xsum(const Nbr &v) {
  return make_float2(__fadd_rn(v.c.y, v.l), __fadd_rn(v.r, v.c.x));
}
// N d1 + M (d2 + d0) for the differences d of the three rows
__device__ __forceinline__ float2 dstencil(const SweepConsts &K, float2 d1, float2 d2, float2 d0) {
  using O = V2;
  return O::fma(K.N, d1, O::mul(K.M, O::add(d2, d0)));
}
// y-derivative from the rows above (u) and below (d)
__device__ __forceinline__ float2 dy_stencil(const SweepConsts &K, const Nbr &u, const Nbr &d) {
  using O = V2;
  const float2 e = O::sub(u.c, d.c);
  const float2 pm = make_float2(__fadd_rn(e.y, __fsub_rn(u.l, d.l)), __fadd_rn(__fsub_rn(u.r, d.r), e.x));
  return O::fma(K.N, e, O::mul(K.M, pm));
}
template <bool kFine>
__device__ __forceinline__ float2 laplacian(const SweepConsts &K, const Nbr &r0, const Nbr &r1, const Nbr &r2) {
  using O = V2;
  const float2 s1 = O::add(xsum(r1), O::add(r2.c, r0.c));
  const float2 s2 = O::add(xsum(r2), xsum(r0));
  if constexpr (kFine) return O::fma(K.m4QR, r1.c, O::fma(K.Q, s1, O::mul(K.R, s2)));
  else return O::fma(K.Q, s1, O::fma(K.R, s2, O::mul(K.m4QR, r1.c)));
}

// Propagated populations of a lane's two sites of row r1 (pull).  With 16-bit
// storage f[1..8] are the deviations d_i = f_i - r_i and f[0] is the rest
// population; with FP32 storage they are the populations.
template <class St>
__device__ __forceinline__ void pull(const typename St::Row &r0, const typename St::Row &r1,
                                     const typename St::Row &r2, float2 *f) {
  f[0] = St::mid(r1, 0); f[1] = St::left(r1, 1); f[3] = St::right(r1, 3);
  f[2] = St::mid(r0, 2); f[5] = St::left(r0, 5); f[6] = St::right(r0, 6);
  f[4] = St::mid(r2, 4); f[7] = St::right(r2, 7); f[8] = St::left(r2, 8);
}

// Deviations <-> populations of the moving links (16-bit storage only).
__device__ __forceinline__ void add_refs(float2 *f, float r_ax, float r_dg) {
#pragma unroll
  for (int q = 1; q < 9; ++q) f[q] = V2::add(f[q], q <= 4 ? make_float2(r_ax, r_ax) : make_float2(r_dg, r_dg));
}

// n-hat of a wall row (Sec. II, moving walls): f the propagated populations,
// r1 the row itself in the ring (its own stored populations).
template <class St>
__device__ __forceinline__ float2 wall_density(bool top, const typename St::Row &r1, const float2 *f, const SweepArgs &A) {
  using O = V2;
  auto own = [&](int q) {
    if constexpr (St::kDev) return q == 0 ? St::mid(r1, 0) : O::add(q <= 4 ? make_float2(A.ref_ax, A.ref_ax) : make_float2(A.ref_dg, A.ref_dg), St::mid(r1, q));
    return St::mid(r1, q);
  };
  float2 n;
  if (!top) {
    n = O::add(O::add(O::add(own(0), own(4)), own(7)), own(8));
    n = O::add(O::add(O::add(O::add(O::add(n, f[1]), f[3]), f[4]), f[7]), f[8]);
  } else {
    n = O::add(O::add(O::add(own(0), own(2)), own(6)), own(5));
    n = O::add(O::add(O::add(O::add(O::add(n, f[1]), f[3]), f[2]), f[6]), f[5]);
  }
  return n;
}

// The propagated populations that a wall row's rule starts from, read from
// the input state (rare: two rows of the lattice); e is the element of the
// lane's first column in the row.  16-bit storage: populations, not
// deviations.
template <class St>
__device__ __forceinline__ void wall_pull(bool top, const StepIO &O, const SweepArgs &A, int e, float2 *f) {
  auto at = [&](int q, int i) -> float {
    if constexpr (St::kDev) {
      using H = typename St::Half;
      const unsigned short u = __ldcg(static_cast<const unsigned short *>(O.fdin) + (size_t)(q - 1) * A.plane + i);
      return __fadd_rn(St::dec(*reinterpret_cast<const H *>(&u)), q <= 4 ? A.ref_ax : A.ref_dg);
    } else {
      return __ldcg(O.fin + (size_t)q * A.plane + i);
    }
  };
  auto two = [&](int q, int i) { return make_float2(at(q, i), at(q, i + 1)); };
#pragma unroll
  for (int q = 0; q < 9; ++q) f[q] = make_float2(0.f, 0.f);
  f[1] = two(1, e - 1);
  f[3] = two(3, e + 1);
  const int r = top ? e - A.pitch : e + A.pitch;
  if (!top) {
    f[4] = two(4, r);
    f[7] = two(7, r + 1);
    f[8] = two(8, r - 1);
  } else {
    f[2] = two(2, r);
    f[5] = two(5, r - 1);
    f[6] = two(6, r + 1);
  }
}

// The wall rule (wall_fill) on both sites of a lane.
__device__ __forceinline__ void wall_fill2(bool top, float U, float2 Fx, float2 Fy, float2 n, float2 *f) {
  float a[9], b[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    a[q] = f[q].x;
    b[q] = f[q].y;
  }
  wall_fill<float>(top, U, Fx.x, Fy.x, n.x, a);
  wall_fill<float>(top, U, Fx.y, Fy.y, n.y, b);
#pragma unroll
  for (int q = 0; q < 9; ++q) f[q] = make_float2(a[q], b[q]);
}

// One collision (Eqs. evoleq, eqfunc, forceterm, coeff) in the moment form
//   f*_i = (1 - omega) f_i + w_i E_i,
//   E_i = omega n [A_i + 3 c.u + 9/2 (c.u)^2 - 3/2 u^2] + 3 c.B + 9/2 C:cc - 3/2 tr C,
// for the eight moving populations (the rest population is the remainder,
// taken by the caller after any storage rounding).  With on = omega n,
// S_i = on (c.u)^2 + C:cc and T_i = on c.u + c.B, w_i E_i splits into a part
// even in c, h_i = e_i + 9/2 w_i S_i with e_i = w_i (on A_i - 3/2 (S_x + S_y))
// (S_x + S_y = on u^2 + tr C), and an odd part t_i = 3 w_i T_i.  On the
// axes (w = 1/9) h_x = e_a + S_x / 2, t_x = T_x / 3; on the diagonals
// (w = 1/36) S_(+-) = S_x + S_y +- 2 X with X = on u_x u_y + C_xy and
// T_(+-) = T_y +- T_x, so h_(+-) = e_d + (S_x + S_y) / 8 +- X / 4 and
// t_(+-) = T_(+-) / 12.  kDev: f holds the deviations d_i = f_i - r_i
// and fs receives d*_i = f*_i - r_i = (1 - omega) d_i + w_i E_i - omega r_i
// (omega r_i joins e_a on the axes and e_d on the diagonals).
template <bool kDev, bool kTau1>
__device__ __forceinline__ void collide(const SweepConsts &K, const float2 *f, float2 n, float2 Jx, float2 Jy, float2 Fx,
                                        float2 Fy, float2 dnx, float2 dny, float2 divJ, float2 *fs) {
  using O = V2;
  const float2 rn = O::inv(n);
  const float2 ux = O::mul(Jx, rn), uy = O::mul(Jy, rn);
  const float2 on = O::mul(K.om, n);
  const float2 onux = O::mul(on, ux), onuy = O::mul(on, uy);
  const float2 ux2 = O::mul(K.two, ux), uy2 = O::mul(K.two, uy);
  // C / g (Eq. coeff)
  const float2 cxx = O::fma(K.th, O::fma(ux2, dnx, divJ), O::mul(ux2, Fx));
  const float2 cyy = O::fma(K.th, O::fma(uy2, dny, divJ), O::mul(uy2, Fy));
  const float2 cxy = O::fma(K.th, O::fma(ux, dny, O::mul(uy, dnx)), O::fma(ux, Fy, O::mul(Fx, uy)));
  const float2 Sx = O::fma(onux, ux, O::mul(K.g, cxx)), Sy = O::fma(onuy, uy, O::mul(K.g, cyy));
  const float2 X = O::fma(onux, uy, O::mul(K.g, cxy));
  const float2 Sxy = O::add(Sx, Sy);  // on u^2 + tr C
  float2 ea, ed;
  if constexpr (kDev) {
    ea = O::fma(on, K.Aax, O::fma(K.m6, Sxy, K.mwr_ax));
    ed = O::fma(on, K.Adg, O::fma(K.m24, Sxy, K.mwr_dg));
  } else {
    ea = O::fma(on, K.Aax, O::mul(Sxy, K.m6));
    ed = O::fma(on, K.Adg, O::mul(Sxy, K.m24));
  }
  const float2 hx = O::fma(K.half, Sx, ea), hy = O::fma(K.half, Sy, ea);
  const float2 h5 = O::fma(K.e8, Sxy, O::fma(K.q4, X, ed));
  const float2 h6 = O::fma(K.e8, Sxy, O::fma(K.mq4, X, ed));
  // odd parts: t_x = T_x / 3, t_(+-) = (T_y +- T_x) / 12
  const float2 Tx = O::fma(K.g, Fx, onux), Ty = O::fma(K.g, Fy, onuy);
  const float2 Tp = O::add(Ty, Tx), Tm = O::sub(Ty, Tx);
  auto relaxed = [&](int q, float2 e) {  // (1 - omega) f + w E
    if constexpr (kTau1) return e;
    else return O::fma(K.om1, f[q], e);
  };
  fs[1] = relaxed(1, O::fma(Tx, K.third, hx));
  fs[3] = relaxed(3, O::fma(Tx, K.mthird, hx));
  fs[2] = relaxed(2, O::fma(Ty, K.third, hy));
  fs[4] = relaxed(4, O::fma(Ty, K.mthird, hy));
  fs[5] = relaxed(5, O::fma(Tp, K.twelfth, h5));
  fs[7] = relaxed(7, O::fma(Tp, K.mtwelfth, h5));
  fs[6] = relaxed(6, O::fma(Tm, K.twelfth, h6));
  fs[8] = relaxed(8, O::fma(Tm, K.mtwelfth, h6));
}

// The rest population as the remainder: n - sum_{i>=1} f*_i (16-bit
// storage: (n - sum r_i) - sum d*_i), which keeps the site's mass exact.
__device__ __forceinline__ float2 rest_remainder(float2 n, const float2 *fs) {
  using O = V2;
  return O::sub(n, O::add(O::add(O::add(fs[1], fs[3]), O::add(fs[2], fs[4])),
                          O::add(O::add(fs[5], fs[7]), O::add(fs[6], fs[8]))));
}

}  // namespace

struct NoDone {
  __device__ void operator()() const {}
};
// The wait of a step launched on its own, as a programmatic dependent of the
// previous step: until that grid has finished and its writes are visible.
struct WaitGrid {
  __device__ bool operator()() const {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return true;
  }
};

// Where a moments launch writes: compact [ny][nx] arrays (null: not wanted)
// of T; a lane's two columns in one store where the arrays are aligned for it.
// kRows (host arrays of odd widths): 32 consecutive columns of a row in one store
// of the warp instead of every other one in two, which cross the link in twice
// as many pieces (doubles, 509 x 256 52 -> 44 us, 4093 x 1024 736 -> 696; device
// arrays take 18 us longer that way).
struct NoMoments {
  static constexpr bool kOn = false, kRows = false;
};
template <class T, bool kByRows = false>
struct Moments {
  static constexpr bool kOn = true, kRows = kByRows;
  T *n, *ux, *uy;
  int pairs;
  __device__ __forceinline__ void put(T *p, size_t s, float2 v, bool half) const {
    if (p == nullptr) return;
    if (half) {
      p[s] = (T)v.x;
    } else if (pairs) {
      struct alignas(2 * sizeof(T)) Two {
        T a, b;
      };
      *reinterpret_cast<Two *>(p + s) = Two{(T)v.x, (T)v.y};
    } else {
      p[s] = (T)v.x;
      p[s + 1] = (T)v.y;
    }
  }
  // The values v of a row of a tile of W columns whose first is element s; the
  // whole warp.
  __device__ __forceinline__ void put_row(T *p, size_t s, int W, float2 v) const {
    if (p == nullptr) return;
    const int t = threadIdx.x;
#pragma unroll
    for (int r = 0; r < 2; ++r) {  // the tile's column 32 r + t, the window's 4 + 32 r + t
      const int c = 32 * r + t, lane = ((4 + c) >> 1) & 31;
      const float x = __shfl_sync(kAll, v.x, lane), y = __shfl_sync(kAll, v.y, lane);
      if (c < W) p[s + c] = (T)(t & 1 ? y : x);
    }
  }
};

// Origin and width of tile column i: base_w columns, the first `extra`
// columns of tiles one quantum wider.
template <class St>
__device__ __forceinline__ void tile_columns(const SweepArgs &A, int i, int &x0, int &W) {
  x0 = i * A.base_w + St::kQuantum * min(i, A.extra);
  W = A.base_w + (i < A.extra ? St::kQuantum : 0);
  if constexpr (St::kOdd) W -= i == A.nstrips - 1 ? A.pad : 0;
}

// One warp's work: tile column `strip`, segment `seg` of the lattice
// described by A, whose input state the tensor maps tin (and tdev, the
// deviation planes of 16-bit storage) describe; results as O says; the tile's
// mass/momentum record goes to rec.  Returns false when a copy wait gave up
// (the warp then stopped and drained the copies still in flight).
// kMulti: called once per tile by the multi-step kernel, which does not
// hand its SM slots to a dependent grid early.  kLow: for low tiles.
template <class St, bool kTau1, bool kMulti = false, bool kLow = false, class Wait = WaitGrid, class Done = NoDone, class Mom = NoMoments>
__device__ __forceinline__ bool sweep_body(const CUtensorMap *tin, const CUtensorMap *tdev, const SweepArgs &A, const SweepConsts &K,
                                           const StepIO &O, const int strip, const int seg, double *rec,
                                           const bool want_records, const Wait &wait = Wait{}, const Done &done = Done{},
                                           const Mom &mom = Mom{}) {
  using Row = typename St::Row;
  using Smem = SmemOf<St, kTau1>;
  using V = V2;
  constexpr int kPairs = Form<St, kTau1>::kPairs;
  // (not of odd widths: half a pair would count a ghost column)
  const bool records = !St::kOdd && want_records;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem &S = *reinterpret_cast<Smem *>(smem_raw);

  const int t = threadIdx.x;
  int x0, W;
  tile_columns<St>(A, strip, x0, W);
  const int ya = seg * A.seg_h;
  const int yb = min(A.ny, ya + A.seg_h);
  const int nx = A.nx, ny = A.ny;
  const bool walls = A.walls != 0;
  const int x = x0 - 4 + 2 * t;  // first of this lane's two columns (may be halo columns)
  const bool actD = 2 * t >= 4 && 2 * t + 1 < W + 4;         // both columns in the tile
  const bool half = St::kOdd && 2 * t >= 4 && 2 * t == W + 3;  // the first one only
  const int kmax = (yb - ya + 5) >> 1;  // last iteration
  const int npairs = kmax + 2;          // rows ya-4 .. ya+2*kmax-1, at most yb+4
  const int pitch = A.pitch, plane = (int)A.plane;
  auto image = [&](int c) { return c < 4 ? nx : (c >= nx - 4 ? -nx : 0); };
  const int im0 = image(x), im1 = St::kOdd ? image(x + 1) : im0;  // to the periodic image columns
  float2 sinx = make_float2(0.f, 0.f);
  if (2 * t >= 2 && 2 * t <= W + 4) {  // a constant table
    auto wrap = [&](int c) { return c < 0 ? c + nx : (c >= nx ? c - nx : c); };
    if constexpr (St::kOdd) sinx = make_float2(A.sinx[wrap(x)], A.sinx[wrap(x + 1)]);
    else sinx = *reinterpret_cast<const float2 *>(A.sinx + wrap(x));
  }
  if (t == 0) {
    for (int s = 0; s < kPairs; ++s) mbar_init(smem_u32(&S.full[s]));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Before any other global access: the input must be complete (it is the
  // output of the step before), and the output buffer read to the end (it was
  // that step's input).
  if (!wait()) return false;
  // TMA writes need 128-byte aligned destinations: refuse to run otherwise.
  if (smem_u32(&S.pops[0][0]) & 127u) {
    if (t == 0) atomicOr(A.err, 2);
    return false;
  }
  auto request = [&](int p, int slot) {  // lane 0: pair p into its slot
    tma_pair<St>(tin, tdev, smem_u32(S.pops[slot]), smem_u32(&S.full[slot]), x0, ya + 2 * p, l2_policy(p < kKeepPairs));
  };
  int issued = min(kPairs, npairs);  // pairs requested so far (lane 0)
  if (t == 0) {
    for (int p = 0; p < issued; ++p) request(p, p);
  }
  __syncwarp();
  const uint32_t limit = kMulti ? kWaitLimit : A.wait_limit;
  bool ok = mbar_wait(smem_u32(&S.full[0]), 0, limit);
  // What the stages carry from one iteration to the next (rows relative to
  // the next iteration's a).
  const float2 zero = make_float2(0.f, 0.f);
  const Nbr none{zero, 0.f, 0.f};
  Nbr N0 = none, N1 = none;                    // n of rows a-2, a-1
  float2 n3 = zero;                            // n of row a-3
  float2 gx3 = zero, gy3 = zero, gx2 = zero, gy2 = zero;  // grad n of rows a-3, a-2
  float2 sx2 = zero, sy2 = zero, sx1 = zero, sy1 = zero;  // raw momentum of rows a-2, a-1
  Nbr P0 = none, P1 = none, L0 = none, L1 = none;         // P, lap n of rows a-3, a-2
  float2 dJ4 = zero, dJ3 = zero, Jx3 = zero;   // x-differences of J_x of rows a-4, a-3; J_x of row a-3
  Nbr Jy4 = none, Jy3 = none;                  // J_y of rows a-4, a-3
  float2 Fx3 = zero, Fy3 = zero;               // force of row a-3
  float2 acc_m = zero, acc_x = zero, acc_y = zero;
  int bad = 0;
  int s0 = 0;        // slot of pair k
  uint32_t par = 0;  // phase parity of pair k+1

  // One iteration; kSteady instantiates it for iterations whose rows are all
  // interior rows of the segment (no wall rows or their mirrors, no warm-up
  // rows, no periodic ghost images in y), where every per-row condition
  // below is known to hold.
  auto iteration = [&](const int k, auto steady_tag) {
    constexpr bool kSteady = decltype(steady_tag)::value;
    const int s1 = s0 == kPairs - 1 ? 0 : s0 + 1;
    // newest pair needed: k+1.  After a wait that gave up a lane waits no more
    // and goes on with whatever is there (in bounds) to the tile's end.
    ok = mbar_wait(smem_u32(&S.full[s1]), par, ok ? limit : 1u) && ok;
    __syncwarp();
    if (s1 == kPairs - 1) par ^= 1u;
    const int a = ya - 3 + 2 * k;
    // rows a-1, a (pair k), a+1, a+2 (pair k+1)
    const Row r1 = St::row(S.pops[s0], 0, t), ra = St::row(S.pops[s0], 1, t);
    const Row rb = St::row(S.pops[s1], 0, t), rc = St::row(S.pops[s1], 1, t);
    // Every lane has read pair p for the last time: pair p + kPairs may take
    // its slot.
    auto refill = [&](int p, int slot) {
      __syncwarp();
      if (t == 0 && ok && p >= 0 && p + kPairs < npairs) {
        request(p + kPairs, slot);
        ++issued;
      }
    };

    // ---------------------------------------- A: rows a, a+1 -- n, raw momentum
    float2 nA[2], sxA[2], syA[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float2 f[9];
      pull<St>(j ? ra : r1, j ? rb : ra, j ? rc : rb, f);
      const int y = a + j;
      if (!kSteady && walls && (y == 0 || y == ny - 1)) {
        if constexpr (St::kDev) add_refs(f, A.ref_ax, A.ref_dg);
        nA[j] = wall_density<St>(y != 0, j ? rb : ra, f, A);
        sxA[j] = syA[j] = zero;  // from the wall rule, stage C
      } else {  // (rows beyond a wall: nothing uses them)
        site_sums<St::kDev, Mom::kOn>(K, f, nA[j], sxA[j], syA[j]);
      }
    }
    if constexpr (kTau1) refill(k, s0);
    const Nbr N2 = spread(nA[0]), N3 = spread(nA[1]);

    // -------------------------------------- B: rows a-1, a -- P, lap n, grad n
    Nbr P2 = none, P3 = none, L2 = none, L3 = none;
    float2 gx1 = zero, gy1 = zero, gx0 = zero, gy0 = zero;
    // The row below a bottom wall row is the mirror image of the row above it,
    // and the other way round at the top (kWall: y may be a wall row).
    auto mirror = [&](int y, auto &down, auto &up) {
      if (walls && y == 0) down = up;
      if (walls && y == ny - 1) up = down;
    };
    if (kSteady || k >= 1) {
      P2 = spread(pressure_diff<Mom::kOn>(K, N1.c));
      P3 = spread(pressure_diff<Mom::kOn>(K, N2.c));
      auto rows = [&](int y, Nbr d, const Nbr &c, Nbr u, Nbr &L, float2 &gx, float2 &gy) {
        if constexpr (!kSteady) mirror(y, d, u);
        L = spread(laplacian<Mom::kOn>(K, d, c, u));
        gx = dstencil(K, xdiff(c), xdiff(u), xdiff(d));
        gy = dy_stencil(K, u, d);
      };
      rows(a - 1, N0, N1, N2, L2, gx1, gy1);
      rows(a, N1, N2, N3, L3, gx0, gy0);
    }

    // -------------------------------------- C: rows a-2, a-1 -- F, n u*
    float2 FxC[2] = {zero, zero}, FyC[2] = {zero, zero}, JxC[2] = {zero, zero}, JyC[2] = {zero, zero};
    if (kSteady || k >= 2) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        Nbr pd = j ? P1 : P0, pu = j ? P3 : P2, ld = j ? L1 : L0, lu = j ? L3 : L2;
        const Nbr &pc = j ? P2 : P1, &lc = j ? L2 : L1;
        if constexpr (!kSteady) {
          mirror(a - 2 + j, pd, pu);
          mirror(a - 2 + j, ld, lu);
        }
        const float2 n = j ? N1.c : N0.c;
        const float2 kn = V::mul(K.kappa, n);
        float2 Fx, Fy;
        if constexpr (Mom::kOn) {
          const float2 dP = dstencil(K, xdiff(pc), xdiff(pu), xdiff(pd)), dL = dstencil(K, xdiff(lc), xdiff(lu), xdiff(ld));
          Fx = V::fma(K.A0, sinx, V::fma(kn, dL, dP));
          Fy = V::fma(kn, dy_stencil(K, lu, ld), dy_stencil(K, pu, pd));
        } else {
          // D P + kappa n D L = D G with G = P + kappa n L at the neighbours
          // (n is the site's own density, a constant of the stencil)
          auto left = [&](const Nbr &p, const Nbr &l) {
            return make_float2(__fmaf_rn(kn.x, l.l, p.l), __fmaf_rn(kn.y, l.c.x, p.c.x));
          };
          auto right = [&](const Nbr &p, const Nbr &l) {
            return make_float2(__fmaf_rn(kn.x, l.c.y, p.c.y), __fmaf_rn(kn.y, l.r, p.r));
          };
          const float2 g0m = left(pd, ld), g0p = right(pd, ld), g1m = left(pc, lc), g1p = right(pc, lc);
          const float2 g2m = left(pu, lu), g2p = right(pu, lu);
          const float2 g0c = V::fma(kn, ld.c, pd.c), g2c = V::fma(kn, lu.c, pu.c);
          Fx = V::fma(K.A0, sinx, dstencil(K, V::sub(g1p, g1m), V::sub(g2p, g2m), V::sub(g0p, g0m)));
          Fy = dstencil(K, V::sub(g2c, g0c), V::sub(g2p, g0p), V::sub(g2m, g0m));
        }
        float2 sx = j ? sx1 : sx2, sy = j ? sy1 : sy2;
        if constexpr (!kSteady) {
          const int y = a - 2 + j;
          if (walls && (y == 0 || y == ny - 1)) {
            float2 f[9];
            wall_pull<St>(y != 0, O, A, (int)A.off + y * pitch + x, f);
            wall_fill2(y != 0, y != 0 ? A.u_top : A.u_bot, Fx, Fy, n, f);
            sx = V::add(V::add(V::sub(f[1], f[3]), V::sub(f[5], f[6])), V::sub(f[8], f[7]));
            sy = V::sub(V::add(V::sub(f[2], f[4]), V::add(f[5], f[6])), V::add(f[7], f[8]));
          }
        }
        FxC[j] = Fx;
        FyC[j] = Fy;
        // n u* = sum f c + F / 2 (Eq. newvel)
        JxC[j] = V::fma(K.half, Fx, sx);
        JyC[j] = V::fma(K.half, Fy, sy);
      }
    }
    if constexpr (Mom::kOn) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int y = a - 2 + j;
        const float2 n = j ? N1.c : N0.c;
        if constexpr (Mom::kRows) {
          if (y < ya || y >= yb) continue;
          auto over_n = [&](float2 J) {  // (halo values may be anything: no quotients of them)
            return actD || half ? make_float2(__fdiv_rn(J.x, n.x), __fdiv_rn(J.y, n.y)) : zero;
          };
          const size_t s = (size_t)y * nx + x0;
          mom.put_row(mom.n, s, W, n);
          mom.put_row(mom.ux, s, W, over_n(JxC[j]));
          mom.put_row(mom.uy, s, W, over_n(JyC[j]));
          continue;
        }
        if (!(actD || half) || y < ya || y >= yb) continue;
        const size_t s = (size_t)y * nx + x;
        mom.put(mom.n, s, n, half);
        if (mom.ux != nullptr) mom.put(mom.ux, s, make_float2(__fdiv_rn(JxC[j].x, n.x), __fdiv_rn(JxC[j].y, n.y)), half);
        if (mom.uy != nullptr) mom.put(mom.uy, s, make_float2(__fdiv_rn(JyC[j].x, n.x), __fdiv_rn(JyC[j].y, n.y)), half);
      }
      n3 = N1.c;
      N0 = N2; N1 = N3;
      sx2 = sxA[0]; sy2 = syA[0]; sx1 = sxA[1]; sy1 = syA[1];
      P0 = P2; P1 = P3; L0 = L2; L1 = L3;
      s0 = s1;
      return;
    }
    const float2 dJ2 = xdiff(spread(JxC[0])), dJ1 = xdiff(spread(JxC[1]));
    const Nbr Jy2 = spread(JyC[0]), Jy1 = spread(JyC[1]);

    // -------------------------------------- D: rows a-3, a-2 -- collide, store
    float2 fs[2][9];
    unsigned code[2][8];  // 16-bit storage: the rounded deviations
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int y = a - 3 + j;
      if (!kSteady && (y < ya || y >= yb)) continue;
      const float2 n = j ? N0.c : n3, Jx = j ? JxC[0] : Jx3, Jy = j ? Jy2.c : Jy3.c;
      const float2 Fx = j ? FxC[0] : Fx3, Fy = j ? FyC[0] : Fy3;
      float2 dJd = j ? dJ3 : dJ4, dJu = j ? dJ1 : dJ2;
      Nbr Jyd = j ? Jy3 : Jy4, Jyu = j ? Jy1 : Jy2;
      if constexpr (!kSteady) {  // mirror rows: J_x even, J_y odd
        mirror(y, dJd, dJu);
        auto odd = [](const Nbr &v) { return Nbr{V::neg(v.c), -v.l, -v.r}; };
        if (walls && y == 0) Jyd = odd(Jyu);
        if (walls && y == ny - 1) Jyu = odd(Jyd);
      }
      const float2 divJ = V::add(dstencil(K, j ? dJ2 : dJ3, dJu, dJd), dy_stencil(K, Jyu, Jyd));
      float2 f[9];
      if constexpr (!kTau1) {
        // rows a-4 (pair k-2, second), a-3, a-2 (pair k-1), a-1 (pair k)
        const int m1 = s0 == 0 ? kPairs - 1 : s0 - 1, m2 = m1 == 0 ? kPairs - 1 : m1 - 1;
        const Row r4 = St::row(S.pops[m2], 1, t), r3 = St::row(S.pops[m1], 0, t), r2 = St::row(S.pops[m1], 1, t);
        pull<St>(j ? r3 : r4, j ? r2 : r3, j ? r1 : r2, f);
        if constexpr (!kSteady) {
          if (walls && (y == 0 || y == ny - 1)) {
            if constexpr (St::kDev) add_refs(f, A.ref_ax, A.ref_dg);
            wall_fill2(y != 0, y != 0 ? A.u_top : A.u_bot, Fx, Fy, n, f);
            if constexpr (St::kDev) add_refs(f, -A.ref_ax, -A.ref_dg);
          }
        }
      }
      collide<St::kDev, kTau1>(K, f, n, Jx, Jy, Fx, Fy, j ? gx2 : gx3, j ? gy2 : gy3, divJ, fs[j]);
      if constexpr (!St::kDev) {
        fs[j][0] = rest_remainder(n, fs[j]);
      } else {
        // Round the deviations (fs[1..8] hold d*_i), then let the rest
        // population carry the remainder of the rounded values (site
        // density kept): f*_0 = (n - sum r_i) - sum rounded d*_i.
#pragma unroll
        for (int q = 1; q < 9; ++q) {
          code[j][q - 1] = St::enc2(fs[j][q]);
          fs[j][q] = St::dec2(code[j][q - 1]);
        }
        fs[j][0] = rest_remainder(V::sub(n, K.r_sum), fs[j]);
      }
    }
    if (actD || half) {
      // the sites' elements in a plane, row j shifted by d elements (0 or to a
      // periodic image)
      auto put = [&](int j, int d, bool stream) {
        const int e = (int)A.off + (a - 3 + j) * pitch + x + d;
        auto at = [&](auto *base, int q) {
          return reinterpret_cast<char *>(base + (size_t)q * plane) + (unsigned)(sizeof(*base) * e);
        };
        if constexpr (!St::kDev) {
#pragma unroll
          for (int q = 0; q < 9; ++q) {
            float2 *p = reinterpret_cast<float2 *>(at(O.fout, q));
            if (stream) __stcs(p, fs[j][q]);
            else *p = fs[j][q];
          }
        } else {
          *reinterpret_cast<float2 *>(at(O.fout, 0)) = fs[j][0];
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<unsigned *>(at(reinterpret_cast<uint16_t *>(O.fdev), q)) = code[j][q];
        }
      };
      // The new state is streamed out (evict-first stores): it is read again
      // only by the next step.
#pragma unroll
      for (int j = 0; j < 2; ++j)
        if (!half && (kSteady || (a - 3 + j >= ya && a - 3 + j < yb))) put(j, 0, true);
      if (im0 != 0 || im1 != 0 || half || records || !kSteady) {  // images of edge sites, the tile's sums
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int y = a - 3 + j;
          if (!kSteady && (y < ya || y >= yb)) continue;
          const int gy = (kSteady || walls) ? 0 : ((y < 4) ? ny : ((y >= ny - 4) ? -ny : 0));
          if constexpr (!St::kOdd) {
            if (im0 != 0) put(j, im0, false);
            if (gy != 0) {
              put(j, gy * pitch, false);
              if (im0 != 0) put(j, gy * pitch + im0, false);
            }
          } else {
            auto put1 = [&](int c, int d) {  // one column
              float *p = O.fout + ((int)A.off + y * pitch + x + c + d);
#pragma unroll
              for (int q = 0; q < 9; ++q) p[(size_t)q * plane] = c ? fs[j][q].y : fs[j][q].x;
            };
            if (half) put1(0, 0);
            if (gy != 0) half ? put1(0, gy * pitch) : put(j, gy * pitch, false);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              const int g = c ? im1 : im0;
              if (g == 0 || (c && half)) continue;
              put1(c, g);
              if (gy != 0) put1(c, gy * pitch + g);
            }
          }
          // Mass and momentum of the stored sites: sum f* = n (by
          // construction), sum f* c = n u* + F/2 (identity of the collision).
          if (records) {
            const float2 n = j ? N0.c : n3, Jx = j ? JxC[0] : Jx3, Jy = j ? Jy2.c : Jy3.c;
            const float2 Fx = j ? FxC[0] : Fx3, Fy = j ? FyC[0] : Fy3;
            const float2 lim = make_float2(fabsf(Jx.x) + fabsf(Jy.x), fabsf(Jx.y) + fabsf(Jy.y));
            if (!(n.x > 0.f && n.x < A.nmax && n.y > 0.f && n.y < A.nmax && lim.x < 3.0e38f && lim.y < 3.0e38f)) bad = 1;
            acc_m = V::add(acc_m, n);
            if constexpr (!St::kDev) {
              acc_x = V::add(acc_x, V::fma(K.half, Fx, Jx));
              acc_y = V::add(acc_y, V::fma(K.half, Fy, Jy));
            } else {  // momentum of the stored (rounded) populations; refs cancel
              const float2 *g = fs[j];
              acc_x = V::add(acc_x, V::add(V::add(V::sub(g[1], g[3]), V::sub(g[5], g[6])), V::sub(g[8], g[7])));
              acc_y = V::add(acc_y, V::sub(V::add(V::sub(g[2], g[4]), V::add(g[5], g[6])), V::add(g[7], g[8])));
            }
          }
        }
      }
    }

    if constexpr (!kTau1) refill(k - 2, s0 >= 2 ? s0 - 2 : s0 - 2 + kPairs);
    n3 = N1.c;
    N0 = N2; N1 = N3;
    gx3 = gx1; gy3 = gy1; gx2 = gx0; gy2 = gy0;
    sx2 = sxA[0]; sy2 = syA[0]; sx1 = sxA[1]; sy1 = syA[1];
    P0 = P2; P1 = P3; L0 = L2; L1 = L3;
    dJ4 = dJ2; dJ3 = dJ1; Jx3 = JxC[1];
    Jy4 = Jy2; Jy3 = Jy1;
    Fx3 = FxC[1]; Fy3 = FyC[1];
    s0 = s1;
  };
  // Iteration k (a = ya - 3 + 2k) is steady -- every row of its four stages
  // interior, see the lambda's note -- when k >= 3, a - 2 < yb and, with
  // walls, 1 <= a - 3 and a + 1 <= ny - 2 (periodic: 4 <= a - 3 and
  // a + 1 < ny - 4).  These are lower and upper bounds on k, so the steady
  // iterations are the range [klo, khi).
  auto ceil2 = [](int v) { return (v + 1) >> 1; };  // ceil(v / 2), any sign
  const int klo = max(3, ceil2((walls ? 7 : 10) - ya));
  const int khi = min(min(kmax + 1, ceil2(yb - ya + 5)), walls ? ((ny - ya) >> 1) + 1 : ceil2(ny - ya - 2));
  // Two steady iterations per turn: what one carries to the next then needs no
  // register moves (an odd last one goes the general way).
  int k = 0;
  if constexpr (!kLow) {
    for (; k < min(klo, kmax + 1); ++k) iteration(k, std::false_type{});
#pragma unroll 1
    for (; k + 1 < khi; k += 2) {
      iteration(k, std::true_type{});
      iteration(k + 1, std::true_type{});
    }
    for (; k <= kmax; ++k) iteration(k, std::false_type{});
  } else {
    // The same with one copy of the general iteration's code.  Where tiles are
    // low, the warps of an SM are spread over all of it, and wait for
    // instructions (7.2 of 11.8 cycles between two of a warp's): per step of 512
    // lattices of 64 x 32, tau 1 and 2, FP32 37.8 -> 37.2 and 43.0 -> 42.4 us, bf16
    // 49.3 -> 45.9 and 59.2 -> 51.1, of 256 of 128 x 64 FP32 56.3 -> 49.0 and 60.2
    // -> 55.0.  It costs registers: single lattices of 4096 x 1024 50.4 -> 50.6, and
    // up to 10 % in launches of one step.
#pragma unroll 1
    while (k <= kmax) {
      iteration(k, std::false_type{});
      ++k;
      if (k >= klo) {
#pragma unroll 1
        for (; k + 1 < khi; k += 2) {
          iteration(k, std::true_type{});
          iteration(k + 1, std::true_type{});
        }
      }
    }
  }
  if (!__all_sync(kAll, ok)) {
    if (t == 0) atomicOr(A.err, 1);
    // A copy wait gave up: wait (again bounded) for every copy this warp may
    // still have in flight -- the last kPairs requested -- so that none
    // lands in shared memory after the warp has moved on, then stop.
    if (t == 0) {
      for (int p = max(0, issued - kPairs); p < issued; ++p)
        (void)mbar_wait(smem_u32(&S.full[p % kPairs]), (uint32_t)((p / kPairs) & 1), kWaitLimit);
    }
    __syncwarp();
    return false;
  }
  // The next step may be scheduled now (it waits for this grid to finish).
  if constexpr (!kMulti) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // Every lane is here: the tile's stores are done.  A multi-step caller
  // publishes its completion now -- the records below touch only the record
  // slots, so dependent tiles need not wait.
  done();

  // The tile's sums of the stored state (a lane's columns summed over rows in
  // FP32, then FP64 in a fixed order), when asked for.
  if (!records) return true;
  auto tree = [](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kAll, v, o);
    return v;
  };
  {
    const double m = tree((double)acc_m.x + (double)acc_m.y), jx = tree((double)acc_x.x + (double)acc_x.y);
    const double jy = tree((double)acc_y.x + (double)acc_y.y);
    const int any = __any_sync(kAll, bad);
    if (t == 0) {
      rec[0] = m;
      rec[1] = jx;
      rec[2] = jy;
      rec[3] = any ? 1.0 : 0.0;
    }
  }
  if (O.arrivals == nullptr) return true;

  // The last warp to finish sums every tile's record (FP64, fixed order:
  // lane t takes records t, t + 32, ..., eight loads in flight, then the
  // tree), so the global sums of the new state need no further kernel.
  const unsigned nrec = O.nrec;
  unsigned last = 0;
  if (t == 0) {
    __threadfence();  // this tile's record before its arrival
    last = (atomicAdd(O.arrivals, 1u) == nrec - 1) ? 1u : 0u;
  }
  if (__shfl_sync(kAll, last, 0) == 0u) return true;
  __threadfence();
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (unsigned b = t; b < nrec; b += 8 * kThreads) {
    double2 v[8][2];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const unsigned r = b + i * kThreads;
      const double2 *p = reinterpret_cast<const double2 *>(O.recs + 4 * (size_t)min(r, nrec - 1));
      v[i][0] = __ldcg(p);
      v[i][1] = __ldcg(p + 1);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (b + i * kThreads >= nrec) break;
      acc[0] += v[i][0].x;
      acc[1] += v[i][0].y;
      acc[2] += v[i][1].x;
      acc[3] += v[i][1].y;
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) acc[q] = tree(acc[q]);
  if (t == 0) {
    const double r[5] = {acc[0], acc[1], acc[2], acc[3] != 0.0 ? 1.0 : 0.0, __ldcg(A.err) != 0 ? 1.0 : 0.0};
    if (O.total) {
#pragma unroll
      for (int q = 0; q < 5; ++q) O.total[q] = r[q];
    }
    if (O.monitor) {
#pragma unroll
      for (int q = 0; q < 5; ++q) O.monitor[q] = r[q];
      O.monitor[5] = O.mon_step;
    }
    *O.arrivals = 0u;
  }
  return true;
}

template <class St, bool kTau1>
__global__ void __launch_bounds__(kThreads, Form<St, kTau1>::kMinBlocks)
sweep_step_kernel(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tdev,
                  const __grid_constant__ SweepArgs A) {
  const StepIO O{A.fin, A.fdin, A.fout, A.fdev, A.partials, gridDim.x * gridDim.y, A.total ? A.arrivals : nullptr,
                 A.total, A.monitor, A.mon_step};
  if (!sweep_body<St, kTau1>(&tin, &tdev, A, A.k, O, blockIdx.x, blockIdx.y,
                             A.partials + 4 * ((size_t)blockIdx.y * gridDim.x + blockIdx.x), A.records != 0)) {
    if (threadIdx.x == 0 && A.total) A.total[4] = 1.0;  // the sums of this launch will not be written
  }
}

// A lattice's arguments into shared memory (constants read by every lane).
__device__ __forceinline__ void stage_args(SweepArgs &A, const SweepArgs *src) {
  static_assert(sizeof(SweepArgs) % 8 == 0, "copied in 8-byte words");
  for (unsigned w = threadIdx.x; w < sizeof(SweepArgs) / 8; w += kThreads)
    reinterpret_cast<unsigned long long *>(&A)[w] = reinterpret_cast<const unsigned long long *>(src)[w];
  __syncwarp();
}

// A value every lane holds alike, in a form the compiler can keep in the
// uniform registers (so that what is computed from it -- loop bounds, plane
// addresses, constants -- stays there too).  It does so only where control
// flow is provably the same for all lanes: tickets and work items broadcast by
// shuffles instead, or a loop over tickets around the sweep, made it load every
// constant into vector registers and spill (66 -> 57 us a step; the batch with
// its constants read from shared memory 92.6 us, this way 79.4).
__device__ __forceinline__ int uniform(int v) { return (int)__reduce_or_sync(kAll, (unsigned)v); }

// The constants of a lattice of a batch: its own, from shared memory into
// uniform registers, and those of the scheme, from the kernel's parameters.
__device__ __forceinline__ SweepConsts lattice_consts(const SweepConsts &own, const SweepConsts &scheme) {
  SweepConsts k = scheme;
  static_assert(offsetof(SweepConsts, one) == kLatticeConsts * sizeof(float2), "the lattice's come first");
  const float2 *src = &own.T;
  float2 *dst = &k.T;
#pragma unroll
  for (int i = 0; i < kLatticeConsts; ++i) {
    const float v = __int_as_float(uniform(__float_as_int(src[i].x)));
    dst[i] = make_float2(v, v);
  }
  return k;
}

// Density and velocity of a state: the same sweep, stages A to C only.  Reads
// the populations once (36 or 20 bytes a site) and writes the three fields.
template <class St, class Mom>
__global__ void __launch_bounds__(kThreads, Form<St, true>::kMinBlocks)
sweep_moments_kernel(const __grid_constant__ CUtensorMap tin, const __grid_constant__ CUtensorMap tdev,
                     const __grid_constant__ SweepArgs A, const Mom M) {
  const StepIO O{A.fin, A.fdin, nullptr, nullptr, nullptr, 0u, nullptr, nullptr, nullptr, 0.0};
  (void)sweep_body<St, true>(&tin, &tdev, A, A.k, O, blockIdx.x, blockIdx.y, nullptr, false, WaitGrid{}, NoDone{}, M);
}

// Batched step: CTA b works on items[b] (instance, strip, segment) of a
// work list over many independent lattices.  Arguments and tensor maps of
// each instance sit in device memory for both buffer parities; an instance
// reads buffer (item.par0 ^ kpar).
template <class St, bool kTau1>
__global__ void __launch_bounds__(kThreads, Form<St, kTau1>::kMinBlocks)
sweep_batch_kernel(const BatchItem *__restrict__ items, const SweepArgs *__restrict__ args,
                   const __grid_constant__ SweepConsts scheme, const CUtensorMap *__restrict__ maps, int kpar,
                   int records) {
  __shared__ SweepArgs A;
  BatchItem it = items[blockIdx.x];
  it = {uniform(it.inst), uniform(it.strip), uniform(it.seg), uniform(it.rec), uniform(it.par0)};
  const int par = it.par0 ^ kpar;
  const CUtensorMap *m = maps + 4 * it.inst + 2 * par;  // [instance][input buffer][map]
  stage_args(A, args + 2 * it.inst + par);
  const SweepConsts K = lattice_consts(A.k, scheme);
  if (threadIdx.x == 0) {
    // the maps were written through the generic proxy (a host copy)
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(m) : "memory");
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(m + 1) : "memory");
  }
  __syncwarp();
  const StepIO O{A.fin, A.fdin, A.fout, A.fdev, A.partials, 0u, nullptr, nullptr, nullptr, 0.0};
  (void)sweep_body<St, kTau1>(m, m + 1, A, K, O, it.strip, it.seg, A.partials + 4 * (size_t)it.rec, records != 0);
}

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(unsigned *p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Multi-step sweeps.  One launch runs P.nsteps steps: one CTA per (step, item),
// each taking its ticket from a counter as it starts, in step-major order,
// items in work-list order.  Instead of a grid-wide barrier between steps, every
// item (one tile of one lattice) carries a completion counter done[item]
// (the steps it has finished, offset by P.epoch): before step k of an item,
// its threads wait until every item it depends on -- the tiles of the same
// lattice whose stored sites (ghost images included) its TMA boxes read,
// and the tiles whose boxes read its own sites (they must have read the
// buffer it is about to overwrite) -- has reached epoch + k.  A tile starts
// as soon as its neighbourhood has finished the previous step and an SM has
// room for it, so SMs do not idle at step boundaries; lattices of a batch
// never wait for one another.  A CTA waits only for smaller tickets, and
// those belong to CTAs that have started before it (the counter hands them out
// in that order) and keep their place until they end, so the smallest
// unfinished ticket always has its dependencies done and can proceed, however
// many CTAs are resident.  Every wait is bounded: on give-up the CTA sets the
// lattice's error flag (bit 4 for a dependency wait) and stops, and the items
// that depend on it give up in turn (a waiting CTA looks at the flag too).

// The next ticket (lane 0 draws).
__device__ __forceinline__ unsigned next_ticket(const MultiArgs &P) {
  unsigned v = 0;
  if (threadIdx.x == 0) v = atomicAdd(P.next, 1u);
  return (unsigned)uniform((int)v);
}

// Bounded wait of the warp (one lane per dependency) until every item item i
// depends on has finished `target` steps; false on give-up.  (Loops with one
// exit, closed by a warp barrier: the warp is whole afterwards.)
__device__ __forceinline__ bool wait_deps(const MultiArgs &P, int i, unsigned target, int *err) {
  const int d1 = P.dep_ofs[i + 1];
  uint32_t n = 0;
  for (int d = P.dep_ofs[i] + (int)threadIdx.x; d < d1; d += kThreads) {
    const unsigned *f = P.done + P.dep_idx[d];
    while ((int)(ld_acquire_gpu(f) - target) < 0 && n < kWaitLimit) {
      n = (n & 1023u) == 1023u && __ldcg(err) != 0 ? kWaitLimit : n + 1;
      __nanosleep(P.poll_ns);
    }
  }
  __syncwarp();
  if (__any_sync(kAll, n >= kWaitLimit)) {
    if (threadIdx.x == 0) atomicOr(err, 4);
    return false;
  }
  // the neighbours' stores, made visible by the acquires, for this warp's TMA
  // (async proxy) reads
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncwarp();
  return true;
}

// Release item i's step: its stores (generic proxy) before the counter,
// ordered for the neighbours' TMA (async proxy) reads.
__device__ __forceinline__ void release_item(const MultiArgs &P, int i, unsigned value) {
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncwarp();
  if (threadIdx.x == 0) st_release_gpu(P.done + i, value);
}

// Batched form: items[i] names the lattice, tile and record; arguments and
// tensor maps of every lattice (both buffer parities) in device memory.
template <class St, bool kTau1>
__global__ void __launch_bounds__(kThreads, Form<St, kTau1>::kMinBlocks)
sweep_batch_multi_kernel(const BatchItem *__restrict__ items, const SweepArgs *__restrict__ args,
                         const __grid_constant__ SweepConsts scheme, const CUtensorMap *__restrict__ maps,
                         const MultiArgs P) {
  __shared__ SweepArgs A;
  const unsigned tk = next_ticket(P);
  const int k = (int)(tk / (unsigned)P.nitems), i = (int)(tk % (unsigned)P.nitems);
  const unsigned target = P.epoch + (unsigned)k;
  BatchItem it = items[i];
  it = {uniform(it.inst), uniform(it.strip), uniform(it.seg), uniform(it.rec), uniform(it.par0)};
  const int par = it.par0 ^ ((P.kpar0 + k) & 1);
  const CUtensorMap *m = maps + 4 * it.inst + 2 * par;  // [instance][input buffer][map]
  stage_args(A, args + 2 * it.inst + par);
  const SweepConsts K = lattice_consts(A.k, scheme);
  if (threadIdx.x == 0) {
    // the maps were written through the generic proxy (a host copy)
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(m) : "memory");
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(m + 1) : "memory");
  }
  const StepIO O{A.fin, A.fdin, A.fout, A.fdev, A.partials, 0u, nullptr, nullptr, nullptr, 0.0};
  (void)sweep_body<St, kTau1, true, true>(m, m + 1, A, K, O, it.strip, it.seg, A.partials + 4 * (size_t)it.rec,
                                          k == P.nsteps - 1, [&] { return wait_deps(P, i, target, A.err); },
                                          [&] { release_item(P, i, target + 1u); });
}

// Single-lattice form: item i is tile i (tile column i % nstrips, segment
// i / nstrips); arguments and maps are kernel parameters.  The last step
// writes the per-tile records and the warp that finishes last adds them into
// `total` (mass, momentum, flags); while monitoring, every step does so into
// its own record slot and writes its record into the host ring.
template <class St, bool kTau1>
__global__ void __launch_bounds__(kThreads, Form<St, kTau1>::kMinBlocks)
sweep_multi_kernel(const __grid_constant__ CUtensorMap tin0, const __grid_constant__ CUtensorMap tdev0,
                   const __grid_constant__ CUtensorMap tin1, const __grid_constant__ CUtensorMap tdev1,
                   const __grid_constant__ SweepArgs A, const MultiArgs P, const MultiOut Q) {
  const unsigned tk = next_ticket(P);
  const int k = (int)(tk / (unsigned)P.nitems), i = (int)(tk % (unsigned)P.nitems);
  const unsigned target = P.epoch + (unsigned)k;
  const int par = (P.kpar0 + k) & 1;  // input buffer of step k
  const bool last = k == P.nsteps - 1;
  const bool mon = Q.mon_ring != nullptr;
  StepIO O;
  O.fin = par ? Q.fout[0] : Q.fout[1];  // (the step that reads buffer b writes buffer b ^ 1)
  O.fdin = par ? Q.fdev[0] : Q.fdev[1];
  O.fout = par ? Q.fout[1] : Q.fout[0];  // (no dynamic indexing of the parameter space)
  O.fdev = par ? Q.fdev[1] : Q.fdev[0];
  O.recs = mon ? Q.mon_recs + 4 * (size_t)P.nitems * k : A.partials;
  O.nrec = (unsigned)P.nitems;
  O.arrivals = mon ? Q.mon_arr + k : (last ? Q.arrivals : nullptr);
  O.total = last ? Q.total : nullptr;
  O.monitor = mon ? Q.mon_ring + 6 * ((Q.mon_step0 + k) % Q.mon_cap) : nullptr;
  O.mon_step = (double)(Q.mon_step0 + k);
  if (!sweep_body<St, kTau1, true>(par ? &tin1 : &tin0, par ? &tdev1 : &tdev0, A, A.k, O, i % A.nstrips, i / A.nstrips,
                                   const_cast<double *>(O.recs) + 4 * (size_t)i, (last && Q.total) || mon,
                                   [&] { return wait_deps(P, i, target, A.err); },
                                   [&] { release_item(P, i, target + 1u); })) {
    if (threadIdx.x == 0 && Q.total) Q.total[4] = 1.0;  // the sums of this launch will not be written
  }
}

namespace {

// cuTensorMapEncodeTiled through the runtime's driver entry point.
typedef CUresult (*encode_tiled_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                    const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                    const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

cudaError_t encode_map(CUtensorMapDataType type, int esize, void *base, int pitch, int ny, long long plane,
                       int nplanes, int box_cols, CUtensorMap *map) {
  static encode_tiled_fn encode = nullptr;
  if (!encode) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    encode = (encode_tiled_fn)fn;
  }
  // 3D view (column, padded row, plane); one box = box_cols columns x 2
  // rows x nplanes planes.
  const cuuint64_t dims[3] = {(cuuint64_t)pitch, (cuuint64_t)(ny + 8), (cuuint64_t)nplanes};
  const cuuint64_t strides[2] = {(cuuint64_t)pitch * esize, (cuuint64_t)plane * esize};
  const cuuint32_t box[3] = {(cuuint32_t)box_cols, 2, (cuuint32_t)nplanes};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = encode(map, type, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

int quantum_of(int store) {
  return store == kStoreF32 || store == kStoreF32Odd ? StoreF32::kQuantum : (store == kStoreBF16 ? StoreBF16::kQuantum : StoreFP16::kQuantum);
}
int maxw_of(int store) {
  return store == kStoreF32 || store == kStoreF32Odd ? StoreF32::kMaxW : (store == kStoreBF16 ? StoreBF16::kMaxW : StoreFP16::kMaxW);
}

template <class St, bool kTau1>
cudaError_t prepare_one(size_t *smem_bytes) {
  *smem_bytes = sizeof(SmemOf<St, kTau1>);
  const int bytes = (int)*smem_bytes;
  constexpr cudaFuncAttribute attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(sweep_step_kernel<St, kTau1>, attr, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(sweep_multi_kernel<St, kTau1>, attr, bytes);
  if constexpr (!St::kOdd) {  // (a batch takes no odd widths)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sweep_batch_kernel<St, kTau1>, attr, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sweep_batch_multi_kernel<St, kTau1>, attr, bytes);
  }
  return e;
}

template <class St, bool kTau1>
cudaError_t launch_batch_one(const BatchItem *items, int nitems, const SweepArgs *args, const SweepConsts &k,
                             const CUtensorMap *maps,
                             int kpar, int records, size_t smem, cudaStream_t st) {
  sweep_batch_kernel<St, kTau1><<<nitems, kThreads, smem, st>>>(items, args, k, maps, kpar, records);
  return cudaGetLastError();
}

template <class St, bool kTau1>
cudaError_t launch_one(const CUtensorMap &m0, const CUtensorMap &m1, const SweepArgs &A, size_t smem,
                       cudaStream_t st) {
  return pdl::launch(sweep_step_kernel<St, kTau1>, dim3((unsigned)A.nstrips, (unsigned)A.nseg), kThreads, smem, st, m0,
                     m1, A);
}

// The multi-step kernels: one CTA per (step, item).
cudaLaunchConfig_t multi_config(const MultiArgs &P, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)P.nsteps * (unsigned)P.nitems);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  return cfg;
}

template <class St, bool kTau1>
cudaError_t launch_batch_multi_one(const BatchItem *items, const SweepArgs *args, const SweepConsts &k, const CUtensorMap *maps,
                                   const MultiArgs &P, size_t smem, cudaStream_t st) {
  const cudaLaunchConfig_t cfg = multi_config(P, smem, st);
  return cudaLaunchKernelEx(&cfg, sweep_batch_multi_kernel<St, kTau1>, items, args, k, maps, P);
}

template <class St, bool kTau1>
cudaError_t launch_multi_one(const CUtensorMap (&m)[2][2], const SweepArgs &A, const MultiArgs &P,
                             const MultiOut &Q, size_t smem, cudaStream_t st) {
  const cudaLaunchConfig_t cfg = multi_config(P, smem, st);
  return cudaLaunchKernelEx(&cfg, sweep_multi_kernel<St, kTau1>, m[0][0], m[0][1], m[1][0], m[1][1], A, P, Q);
}

template <class St, class T, bool kRows = false>
cudaError_t launch_moments_one(const CUtensorMap &m0, const CUtensorMap &m1, const SweepArgs &A, void *n, void *ux,
                               void *uy, cudaStream_t st) {
  const int smem = (int)sizeof(SmemOf<St, true>);
  using Mom = Moments<T, kRows>;
  cudaError_t e = cudaFuncSetAttribute(sweep_moments_kernel<St, Mom>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const uintptr_t all = (uintptr_t)n | (uintptr_t)ux | (uintptr_t)uy;  // (even nx: rows keep the alignment)
  const Mom M{(T *)n, (T *)ux, (T *)uy, all % (2 * sizeof(T)) == 0 && A.nx % 2 == 0};
  return pdl::launch(sweep_moments_kernel<St, Mom>, dim3((unsigned)A.nstrips, (unsigned)A.nseg), kThreads, (size_t)smem,
                     st, m0, m1, A, M);
}

}  // namespace

bool sweep_supported(int store, int nx, int ny) {
  if (store != kStoreF32 && store != kStoreF32Odd && store != kStoreBF16 && store != kStoreFP16) return false;
  const double pitch = (double)(((nx + 8 + 31) / 32) * 32);
  return (nx % quantum_of(store) == 0) == (store != kStoreF32Odd) && nx >= 8 && ny >= 8 && 9.0 * pitch * (double)(ny + 8) < 2147483647.0;
}

size_t sweep_buffer_bytes(int store, long long plane) {
  return store == kStoreF32 || store == kStoreF32Odd ? 9 * (size_t)plane * sizeof(float) : (size_t)plane * (sizeof(float) + 8 * 2);
}

cudaError_t sweep_make_maps(int store, void *base, int pitch, int ny, long long plane, CUtensorMap *m0,
                            CUtensorMap *m1) {
  if (store == kStoreF32 || store == kStoreF32Odd) {
    static_assert(StoreF32::kTxBytes == 9 * 2 * kCols * sizeof(float), "TMA box must match the slot");
    cudaError_t e = encode_map(CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, pitch, ny, plane, 9, kCols, m0);
    *m1 = *m0;
    return e;
  }
  static_assert(StoreBF16::kRestBytes == 2 * kCols * sizeof(float) && StoreBF16::kDevBytes == 2 * kCols * 8 * 2 &&
                    StoreFP16::kTxBytes == StoreBF16::kTxBytes,
                "TMA boxes must match the slot");
  cudaError_t e = encode_map(CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, pitch, ny, plane, 1, kCols, m0);
  if (e != cudaSuccess) return e;
  void *dev = static_cast<char *>(base) + (size_t)plane * sizeof(float);
  return encode_map(store == kStoreBF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, dev,
                    pitch, ny, plane, 8, kCols, m1);
}

void sweep_strips(int store, int nx, int nstrips, int *base_w, int *extra) {
  const int qn = quantum_of(store), whole = (nx + qn - 1) / qn * qn;  // (the last strip loses whole - nx)
  *base_w = qn * (whole / (qn * nstrips));
  *extra = (whole - *base_w * nstrips) / qn;
}

int sweep_min_strips(int store, int nx) { return (nx + maxw_of(store) - 1) / maxw_of(store); }

int sweep_warps_per_sm(int store, bool tau1) {
  return store == kStoreBF16 || store == kStoreFP16 ? Form<StoreBF16, true>::kMinBlocks
                            : (tau1 ? Form<StoreF32, true>::kMinBlocks : Form<StoreF32, false>::kMinBlocks);
}

int sweep_seg_rule(double cols, int ny, int resident, bool batch) {
  const double rows = ny * cols / ((batch ? kTilesPerWarpBatch : kTilesPerWarp) * std::max(resident, 1));
  const int h = rows < 3.0 ? 2 : std::min(kSegMax, 4 * std::max(1, (int)(rows / 4.0 + 0.5)));
  return std::min(ny, h);
}

// Where the device holds more warps than three quarters of a step's tiles need,
// the others wait for most of a step, and their looks at the counters (a lane
// per dependency, some 20 of them) slow the tiles that run: 256 ns between
// them.  Measured per step against 64 ns: FP32 64 x 32 8.5 -> 7.45 us, 256 x 128
// 11.6 -> 9.7, 512 x 256 (0.70 of the warps) 9.6 -> 8.7; batches of four lattices
// of 64 x 32 7.1 -> 6.2, of 128 x 64 9.4 -> 6.9.  Nearer to one tile a warp the
// waits are short and end late with 256 ns: 768 x 256 (0.98) 9.5 us at 64, 10.2
// at 256; from 1024 x 256 on there is no difference.
unsigned sweep_poll_ns(int nitems, int resident) { return 4ll * nitems <= 3ll * resident ? 256u : 64u; }

void sweep_plan(int store, int nx, int ny, int *nstrips, int *seg_h) {
  *nstrips = sweep_min_strips(store, nx);
  *seg_h = std::min(ny, kSegMax);
}

int sweep_tile_cols(int store, int nx, int nstrips) {
  int base = 0, extra = 0;
  sweep_strips(store, nx, nstrips, &base, &extra);
  return base + (extra > 0 ? quantum_of(store) : 0) <= kTileW ? nstrips : (nx + kTileW - 1) / kTileW;
}

// f<storage policy, tau == 1>() for the runtime pair (store, tau1): the formats
// a batch takes, and those of a single lattice.
#define LB_SWEEP_BATCH_FORM(store, tau1, f, ...)                                                       \
  switch (store) {                                                                                     \
    case kStoreF32: return (tau1) ? f<StoreF32, true>(__VA_ARGS__) : f<StoreF32, false>(__VA_ARGS__);    \
    case kStoreBF16: return (tau1) ? f<StoreBF16, true>(__VA_ARGS__) : f<StoreBF16, false>(__VA_ARGS__); \
    case kStoreFP16: return (tau1) ? f<StoreFP16, true>(__VA_ARGS__) : f<StoreFP16, false>(__VA_ARGS__); \
  }                                                                                                    \
  return cudaErrorInvalidValue
#define LB_SWEEP_FORM(store, tau1, f, ...)                                                             \
  if (store == kStoreF32Odd)                                                                           \
    return (tau1) ? f<StoreF32Odd, true>(__VA_ARGS__) : f<StoreF32Odd, false>(__VA_ARGS__);            \
  LB_SWEEP_BATCH_FORM(store, tau1, f, __VA_ARGS__)

cudaError_t sweep_prepare(int store, bool tau1, size_t *smem_bytes) {
  LB_SWEEP_FORM(store, tau1, prepare_one, smem_bytes);
}

cudaError_t launch_sweep(int store, bool tau1, const CUtensorMap &m0, const CUtensorMap &m1, const SweepArgs &A,
                         size_t smem, cudaStream_t st) {
  LB_SWEEP_FORM(store, tau1, launch_one, m0, m1, A, smem, st);
}

cudaError_t launch_sweep_moments(int store, const CUtensorMap &m0, const CUtensorMap &m1, const SweepArgs &A, void *n,
                                 void *ux, void *uy, int dtype, bool host, cudaStream_t st) {
  if (host && store == kStoreF32Odd)
    return dtype == 0 ? launch_moments_one<StoreF32Odd, double, true>(m0, m1, A, n, ux, uy, st)
                      : launch_moments_one<StoreF32Odd, float, true>(m0, m1, A, n, ux, uy, st);
  switch (store) {
    case kStoreF32:
      return dtype == 0 ? launch_moments_one<StoreF32, double>(m0, m1, A, n, ux, uy, st)
                        : launch_moments_one<StoreF32, float>(m0, m1, A, n, ux, uy, st);
    case kStoreF32Odd:
      return dtype == 0 ? launch_moments_one<StoreF32Odd, double>(m0, m1, A, n, ux, uy, st)
                        : launch_moments_one<StoreF32Odd, float>(m0, m1, A, n, ux, uy, st);
    case kStoreBF16:
      return dtype == 0 ? launch_moments_one<StoreBF16, double>(m0, m1, A, n, ux, uy, st)
                        : launch_moments_one<StoreBF16, float>(m0, m1, A, n, ux, uy, st);
    case kStoreFP16:
      return dtype == 0 ? launch_moments_one<StoreFP16, double>(m0, m1, A, n, ux, uy, st)
                        : launch_moments_one<StoreFP16, float>(m0, m1, A, n, ux, uy, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_sweep_batch(int store, bool tau1, const BatchItem *items, int nitems, const SweepArgs *args,
                               const SweepConsts &k, const CUtensorMap *maps, int kpar, int records, size_t smem, cudaStream_t st) {
  if (nitems < 1) return cudaSuccess;
  LB_SWEEP_BATCH_FORM(store, tau1, launch_batch_one, items, nitems, args, k, maps, kpar, records, smem, st);
}

cudaError_t launch_sweep_multi(int store, bool tau1, const CUtensorMap (&maps)[2][2], const SweepArgs &A,
                               const MultiArgs &P, const MultiOut &Q, size_t smem, cudaStream_t st) {
  LB_SWEEP_FORM(store, tau1, launch_multi_one, maps, A, P, Q, smem, st);
}

cudaError_t launch_sweep_batch_multi(int store, bool tau1, const BatchItem *items, const SweepArgs *args,
                                     const SweepConsts &k, const CUtensorMap *maps, const MultiArgs &P, size_t smem, cudaStream_t st) {
  LB_SWEEP_BATCH_FORM(store, tau1, launch_batch_multi_one, items, args, k, maps, P, smem, st);
}

// Tiles each tile of the sweep depends on (see sweep_batch_multi_kernel): the
// owners of every site its TMA boxes read -- `window` columns from x0-4 and
// rows ya-4 .. yb+4, periodic images mapped back to the site they copy
// (rows outside the lattice with walls are never written) -- and,
// symmetrically, every tile whose window reads its sites.  A tile (s, g)
// reads the product of the columns C(s) and the segments G(g); its list is
// C(s) x G(g) and the same of the transposed relations, in index order.
void sweep_deps(int store, int nx, int ny, int walls, int ncol, int base_w, int extra, int seg_h, int window,
                std::vector<int> &ofs, std::vector<int> &idx) {
  const int qn = quantum_of(store);
  const int nseg = (ny + seg_h - 1) / seg_h;
  auto col_of = [&](int x) {
    const int wide = extra * (base_w + qn);
    return x < wide ? x / (base_w + qn) : extra + (x - wide) / base_w;
  };
  // per column / segment: (index, 1: read by it | 2: reads it), in index order
  struct Rel {
    int i, how;
  };
  auto relation = [](int n, auto &&reads) {
    std::vector<std::vector<Rel>> r(n);
    std::vector<std::vector<int>> out(n), in(n);
    for (int a = 0; a < n; ++a) {
      reads(a, out[a]);
      std::sort(out[a].begin(), out[a].end());
      out[a].erase(std::unique(out[a].begin(), out[a].end()), out[a].end());
      for (int b : out[a]) in[b].push_back(a);  // ascending in a
    }
    for (int a = 0; a < n; ++a) {
      size_t p = 0, q = 0;
      while (p < out[a].size() || q < in[a].size()) {
        const int b = p == out[a].size() ? in[a][q] : (q == in[a].size() ? out[a][p] : std::min(out[a][p], in[a][q]));
        int how = 0;
        if (p < out[a].size() && out[a][p] == b) how |= 1, ++p;
        if (q < in[a].size() && in[a][q] == b) how |= 2, ++q;
        r[a].push_back({b, how});
      }
    }
    return r;
  };
  const auto cols = relation(ncol, [&](int s, std::vector<int> &v) {
    const int x0 = s * base_w + qn * std::min(s, extra);
    for (int x = x0 - 4; x < x0 - 4 + window; ++x) {
      const int c = col_of(((x % nx) + nx) % nx);
      if (v.empty() || v.back() != c) v.push_back(c);
    }
  });
  const auto segs = relation(nseg, [&](int g, std::vector<int> &v) {
    const int ya = g * seg_h, yb = std::min(ny, ya + seg_h);
    for (int y = ya - 4; y <= yb + 4; ++y) {
      if (walls && (y < 0 || y >= ny)) continue;
      const int h = (((y % ny) + ny) % ny) / seg_h;
      if (v.empty() || v.back() != h) v.push_back(h);
    }
  });
  ofs.assign((size_t)ncol * nseg + 1, 0);
  idx.clear();
  for (int g = 0; g < nseg; ++g)
    for (int s = 0; s < ncol; ++s) {
      for (const Rel &v : segs[g])
        for (const Rel &c : cols[s])
          if (v.how & c.how) idx.push_back(c.i + ncol * v.i);
      ofs[(size_t)s + (size_t)ncol * g + 1] = (int)idx.size();
    }
}

}  // namespace lbk
