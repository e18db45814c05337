// fno_fused.cu -- forward and backward of the network's layers and projection
// (include/fno.h) as fused tensor-core kernels, for the width the warm start
// uses (32 channels, 32 or 64 hidden).
//
// A tile is 128 sites of one lattice row: the rows of an MMA.  (Rows that leave
// part of the last tile empty, 64 or 136 sites, leave that part of the
// accumulators and of the epilogue's lanes idle; the kernels are the faster ones
// all the same, see below.)  Per site the
// layer is two products with K <= 64 -- the channel mixing (the site-major
// BF16 copy of v against W) and the inverse x-transform (the table FxiT[x][j]
// against the 2 modes_x transformed values of each channel at this y) -- so one
// CTA brings all four operand tiles by TMA (128-byte swizzle, zero fill where
// K < 64), one thread issues the MMAs into two accumulators in tensor memory,
// and each of the four warps then holds 32 sites by all 32 channels in
// registers: bias, activation, and every copy the next products need (BF16
// channel-major and site-major), with no pass over memory of its own.  The
// backward kernels do the same with the transposed operands, multiply by
// gelu', and add the tile's channel sums (weight gradients of the biases, the
// lift and the projection) with a shuffle tree in FP32, FP64 across warps and
// tiles.
//
// The separate kernels this replaces moved every FP32 activation through memory
// four to six times (z written by one product, read and written by the next,
// then by the bias and activation, then transposed: 570 MB a layer for 8 fields
// of 512 x 128 against 170 here).  The sums of a product are grouped as before
// (each product in its own accumulator, then added, then the bias), so a
// layer's values are the same bits.  Bound by the activations (normcdff) and
// by memory about equally.  Measured: training step of 16 fields of 256 x 64
// 1.61 -> 1.07 ms, of 8 fields of 512 x 128 2.74 -> 1.65 ms (0.86 and 1.27 with
// the weight gradients beside them and launches overlapped), of 16 fields of 64 x
// 64 0.86 -> 0.57 and of 32 x 16 0.61 -> 0.39; warm start of a 2048 x 512 lattice
// (forward pass, fields, initial state) 2.36 -> 0.83 ms.
#include "fno_fused.h"

#include <algorithm>

#include "fno_math.cuh"
#include "gemm_tc.h"
#include "pdl.cuh"
#include "tc_device.cuh"

namespace fno {

namespace {

constexpr int kThreads = 128;
constexpr int C = kWidth;

// The tile of a block: tiles of a row in turn, then rows, all along the grid's
// x (its y ends at 65,535: fewer than a field's rows may be), fields along z.
struct Tile {
  int x, y, b;
};
__device__ __forceinline__ Tile tile_of(int nx) {
  const unsigned across = (unsigned)(nx + tc::kBM - 1) / tc::kBM, y = blockIdx.x / across;
  return {(int)(blockIdx.x - y * across) * tc::kBM, (int)y, (int)blockIdx.z};
}

// Operand tiles of a layer kernel; kK: K columns of a tile (32 where 2 modes_x
// allows, with 64-byte swizzle rows: half the shared memory, twice the CTAs).
template <int kK>
struct __align__(1024) LayerSmem {
  __nv_bfloat16 a1[tc::kBM * kK], a2[tc::kBM * kK];
  __nv_bfloat16 b1[C * kK], b2[C * kK];
  unsigned long long full, done;
  uint32_t tmem;
};

// Tensor memory of a CTA: `cols` columns (a power of two >= 32), and the
// barriers' initialisation; all threads.
__device__ __forceinline__ uint32_t setup(uint32_t *slot, uint32_t cols, unsigned long long *bars, int nbars) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < nbars; ++i) tc::mbar_init(tc::smem_u32(bars + i));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(slot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return *slot;
}
__device__ __forceinline__ void release_tmem(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
  }
}

// The MMAs a thread issued are complete (every thread calls it); false after a
// bounded wait that gave up.
__device__ __forceinline__ bool wait_done(unsigned long long *bar, int *err) {
  const bool ok = tc::mbar_try(tc::smem_u32(bar), 0u);
  if (!ok && (threadIdx.x & 31) == 0) atomicOr(err, 1);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return ok;
}

// Sums of v[0..7] over the warp's lanes: lane l returns that of v[l >> 2] (the
// first three stages halve the values a lane still carries).
__device__ __forceinline__ float warp_sums(const float (&v)[8]) {
  const int lane = threadIdx.x & 31;
  float h[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) h[i] = v[i];
#pragma unroll
  for (int o = 4; o >= 1; o >>= 1) {
    const bool up = lane & (4 * o);
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float send = up ? h[i] : h[i + o], keep = up ? h[i + o] : h[i];
      h[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * o);
    }
  }
  h[0] += __shfl_xor_sync(0xffffffffu, h[0], 2);
  return h[0] + __shfl_xor_sync(0xffffffffu, h[0], 1);
}

// Sums of eight channels over groups of four sites (the lanes 4g .. 4g+3),
// ((x0 + x1) + (x2 + x3)) as a float4 sum of a row takes them, into quads[c][s / 4]
// (lanes of valid sites; rows are whole groups of four).
__device__ __forceinline__ void put_quads(const float (&v)[8], bool valid, float *quads, long long S4, long long s) {
  const int lane = threadIdx.x & 31;
  float h[4], q[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float send = lane & 1 ? v[i] : v[i + 4], keep = lane & 1 ? v[i + 4] : v[i];
    h[i] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float send = lane & 2 ? h[i] : h[i + 2], keep = lane & 2 ? h[i + 2] : h[i];
    q[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  if (!valid) return;
  const int c0 = 4 * (lane & 1) + 2 * ((lane >> 1) & 1);
#pragma unroll
  for (int i = 0; i < 2; ++i) quads[(c0 + i) * S4 + (s >> 2)] = q[i];
}

// Eight channels of a site as BF16: channel-major (32 sites of a channel are
// consecutive) and 16 bytes of the site's row of the site-major copy.
__device__ __forceinline__ void put_bf16(const float (&v)[8], bool valid, __nv_bfloat16 *cm, long long S,
                                         __nv_bfloat16 *sm) {
  if (!valid) return;
  __align__(16) __nv_bfloat16 h[8];
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    h[o] = __float2bfloat16_rn(v[o]);
    cm[o * S] = h[o];
  }
  *reinterpret_cast<uint4 *>(sm) = *reinterpret_cast<const uint4 *>(h);
}

// x, as a value of its own to the compiler: gelu and gelu' of the same z are
// then contracted as they are in the kernels that evaluate one of them (with a
// shared normcdff result, or Phi recovered from gelu', the last bit of gelu'
// changes, and with it BF16 roundings of the whole backward pass).
__device__ __forceinline__ float opaque(float x) {
  asm volatile("" : "+f"(x));
  return x;
}

enum Mode { kForward, kForwardLast, kBackward, kBackwardFirst };

struct LayerArgs {
  int nx, ny, K2;
  const float *w;               // forward: bias
  float *z;                     // forward: z (out)
  const float *zprev;           // backward: z of the layer below
  __nv_bfloat16 *cm, *sm;       // results
  float *quads;                 // backward: sums of dz over groups of four sites
  float *dv;                    // backward, first layer: dv
  int *err;
};

// One tile (x0 .. x0+127 of row y, field b) through both products.  The
// epilogue takes eight channels at a time (unrolled over all 32 its code did
// not fit the instruction cache: 1.05 of 6.7 stall cycles an instruction).
template <int kMode, int kK>
__global__ void __launch_bounds__(kThreads, kK == 32 ? 8 : 5)
layer_kernel(const __grid_constant__ CUtensorMap ma1, const __grid_constant__ CUtensorMap mb1,
             const __grid_constant__ CUtensorMap ma2, const __grid_constant__ CUtensorMap mb2, const LayerArgs p) {
  pdl::begin();
  extern __shared__ unsigned char raw[];
  using Sm = LayerSmem<kK>;
  Sm &S = *reinterpret_cast<Sm *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const Tile T = tile_of(p.nx);
  const int xt = T.x, y = T.y, b = T.b;
  const uint32_t tmem = setup(&S.tmem, 64, &S.full, 2);
  if (t == 0) {
    const uint32_t bar = tc::smem_u32(&S.full);
    constexpr uint32_t tx = 2 * (tc::kBM + C) * kK * 2;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(tx) : "memory");
    tc::tma_load_3d(&ma1, tc::smem_u32(S.a1), bar, 0, xt, b * p.ny + y);
    tc::tma_load_3d(&mb1, tc::smem_u32(S.b1), bar, 0, 0, 0);
    tc::tma_load_3d(&ma2, tc::smem_u32(S.a2), bar, 0, xt, 0);
    tc::tma_load_3d(&mb2, tc::smem_u32(S.b2), bar, 0, b * C, y);
    if (tc::mbar_try(bar, 0u)) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      constexpr uint32_t idesc = tc::idesc_bf16<C>();
      tc::mma_tile<2 * kK>(tmem, tc::smem_u32(S.a1), tc::smem_u32(S.b1), C / 16, idesc);
      tc::mma_tile<2 * kK>(tmem + C, tc::smem_u32(S.a2), tc::smem_u32(S.b2), p.K2 / 16, idesc);
    } else {  // (the copies in flight land before the CTA leaves: waited for once more)
      atomicOr(p.err, 1);
      (void)tc::mbar_try(bar, 0u);
    }
    tc::mma_commit(tc::smem_u32(&S.done));
  }
  __syncthreads();
  (void)wait_done(&S.done, p.err);

  const int x = xt + warp * 32 + lane;
  const bool valid = x < p.nx;
  const long long sites = (long long)p.nx * p.ny, s = (long long)y * p.nx + x;
  const long long row = (long long)b * C * sites + s;
  const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
  for (int c0 = 0; c0 < C; c0 += 8) {
    float v[8], u[8];
    tc::tmem_load8(lanes + c0, v);      // the channel mixing
    tc::tmem_load8(lanes + C + c0, u);  // the transform
    const long long e = row + c0 * sites;
    __nv_bfloat16 *cm = p.cm + e, *sm = p.sm + ((long long)b * sites + s) * C + c0;
    if constexpr (kMode == kForward || kMode == kForwardLast) {
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const float zz = (u[o] + v[o]) + p.w[c0 + o];
        if (valid) p.z[e + o * sites] = zz;
        v[o] = kMode == kForward ? gelu(zz) : zz;
      }
      put_bf16(v, valid, cm, sites, sm);
    } else if constexpr (kMode == kBackward) {
      float z[8];
#pragma unroll
      for (int o = 0; o < 8; ++o) z[o] = valid ? p.zprev[e + o * sites] : 0.f;
#pragma unroll
      for (int o = 0; o < 8; ++o) u[o] = (v[o] + u[o]) * gelu_grad(z[o]);
      put_bf16(u, valid, cm, sites, sm);
      put_quads(u, valid, p.quads + ((long long)b * C + c0) * (sites / 4), sites / 4, s);
    } else {
#pragma unroll
      for (int o = 0; o < 8; ++o)
        if (valid) p.dv[e + o * sites] = v[o] + u[o];
    }
  }
  release_tmem(tmem, 64);
}

// Features of a site (include/fno.h).
__device__ __forceinline__ void features(const float *prm, int b, int x, int y, int ny, float *f) {
  const float uw = prm[4 * b], a0 = prm[4 * b + 1], lam = prm[4 * b + 2], tr = prm[4 * b + 3];
  float sn, cs;
  sincospif(2.0f * (float)x / lam, &sn, &cs);
  const float yy = 2.0f * (float)y / (float)(ny - 1) - 1.0f;
  f[0] = (a0 / 1e-3f) * sn;
  f[1] = (a0 / 1e-3f) * cs;
  f[2] = (uw / 0.05f) * yy;
  f[3] = (tr - 0.94f) / 0.02f;
  f[4] = yy;
}

__global__ void __launch_bounds__(kThreads)
lift_kernel(int nx, int ny, const float *__restrict__ prm, const float *__restrict__ P, const float *__restrict__ pb,
            float *__restrict__ x0, __nv_bfloat16 *__restrict__ cm, __nv_bfloat16 *__restrict__ sm) {
  pdl::begin();
  __shared__ float Ps[C * kFeat], ps[C];
  for (int i = threadIdx.x; i < C * kFeat; i += kThreads) Ps[i] = P[i];
  if (threadIdx.x < C) ps[threadIdx.x] = pb[threadIdx.x];
  __syncthreads();
  const Tile T = tile_of(nx);
  const int x = T.x + threadIdx.x, y = T.y, b = T.b;
  if (x >= nx) return;
  const long long sites = (long long)nx * ny, s = (long long)y * nx + x;
  float f[kFeat];
  features(prm, b, x, y, ny, f);
#pragma unroll
  for (int c = 0; c < kFeat; ++c) x0[((long long)b * kFeat + c) * sites + s] = f[c];
#pragma unroll
  for (int c0 = 0; c0 < C; c0 += 8) {
    float v[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      float acc = ps[c0 + o];
#pragma unroll
      for (int c = 0; c < kFeat; ++c) acc += Ps[(c0 + o) * kFeat + c] * f[c];
      v[o] = acc;
    }
    put_bf16(v, true, cm + ((long long)b * C + c0) * sites + s, sites, sm + ((long long)b * sites + s) * C + c0);
  }
}

// ---------------------------------------------------------- the projection

constexpr int kMaxO = 4;

template <int H>
struct __align__(1024) ProjSmem {
  __nv_bfloat16 a[tc::kBM * tc::kBK];   // v tile (K = C); then dhp tile (K = H)
  __nv_bfloat16 b1[H * tc::kBK];        // Q1 [h][c]
  __nv_bfloat16 b2[C * tc::kBK];        // Q1^T [c][h] (backward)
  float q1[H], Q2[kMaxO * H], q2[kMaxO];
  double red[4][H * (1 + kMaxO) + kMaxO + 1];
  unsigned long long full, done, done2;
  uint32_t tmem;
};

struct ProjArgs {
  int nx, ny, O;
  const float *q1, *Q2, *q2;
  float *out, *out_user;        // forward
  const float *o_in, *target;   // backward
  float scale;                  // 2 / (elements of out)
  __nv_bfloat16 *dhp, *cm, *sm;
  float *quads;
  double *part;
  int *err;
};

template <int H, bool kBack>
__global__ void __launch_bounds__(kThreads, kBack ? 4 : 5)
project_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb1,
               const __grid_constant__ CUtensorMap mb2, const ProjArgs p) {
  pdl::begin();
  extern __shared__ unsigned char raw[];
  using Sm = ProjSmem<H>;
  Sm &S = *reinterpret_cast<Sm *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const Tile T = tile_of(p.nx);
  const int xt = T.x, y = T.y, b = T.b;
  constexpr uint32_t kCols = kBack ? 128 : H;  // accumulators: H, then C (a power of two in all)
  for (int i = t; i < H; i += kThreads) S.q1[i] = p.q1[i];
  for (int i = t; i < p.O * H; i += kThreads) S.Q2[i] = p.Q2[i];
  if (!kBack && t < p.O) S.q2[t] = p.q2[t];
  const uint32_t tmem = setup(&S.tmem, kCols, &S.full, 3);
  if (t == 0) {
    const uint32_t bar = tc::smem_u32(&S.full);
    const uint32_t tx = (uint32_t)(tc::kBM + H + (kBack ? C : 0)) * tc::kBK * 2;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(tx) : "memory");
    tc::tma_load_3d(&ma, tc::smem_u32(S.a), bar, 0, xt, b * p.ny + y);
    tc::tma_load_3d(&mb1, tc::smem_u32(S.b1), bar, 0, 0, 0);
    if (kBack) tc::tma_load_3d(&mb2, tc::smem_u32(S.b2), bar, 0, 0, 0);
    if (tc::mbar_try(bar, 0u)) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      tc::mma_tile<128>(tmem, tc::smem_u32(S.a), tc::smem_u32(S.b1), C / 16, tc::idesc_bf16<H>());
    } else {
      atomicOr(p.err, 1);
      (void)tc::mbar_try(bar, 0u);
    }
    tc::mma_commit(tc::smem_u32(&S.done));
  }
  __syncthreads();
  (void)wait_done(&S.done, p.err);

  const int r = warp * 32 + lane, x = xt + r;
  const bool valid = x < p.nx;
  const long long sites = (long long)p.nx * p.ny, s = (long long)y * p.nx + x;
  const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
  if constexpr (!kBack) {
    float acc[kMaxO];
#pragma unroll
    for (int j = 0; j < kMaxO; ++j) acc[j] = j < p.O ? S.q2[j] : 0.f;
#pragma unroll 1
    for (int h0 = 0; h0 < H; h0 += 8) {
      float v[8];
      tc::tmem_load8(lanes + h0, v);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float a = gelu(v[i] + S.q1[h0 + i]);
#pragma unroll
        for (int j = 0; j < kMaxO; ++j)
          if (j < p.O) acc[j] += S.Q2[j * H + h0 + i] * a;
      }
    }
    if (valid) {
      for (int j = 0; j < p.O; ++j) {
        const long long e = ((long long)b * p.O + j) * sites + s;
        p.out[e] = acc[j];
        if (p.out_user) p.out_user[e] = acc[j];
      }
    }
  } else {
    // d loss / d out of this site, and the loss
    float dout[kMaxO];
    double loss = 0.0;
#pragma unroll
    for (int j = 0; j < kMaxO; ++j) {
      dout[j] = 0.f;
      if (j < p.O && valid) {
        const long long e = ((long long)b * p.O + j) * sites + s;
        const float d = p.o_in[e] - p.target[e];
        dout[j] = p.scale * d;
        loss += (double)d * (double)d;
      }
    }
    unsigned char *arow = reinterpret_cast<unsigned char *>(S.a) + r * 128;  // this site's row of the dhp tile
#pragma unroll 1
    for (int h0 = 0; h0 < H; h0 += 8) {
      float a[8], d[8];
      tc::tmem_load8(lanes + h0, a);
      __nv_bfloat16 *dh = p.dhp + ((long long)b * H + h0) * sites + s;
      __align__(16) __nv_bfloat16 hb[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float z = a[i] + S.q1[h0 + i];
        float q = 0.f;
#pragma unroll
        for (int j = 0; j < kMaxO; ++j)
          if (j < p.O) q += S.Q2[j * H + h0 + i] * dout[j];
        d[i] = q * gelu_grad(z);
        a[i] = gelu(opaque(z));
        hb[i] = __float2bfloat16_rn(d[i]);
        if (valid) dh[i * sites] = hb[i];
      }
      // 16-byte chunk c of row r sits at chunk c ^ (r & 7) (128-byte swizzle)
      *reinterpret_cast<uint4 *>(arow + (((h0 / 8) ^ (r & 7)) << 4)) = *reinterpret_cast<const uint4 *>(hb);
      const float ds = warp_sums(d);
      if ((lane & 3) == 0) S.red[warp][h0 + (lane >> 2)] = (double)ds;
#pragma unroll
      for (int j = 0; j < kMaxO; ++j) {
        if (j >= p.O) break;
#pragma unroll
        for (int i = 0; i < 8; ++i) d[i] = dout[j] * a[i];
        const float as = warp_sums(d);
        if ((lane & 3) == 0) S.red[warp][H + j * H + h0 + (lane >> 2)] = (double)as;
      }
    }
    // dv = Q1^T dhp: the tile just written against Q1^T
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (t == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      tc::mma_tile<128>(tmem + H, tc::smem_u32(S.a), tc::smem_u32(S.b2), H / 16, tc::idesc_bf16<C>());
      tc::mma_commit(tc::smem_u32(&S.done2));
    }
    __syncwarp();
    (void)wait_done(&S.done2, p.err);
#pragma unroll 1
    for (int c0 = 0; c0 < C; c0 += 8) {
      float v[8];
      tc::tmem_load8(lanes + H + c0, v);
      put_bf16(v, valid, p.cm + ((long long)b * C + c0) * sites + s, sites, p.sm + ((long long)b * sites + s) * C + c0);
      put_quads(v, valid, p.quads + ((long long)b * C + c0) * (sites / 4), sites / 4, s);
    }
    const int base = H * (1 + p.O), n = base + p.O + 1;
    double tail[kMaxO + 1];
#pragma unroll
    for (int j = 0; j < kMaxO; ++j) tail[j] = (double)dout[j];
    tail[kMaxO] = loss;
#pragma unroll
    for (int j = 0; j <= kMaxO; ++j)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) tail[j] += __shfl_down_sync(0xffffffffu, tail[j], o);
    if (lane == 0) {
      for (int j = 0; j < p.O; ++j) S.red[warp][base + j] = j == 0 ? tail[0] : (j == 1 ? tail[1] : (j == 2 ? tail[2] : tail[3]));
      S.red[warp][base + p.O] = tail[kMaxO];
    }
    __syncthreads();
    double *part = p.part + ((long long)b * gridDim.x + blockIdx.x) * n;
    for (int i = t; i < n; i += kThreads) part[i] = ((S.red[0][i] + S.red[1][i]) + S.red[2][i]) + S.red[3][i];
  }
  release_tmem(tmem, kCols);
}

// ------------------------------------------------------------- tile sums

constexpr int kSumWarps = 8, kSumSplits = 16;

// Block (k, q) adds values 32k .. 32k+31 over tiles q, q + 16, ...: warp w every
// eighth of them, four loads in flight; then the warps' sums in order, into
// split q of part2.
__global__ void __launch_bounds__(32 * kSumWarps)
tile_sums_kernel(const double *__restrict__ part, long long tiles, int nval, double *__restrict__ part2) {
  pdl::begin();
  __shared__ double ws[kSumWarps][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  double acc = 0.0;
  if (i < nval) {
    constexpr long long step = kSumWarps * kSumSplits;
    long long k = blockIdx.y + (long long)w * kSumSplits;
    for (; k + 3 * step < tiles; k += 4 * step) {
      double v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = part[(k + q * step) * nval + i];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc += v[q];
    }
    for (; k < tiles; k += step) acc += part[k * nval + i];
  }
  ws[w][lane] = acc;
  __syncthreads();
  if (w == 0 && i < nval) {
    double r = ws[0][lane];
    for (int q = 1; q < kSumWarps; ++q) r += ws[q][lane];
    part2[blockIdx.y * nval + i] = r;
  }
}

// The splits' sums, in order, into up to three ranges of outputs and the loss.
__global__ void finish_kernel(const double *__restrict__ part2, int nval, SumOut o0, SumOut o1, SumOut o2,
                              double *__restrict__ loss, double count) {
  pdl::begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nval) return;
  double r = part2[i];
  for (int q = 1; q < kSumSplits; ++q) r += part2[q * nval + i];
  int e = i;
  const SumOut o[3] = {o0, o1, o2};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (e >= 0 && e < o[q].n) o[q].out[e] = (float)r;
    e -= o[q].n;
  }
  if (e == 0) *loss = r / count;
}

dim3 tile_grid(const Shape &s) {
  return dim3((unsigned)((s.nx + tc::kBM - 1) / tc::kBM) * (unsigned)s.ny, 1, (unsigned)s.B);
}

template <class K>
cudaError_t allow_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

struct LayerMaps {
  CUtensorMap a1, b1, a2, b2;
};

cudaError_t layer_maps(const Shape &s, const __nv_bfloat16 *a1, const __nv_bfloat16 *b1, const __nv_bfloat16 *a2,
                       const __nv_bfloat16 *b2, LayerMaps *m) {
  const int kk = s.K2 <= 32 ? 32 : 64;
  cudaError_t e = tc::operand_map(a1, C, s.nx, C, (long long)s.nx * C, s.B * s.ny, tc::kBM, &m->a1, kk);
  if (e == cudaSuccess) e = tc::operand_map(b1, C, C, C, 0, 1, C, &m->b1, kk);
  if (e == cudaSuccess) e = tc::operand_map(a2, s.K2, s.nx, s.K2, 0, 1, tc::kBM, &m->a2, kk);
  // rows: the channels of all fields at one y
  if (e == cudaSuccess) e = tc::operand_map(b2, s.K2, s.B * C, s.ny * s.K2, s.K2, s.ny, C, &m->b2, kk);
  return e;
}

template <int kMode, int kK>
cudaError_t launch_layer_k(const Shape &s, const LayerMaps &m, const LayerArgs &p, cudaStream_t st) {
  const size_t smem = sizeof(LayerSmem<kK>) + 1024;
  const cudaError_t e = allow_smem(layer_kernel<kMode, kK>, smem);
  if (e != cudaSuccess) return e;
  return pdl::launch(layer_kernel<kMode, kK>, tile_grid(s), kThreads, smem, st, m.a1, m.b1, m.a2, m.b2, p);
}
template <int kMode>
cudaError_t launch_layer(const Shape &s, const LayerMaps &m, const LayerArgs &p, cudaStream_t st) {
  return s.K2 <= 32 ? launch_layer_k<kMode, 32>(s, m, p, st) : launch_layer_k<kMode, 64>(s, m, p, st);
}

template <int H, bool kBack>
cudaError_t launch_project(const Shape &s, const __nv_bfloat16 *v_sm, const __nv_bfloat16 *Q1, const __nv_bfloat16 *Q1T,
                           const ProjArgs &p, cudaStream_t st) {
  CUtensorMap ma, mb1, mb2;
  cudaError_t e = tc::operand_map(v_sm, C, s.nx, C, (long long)s.nx * C, s.B * s.ny, tc::kBM, &ma);
  if (e == cudaSuccess) e = tc::operand_map(Q1, C, H, C, 0, 1, H, &mb1);
  mb2 = mb1;
  if (e == cudaSuccess && kBack) e = tc::operand_map(Q1T, H, C, H, 0, 1, C, &mb2);
  const size_t smem = sizeof(ProjSmem<H>) + 1024;
  if (e == cudaSuccess) e = allow_smem(project_kernel<H, kBack>, smem);
  if (e != cudaSuccess) return e;
  return pdl::launch(project_kernel<H, kBack>, tile_grid(s), kThreads, smem, st, ma, mb1, mb2, p);
}

}  // namespace

// The sizes the tiles are laid out for; other networks take the separate
// products and pointwise kernels of fno.cu.
bool fused_supported(int width, int hidden, int modes_x) {
  return width == C && (hidden == 32 || hidden == 64) && modes_x % 8 == 0 && 2 * modes_x <= tc::kBK;
}

long long fused_tiles(const Shape &s) { return (long long)((s.nx + tc::kBM - 1) / tc::kBM) * s.ny * s.B; }

cudaError_t lift(const Shape &s, const float *prm, const float *P, const float *pb, float *x0, __nv_bfloat16 *cm,
                 __nv_bfloat16 *sm, cudaStream_t st) {
  return pdl::launch(lift_kernel, tile_grid(s), kThreads, 0, st, s.nx, s.ny, prm, P, pb, x0, cm, sm);
}

cudaError_t layer_forward(const Shape &s, const __nv_bfloat16 *v_sm, const __nv_bfloat16 *W, const float *w,
                          const __nv_bfloat16 *G, const __nv_bfloat16 *FxiT, bool last, float *z, __nv_bfloat16 *cm,
                          __nv_bfloat16 *sm, int *err, cudaStream_t st) {
  LayerMaps m;
  const cudaError_t e = layer_maps(s, v_sm, W, FxiT, G, &m);
  if (e != cudaSuccess) return e;
  const LayerArgs p{s.nx, s.ny, s.K2, w, z, nullptr, cm, sm, nullptr, nullptr, err};
  return last ? launch_layer<kForwardLast>(s, m, p, st) : launch_layer<kForward>(s, m, p, st);
}

cudaError_t project_forward(const Shape &s, const __nv_bfloat16 *v_sm, const __nv_bfloat16 *Q1, const float *q1,
                            const float *Q2, const float *q2, float *out, float *out_user, int *err, cudaStream_t st) {
  ProjArgs p{};
  p.nx = s.nx;
  p.ny = s.ny;
  p.O = s.O;
  p.q1 = q1;
  p.Q2 = Q2;
  p.q2 = q2;
  p.out = out;
  p.out_user = out_user;
  p.err = err;
  return s.H == 64 ? launch_project<64, false>(s, v_sm, Q1, nullptr, p, st)
                   : launch_project<32, false>(s, v_sm, Q1, nullptr, p, st);
}

int project_back_sums(const Shape &s) { return s.H * (1 + s.O) + s.O + 1; }

cudaError_t project_backward(const Shape &s, const __nv_bfloat16 *v_sm, const __nv_bfloat16 *Q1, const float *q1,
                             const float *Q2, const __nv_bfloat16 *Q1T, const float *out, const float *target,
                             __nv_bfloat16 *dhp, __nv_bfloat16 *dz_cm, __nv_bfloat16 *dz_sm, float *quads, double *part,
                             int *err, cudaStream_t st) {
  ProjArgs p{};
  p.nx = s.nx;
  p.ny = s.ny;
  p.O = s.O;
  p.q1 = q1;
  p.Q2 = Q2;
  p.o_in = out;
  p.target = target;
  p.scale = 2.0f / (float)((long long)s.B * s.O * s.nx * s.ny);
  p.dhp = dhp;
  p.cm = dz_cm;
  p.sm = dz_sm;
  p.quads = quads;
  p.part = part;
  p.err = err;
  return s.H == 64 ? launch_project<64, true>(s, v_sm, Q1, Q1T, p, st)
                   : launch_project<32, true>(s, v_sm, Q1, Q1T, p, st);
}

cudaError_t layer_backward(const Shape &s, const __nv_bfloat16 *dz_sm, const __nv_bfloat16 *WT, const __nv_bfloat16 *dA,
                           const __nv_bfloat16 *Fx, const float *zprev, __nv_bfloat16 *cm, __nv_bfloat16 *sm,
                           float *quads, float *dv, int *err, cudaStream_t st) {
  LayerMaps m;
  const cudaError_t e = layer_maps(s, dz_sm, WT, Fx, dA, &m);
  if (e != cudaSuccess) return e;
  const LayerArgs p{s.nx, s.ny, s.K2, nullptr, nullptr, zprev, cm, sm, quads, dv, err};
  return zprev ? launch_layer<kBackward>(s, m, p, st) : launch_layer<kBackwardFirst>(s, m, p, st);
}

cudaError_t finish_sums(const double *part, long long tiles, int nval, const SumOut (&o)[3], double *loss, double count,
                        double *part2, cudaStream_t st) {
  (void)pdl::launch(tile_sums_kernel, dim3((nval + 31) / 32, kSumSplits), 32 * kSumWarps, 0, st, part, tiles, nval,
                    part2);
  return pdl::launch(finish_kernel, (nval + 127) / 128, 128, 0, st, part2, nval, o[0], o[1], o[2], loss, count);
}

long long finish_scratch(int nval) { return (long long)kSumSplits * nval; }

}  // namespace fno
