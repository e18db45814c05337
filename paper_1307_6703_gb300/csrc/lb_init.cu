// lb_init.cu -- initial states of the FP32 and 16-bit lattices: f*_i =
// f_i^eq(n0, u0) (Eq. eqfunc of arXiv:1307.6703), each population the FP64
// value rounded to FP32, in one pass that also writes the ghost band and, for
// 16-bit storage, the storage format.
//
// The equilibrium is evaluated in double-FP32 arithmetic (a value as the sum of
// two floats; error-free transformations of Dekker, Numer. Math. 18 (1971) 224,
// and Knuth, TAOCP 2, 4.2.2), good to 2^-43 for densities and velocities within
// the bounds below.  A population that lies so close to the middle of two floats
// that this does not decide its rounding (one in 2^17), and a site whose fields
// are outside the bounds -- infinities and NaN among them -- are evaluated in
// FP64.  FP64 for every site runs at 1/64 of the FP32 rate on this part and bound
// the kernel: 4096 x 1024 from noise 174 us, 2048 x 512 from density and velocity
// 850 us.  Now bound by memory: 36 (FP32) or 20 (16-bit) bytes written a site, and
// 8 bytes read per field given; 4096 x 1024 FP32 from noise 24.9 us, from a density
// 44.7, with one velocity 77 (25.5, 45.0 and 71 if nothing were decided again).
#include <algorithm>
#include <cmath>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lb_device.cuh"
#include "lb_internal.h"
#include "pdl.cuh"

namespace lbk {

namespace {

// ------------------------------------------------- double-FP32 arithmetic

struct Ff {
  float h, l;
};

__device__ __forceinline__ Ff ff_sum(float a, float b) {  // a + b exactly
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Ff ff_add(Ff a, Ff b) {
  const Ff s = ff_sum(a.h, b.h);
  const float e = __fadd_rn(s.l, __fadd_rn(a.l, b.l));
  const float h = __fadd_rn(s.h, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s.h))};
}
__device__ __forceinline__ Ff ff_neg(Ff a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Ff ff_mul(Ff a, Ff b) {
  const float p = __fmul_rn(a.h, b.h);
  return {p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)))};
}
// a, known to within d, as a float; where that leaves two, `links` are marked
// undecided.
__device__ __forceinline__ float ff_round(Ff a, float d, unsigned links, unsigned &open) {
  const float lo = __fadd_rn(a.h, __fsub_rn(a.l, d)), hi = __fadd_rn(a.h, __fadd_rn(a.l, d));
  if (lo != hi) open |= links;
  return lo;
}

// A double as two floats: its first 24 bits and the remaining 29 (rounded to
// 24), by integer arithmetic; out of the range where that is exact (tiny,
// huge, non-finite values) the rounded value alone.
__device__ __forceinline__ Ff ff_of(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  if (e > -70 && e < 127) {
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const float h = __uint_as_float(sign | ((unsigned)(e + 127) << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
    const float scale = __uint_as_float(sign | ((unsigned)(e - 52 + 127) << 23));
    return {h, __fmul_rn((float)((unsigned)b & 0x1fffffffu), scale)};
  }
  return {(float)d, 0.f};
}

// -------------------------------------------------------------- the kernel

// Geometry of a state buffer and what the sites are set to.
struct InitArgs {
  int nx, ny, pitch;
  long long plane, off;
  int images;          // write the periodic images into the ghost band: 1 x only (walls), 2 x and y
  uint64_t seed;
  Ff rho, amp;         // noise: n0 = rho + amp x, x in [-1, 1)
  const double *n0, *ux, *uy;  // fields (noise: null)
  bool pairs;          // fields aligned for 16-byte loads
  Ff wiso[3];          // w_i (1 + t3_i) of the rest, axis and diagonal links
  Ff iso[3], w[3];     // its factors
  float ref_ax, ref_dg;
  // FP64 forms, and the error of the double-FP32 ones: each population is known
  // to within `slack` times its class's w_i n
  double rho64, amp64, t3[3];
  float slack;
};

// Where the double-FP32 arithmetic is good to `slack`: densities that leave room
// for the low parts, velocities at which no sum cancels (terms of at most 0.75
// beside the rest factor's 1 or so).
constexpr unsigned kLinks = 0x1ff;  // all nine
constexpr float kMinN = 0x1p-60f, kMaxN = 0x1p+60f, kMaxU = 0.125f;

// Noise of site s: x = 2 U - 1 with U the top 53 bits of SplitMix64, exact up
// to the last 5 bits.
__device__ __forceinline__ Ff noise_at(uint64_t seed, uint64_t s) {
  const long long j = (long long)(splitmix64_at(seed, s) >> 11) - (1ll << 52);
  return {(float)(int)(j >> 29) * 0x1p-23f, (float)(unsigned)(j & 0x1fffffff) * 0x1p-52f};
}

// Population of link q of a moving site in FP64 (feq9's expressions), rounded
// once.
__device__ __noinline__ float link64(double cu, double n, double u, double v, double w, double t3) {
  constexpr double T0 = Consts<double>::T0, c2 = 2.0 * T0 * T0;
  const double t1 = div_const(cu, T0, 1.0 / T0), t2 = div_const(cu * cu - T0 * (u * u + v * v), c2, 1.0 / c2);
  return (float)(w * n * (((1.0 + t1) + t2) + t3));
}

// Equilibrium of one site.  Class 0: rest, 1: axes, 2: diagonals.  Returns the
// links whose rounding is not decided.
template <bool kMoving>
__device__ __forceinline__ unsigned equilibrium(const InitArgs &A, Ff n, Ff u, Ff v, float *f) {
  unsigned open = 0;
  if (!(fabsf(n.h) >= kMinN && fabsf(n.h) <= kMaxN && fabsf(u.h) <= kMaxU && fabsf(v.h) <= kMaxU)) open = kLinks;
  if constexpr (!kMoving) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const Ff p = ff_mul(A.wiso[c], n);
      const float e = ff_round(p, __fmul_rn(fabsf(p.h), A.slack), kLinks, open);
#pragma unroll
      for (int i = 0; i < 9; ++i)
        if (cx(i) * cx(i) + cy(i) * cy(i) == c) f[i] = e;
    }
  } else {
    // w n (1 + t3 + 3 c.u + 9/2 (c.u)^2 - 3/2 u.u)
    const Ff three{3.f, 0.f}, nine2{4.5f, 0.f}, m32{-1.5f, 0.f};
    const Ff uu = ff_mul(m32, ff_add(ff_mul(u, u), ff_mul(v, v)));
    Ff base[3], wn[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      base[c] = ff_add(A.iso[c], uu);
      wn[c] = ff_mul(A.w[c], n);
    }
    f[0] = ff_round(ff_mul(wn[0], base[0]), __fmul_rn(fabsf(wn[0].h), A.slack), 1u, open);
    // the four directions and their opposites
    auto pair = [&](int i, int j, int c, Ff cu) {
      const Ff even = ff_add(base[c], ff_mul(nine2, ff_mul(cu, cu))), odd = ff_mul(three, cu);
      const float d = __fmul_rn(fabsf(wn[c].h), A.slack);
      f[i] = ff_round(ff_mul(wn[c], ff_add(even, odd)), d, 1u << i, open);
      f[j] = ff_round(ff_mul(wn[c], ff_add(even, ff_neg(odd))), d, 1u << j, open);
    };
    pair(1, 3, 1, u);
    pair(2, 4, 1, v);
    pair(5, 7, 2, ff_add(u, v));
    pair(6, 8, 2, ff_add(v, ff_neg(u)));
  }
  return open;
}

// Storage: nine float planes, or the float rest plane and eight 16-bit planes
// of deviations from the reference populations (each rounded to nearest even;
// the rest population takes the remainder of the rounded values, so the site
// keeps the float sum of the nine).
struct PutF32 {
  float *f;
  template <int kCols>
  __device__ __forceinline__ void encode(const InitArgs &, float (*)[9]) {}
  template <int kCols>
  __device__ __forceinline__ void store(const InitArgs &A, long long e, const float (*f9)[9]) const {
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      float *p = f + q * A.plane + e;
      if constexpr (kCols == 2) *reinterpret_cast<float2 *>(p) = make_float2(f9[0][q], f9[1][q]);
      else *p = f9[0][q];
    }
  }
};

template <class H>
struct PutDev {
  float *f;
  H *d;
  H code[2][8];
  __device__ static H enc(float v);
  __device__ static float dec(H v);
  template <int kCols>
  __device__ __forceinline__ void encode(const InitArgs &A, float (*f9)[9]) {
#pragma unroll
    for (int c = 0; c < kCols; ++c) {
      float *g = f9[c];
      const float n = (((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]))) + g[8];
#pragma unroll
      for (int q = 1; q < 9; ++q) {
        const float r = q <= 4 ? A.ref_ax : A.ref_dg;
        code[c][q - 1] = enc(g[q] - r);
        g[q] = r + dec(code[c][q - 1]);
      }
      g[0] = n - (((g[1] + g[3]) + (g[2] + g[4])) + ((g[5] + g[7]) + (g[6] + g[8])));
    }
  }
  template <int kCols>
  __device__ __forceinline__ void store(const InitArgs &A, long long e, const float (*f9)[9]) const {
    static_assert(kCols == 2, "16-bit lattices have an even number of columns");
    *reinterpret_cast<float2 *>(f + e) = make_float2(f9[0][0], f9[1][0]);
    struct alignas(4) Two {
      H a, b;
    };
#pragma unroll
    for (int q = 0; q < 8; ++q) *reinterpret_cast<Two *>(d + q * A.plane + e) = Two{code[0][q], code[1][q]};
  }
};
template <>
__device__ __forceinline__ __nv_bfloat16 PutDev<__nv_bfloat16>::enc(float v) { return __float2bfloat16_rn(v); }
template <>
__device__ __forceinline__ float PutDev<__nv_bfloat16>::dec(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ __half PutDev<__half>::enc(float v) { return __float2half_rn(v); }
template <>
__device__ __forceinline__ float PutDev<__half>::dec(__half v) { return __half2float(v); }

// Threads along x (kCols columns each: 2 where the layout keeps pairs of
// columns aligned), blocks strided over rows.
template <class Put, int kCols, bool kMoving>
__global__ void __launch_bounds__(256, kMoving ? 4 : 8) init_f32_kernel(Put put, const __grid_constant__ InitArgs A) {
  pdl::begin();
  const int cols = A.nx / kCols;
  for (int y = blockIdx.y; y < A.ny; y += gridDim.y) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cols; c += gridDim.x * blockDim.x) {
      const int x = c * kCols;
      const size_t s = (size_t)y * A.nx + x;
      float f[kCols][9];
      double n0[kCols], u0[kCols] = {}, v0[kCols] = {};
      // (host fields are read over the link: one 16-byte load per pair)
      auto load = [&](const double *p, double *to) {
        if (kCols == 2 && A.pairs) {
          const double2 d = *reinterpret_cast<const double2 *>(p + s);
          to[0] = d.x;
          to[kCols - 1] = d.y;
        } else {
#pragma unroll
          for (int j = 0; j < kCols; ++j) to[j] = p[s + j];
        }
      };
      if (A.n0 != nullptr) load(A.n0, n0);
      if constexpr (kMoving) {
        if (A.ux != nullptr) load(A.ux, u0);
        if (A.uy != nullptr) load(A.uy, v0);
      }
#pragma unroll
      for (int j = 0; j < kCols; ++j) {
        const Ff n = A.n0 == nullptr ? ff_add(A.rho, ff_mul(A.amp, noise_at(A.seed, s + j))) : ff_of(n0[j]);
        const unsigned open = equilibrium<kMoving>(A, n, ff_of(u0[j]), ff_of(v0[j]), f[j]);
        if (open != 0) {
          const double U = (double)(splitmix64_at(A.seed, s + j) >> 11) * 0x1.0p-53;
          const double m = A.n0 == nullptr ? A.rho64 + A.amp64 * (2.0 * U - 1.0) : n0[j];
#pragma unroll
          for (int q = 0; q < 9; ++q) {
            const double w = Consts<double>::w(q), t3 = A.t3[cx(q) * cx(q) + cy(q) * cy(q)];
            if (!(open >> q & 1u)) continue;
            if constexpr (kMoving) f[j][q] = link64(cx(q) * u0[j] + cy(q) * v0[j], m, u0[j], v0[j], w, t3);
            else f[j][q] = (float)(w * m * (1.0 + t3));
          }
        }
      }
      put.template encode<kCols>(A, f);
      const long long e = A.off + (long long)y * A.pitch + x;
      put.template store<kCols>(A, e, f);
      if (A.images != 0) {  // (with pairs nx is even: columns 0..3 and nx-4..nx-1 are whole pairs)
        const int gx = x < 4 ? A.nx : (x >= A.nx - 4 ? -A.nx : 0);
        if (gx != 0) put.template store<kCols>(A, e + gx, f);
        if (A.images == 2) {
          const long long gy = (y < 4 ? A.ny : (y >= A.ny - 4 ? -A.ny : 0)) * (long long)A.pitch;
          if (gy != 0) {
            put.template store<kCols>(A, e + gy, f);
            if (gx != 0) put.template store<kCols>(A, e + gy + gx, f);
          }
        }
      }
    }
  }
}

template <class Put, int kCols>
cudaError_t launch_cols(const Put &put, const InitArgs &A, cudaStream_t st) {
  const unsigned bx = (unsigned)((A.nx / kCols + 255) / 256);
  const dim3 grid(std::min(bx, 64u), (unsigned)std::min(A.ny, 2048));
  return A.ux != nullptr || A.uy != nullptr ? pdl::launch(init_f32_kernel<Put, kCols, true>, grid, 256, 0, st, put, A)
                                            : pdl::launch(init_f32_kernel<Put, kCols, false>, grid, 256, 0, st, put, A);
}

Ff ff_host(double d) {
  const float h = (float)d;
  return {h, (float)(d - (double)h)};
}

}  // namespace

cudaError_t launch_init_f32(int store, void *buf, const InitState &I, cudaStream_t st) {
  InitArgs A{};
  A.nx = I.nx;
  A.ny = I.ny;
  A.pitch = I.pitch;
  A.plane = I.plane;
  A.off = I.off;
  A.images = I.images;
  A.seed = I.seed;
  A.rho = ff_host(I.rho_mean);
  A.amp = ff_host(I.amp);
  A.n0 = I.n0;
  A.ux = I.ux;
  A.uy = I.uy;
  A.pairs = (((uintptr_t)I.n0 | (uintptr_t)I.ux | (uintptr_t)I.uy) & 15) == 0;
  A.ref_ax = I.ref_ax;
  A.ref_dg = I.ref_dg;
  A.rho64 = I.rho_mean;
  A.amp64 = I.amp;
  const double T0 = 1.0 / 3.0, w[3] = {4.0 / 9.0, 1.0 / 9.0, 1.0 / 36.0};
  for (int c = 0; c < 3; ++c) {
    const double t3 = (I.T - T0) * ((double)c - 2.0 * T0) / (2.0 * T0 * T0), iso = 1.0 + t3;
    A.iso[c] = ff_host(iso);
    A.t3[c] = t3;
    A.w[c] = ff_host(w[c]);
    A.wiso[c] = ff_host(w[c] * iso);
    A.slack = std::max(A.slack, (float)(0x1p-43 * (1.0 + std::abs(iso))));
  }
  float *f = static_cast<float *>(buf);
  void *dev = f + I.plane;  // (16-bit storage: the deviation planes follow the rest plane)
  switch (store) {
    case kStoreBF16: return launch_cols<PutDev<__nv_bfloat16>, 2>({f, (__nv_bfloat16 *)dev}, A, st);
    case kStoreFP16: return launch_cols<PutDev<__half>, 2>({f, (__half *)dev}, A, st);
    case kStoreF32:
    case kStoreF32Odd:
      // pairs of columns: an even number of them, rows and planes of even pitch
      if (I.nx % 2 == 0 && I.pitch % 2 == 0 && I.plane % 2 == 0 && I.off % 2 == 0)
        return launch_cols<PutF32, 2>({f}, A, st);
      return launch_cols<PutF32, 1>({f}, A, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbk
