// tc_device.cuh -- pieces shared by the kernels that use the fifth-generation
// tensor cores (gemm_tc.cu, fno_fused.cu): mbarrier waits, matrix and
// instruction descriptors, TMA loads, tensor memory.
#pragma once

#include <cstdint>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace tc {

constexpr int kBM = 128;                     // rows of an MMA (accumulator lanes)
constexpr int kBK = 64;                      // K columns of an operand tile: one 128-byte swizzle row
constexpr uint32_t kWaitLimit = 1u << 24;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < kWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Shared-memory matrix descriptor of a K-major, 128-byte swizzled operand
// tile (tcgen05 format): start address >> 4 in bits 0-13, leading byte
// offset (unused for swizzled K-major operands) 0, stride byte offset
// (between 8-row groups: 1024 bytes) >> 4 in bits 32-45, descriptor version
// 1 in bits 46-47, swizzle mode 128 B (2) in bits 61-63.
__device__ __forceinline__ uint64_t kmajor_sw128_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// The same for 64-byte rows (K = 32): 64-byte swizzle (4), eight rows 512 bytes.
__device__ __forceinline__ uint64_t kmajor_sw64_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9 and 10-12 = 1, the same type for both), both K-major (bits 15,
// 16 = 0), N >> 3 in bits 17-22, M >> 4 in bits 24-28.
template <int BN>
__host__ __device__ constexpr uint32_t idesc_bf16() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

__device__ __forceinline__ void tma_load_3d(const CUtensorMap *map, uint32_t dst, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}


__device__ __forceinline__ void mbar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}

// D = A B^T on `nk` K = 16 steps of two K-major tiles with rows of kRow bytes
// (one thread issues).
template <int kRow>
__device__ __forceinline__ void mma_tile(uint32_t tmem, uint32_t a, uint32_t b, int nk, uint32_t idesc) {
  static_assert(kRow == 128 || kRow == 64, "swizzle rows");
  for (int j = 0; j < nk; ++j) {  // K = 16 per MMA: 32 bytes along the swizzle row
    const uint64_t ad = kRow == 128 ? kmajor_sw128_desc(a + 32 * j) : kmajor_sw64_desc(a + 32 * j);
    const uint64_t bd = kRow == 128 ? kmajor_sw128_desc(b + 32 * j) : kmajor_sw64_desc(b + 32 * j);
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(j > 0 ? 1u : 0u)
        : "memory");
  }
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Eight accumulator columns of this warp's 32 rows: lane = row.
__device__ __forceinline__ void tmem_load8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace tc
