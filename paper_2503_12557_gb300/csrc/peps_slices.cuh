// Digit slices for FP64-accurate products on the tensor cores (see peps_gram_sl.cu for the number
// format and why every product is exact): shared by the Gram kernel and the Cholesky update.
#pragma once
#include <cuda_bf16.h>

#include "peps_tma.cuh"

namespace peps {
namespace {

constexpr int NS = 7;                        // digits
constexpr int SM_ = 128;                     // tile rows and columns
constexpr int CK = 32;                       // columns of Obar per stage (64 bytes: one 64B-swizzle row)
constexpr int SSTAGES = 2;
constexpr int STILE = SM_ * CK * 2;          // 8 KB: one digit of one row block
constexpr int SOPND = NS * STILE;            // 56 KB
constexpr int SSTAGE = 2 * SOPND;            // 112 KB
constexpr int EPI_WARPS = 8;
constexpr int SL_THREADS = (EPI_WARPS + 2) * 32;
constexpr int ROW_NONFINITE = -1;

// Fixed-point integer (below 2^55) of the double with bits b in a row whose largest biased
// exponent is E: x 2^(1077 - E), rounded half to even (ties are half of the entries that lose one bit:
// half up in magnitude, the diagonal of a Gram matrix came out 1e-16 too large).
__device__ __forceinline__ long long fixed_point(unsigned long long b, int E) {
  const int ex = (int)(b >> 52) & 0x7ff;
  const int sh = E - max(ex, 1);
  unsigned long long m = (b & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0ull);
  m <<= 2;
  if (sh > 0) m = sh < 60 ? (m + (1ull << (sh - 1)) - 1 + ((m >> sh) & 1)) >> sh : 0ull;
  return (b >> 63) ? -(long long)m : (long long)m;
}
// The NS signed digits of q, as BF16, into position j of eight packed per digit
__device__ __forceinline__ void put_digits(long long q, int j, uint32_t (&w)[NS][4]) {
#pragma unroll
  for (int p = NS - 1; p >= 0; --p) {
    const int d = p ? (int)(signed char)(q & 0xff) : (int)q;
    if (p) q = (q - d) >> 8;
    const uint32_t h = (uint32_t)__bfloat16_as_ushort(__int2bfloat16_rn(d));
    if (j & 1) w[p][j >> 1] |= h << 16;
    else w[p][j >> 1] = h;
  }
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          smem_u32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// K-major operand tile of 128 rows x 32 bf16 in the 64-byte swizzle: 8-row groups 512 bytes apart
// (stride byte offset), layout code 4 at bits [61, 64); the other fields as for 128 bytes.
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | (1ull << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}
constexpr uint32_t SL_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(SM_ >> 3) << 17) | ((uint32_t)(SM_ >> 4) << 24);
__device__ __forceinline__ void mma_sl(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(SL_IDESC), "r"(acc));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// bounded wait that also gives up when another role of the CTA has failed
__device__ __forceinline__ bool wait_ok(uint64_t* bar, uint32_t parity, int* failed) {
  if (mbar_try(bar, parity)) return true;
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
  do {
    if (mbar_try(bar, parity)) return true;
    if (*(volatile int*)failed) return false;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  } while (t - t0 < 1000000000ull);  // one second; a unit takes microseconds
  atomicExch(failed, 1);
  return false;
}
// 16 accumulator columns of this warp's 32 tensor-memory lanes
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
  uint32_t u[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
        "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
      : "r"(addr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(u[i]);
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// integer of an exact FP32 integer |v| <= 2^22
__device__ __forceinline__ int f2i_exact(float v) { return __float_as_int(__fadd_rn(v, 12582912.f)) - 0x4B400000; }

}  // namespace
}  // namespace peps
