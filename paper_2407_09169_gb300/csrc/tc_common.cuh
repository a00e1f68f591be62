// PTX wrappers (mbarrier, TMA, tcgen05, TMEM) and bit-level FP64 / FP32
// conversions shared by the tensor-core GEMM kernels.
#pragma once

#include <cuda.h>
#include <cstdint>

#include "gemm_tc.cuh"

namespace qtt {

namespace {

constexpr int BM = 128;
constexpr long long kWaitLimit = 1LL << 26;  // try_wait iterations before giving up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after kWaitLimit polls or 2 s of wall time.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const unsigned long long t0 = global_ns();
  for (long long it = 0; it < kWaitLimit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255) == 255 && global_ns() - t0 > 2000000000ull) return false;
  }
  return false;
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, uint64_t* bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::
          "r"(smem_u32(dst)),
      "l"((uint64_t)tm), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

template <bool TF32>
__device__ __forceinline__ void mma_issue(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if (TF32)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::
            "r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::
            "r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major tile written by TMA with the
// 128-byte swizzle: rows of 128 bytes, 8-row atoms 1024 bytes apart.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused with this swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;          // stride byte offset: next 8-row atom
  d |= (uint64_t)1 << 46;                    // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                    // 128-byte swizzle
  return d;
}

// Instruction descriptor: D f32, A/B of type `fmt` (bf16 = 1, tf32 = 2),
// both K-major, M = 128, N = bn.
__host__ __device__ constexpr uint32_t make_idesc(uint32_t fmt, uint32_t bn) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((bn >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

// ---------------------------------------------------------------------------
// Conversions between FP64 and FP32 by bit manipulation.  The FP64 pipe of
// this GPU issues two operations per clock per SM, so the packing and the
// epilogue (which touch every operand and output element) use only integer
// and FP32 instructions.

// float -> double, exact (zero, normal, inf and NaN by bits; denormals, which
// the accumulators of these products do not produce in practice, by the
// hardware conversion).
__device__ __forceinline__ unsigned long long float_to_double_bits(uint32_t f) {
  const uint32_t e = (f >> 23) & 0xFFu;
  const unsigned long long sign = (unsigned long long)(f >> 31) << 63;
  if (e == 0u) {
    if ((f & 0x7FFFFFu) == 0u) return sign;
    return (unsigned long long)__double_as_longlong((double)__uint_as_float(f));
  }
  const unsigned long long de = (e == 0xFFu) ? 0x7FFull : (unsigned long long)(e + 896u);
  return sign | (de << 52) | ((unsigned long long)(f & 0x7FFFFFu) << 29);
}

// S 2^scale as a double, exact for |S| < 2^53; results below the normal range
// flush to zero.
__device__ __forceinline__ unsigned long long int_to_double_bits(long long S, int scale) {
  if (S == 0) return 0ull;
  const unsigned long long sign = S < 0 ? (1ull << 63) : 0ull;
  const unsigned long long a = (unsigned long long)(S < 0 ? -S : S);
  const int lz = __clzll((long long)a);
  const int ex = (63 - lz) + 1023 + scale;  // a = 1.m 2^(63 - lz)
  if (ex <= 0) return sign;
  if (ex >= 2047) return sign | (0x7FFull << 52);
  const unsigned long long mant = ((a << lz) << 1) >> 12;  // drop the leading one, keep 52 bits
  return sign | ((unsigned long long)ex << 52) | mant;
}

// double -> float, round to nearest even; results below the normal float
// range flush to zero, results above it become infinities.
__device__ __forceinline__ float double_bits_to_float(unsigned long long u) {
  const uint32_t sign = (uint32_t)(u >> 32) & 0x80000000u;
  const int e = (int)((u >> 52) & 0x7FFull);
  const unsigned long long m = u & 0xFFFFFFFFFFFFFull;
  if (e == 0x7FF) return __uint_as_float(sign | 0x7F800000u | (m ? 0x400000u : 0u));
  const int fe = e - 1023 + 127;
  if (fe <= 0) return __uint_as_float(sign);
  if (fe >= 255) return __uint_as_float(sign | 0x7F800000u);
  const unsigned long long rem = m & 0x1FFFFFFFull;  // 29 dropped bits
  uint32_t r = ((uint32_t)fe << 23) | (uint32_t)(m >> 29);
  if (rem > 0x10000000ull || (rem == 0x10000000ull && (r & 1u))) r += 1u;  // a carry into the exponent is correct
  return __uint_as_float(sign | r);
}

// |x| as an order-preserving integer (the bits of a non-negative double).
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// x 2^k by exponent arithmetic (x normal, result normal or flushed to zero).
__device__ __forceinline__ unsigned long long scale_bits(unsigned long long u, int k) {
  const int e = (int)((u >> 52) & 0x7FFull);
  if (e == 0) return u & (1ull << 63);  // zero (or a denormal, flushed)
  const int ne = e + k;
  if (ne <= 0) return u & (1ull << 63);
  if (ne >= 2047) return (u & (1ull << 63)) | (0x7FFull << 52);
  return (u & ~(0x7FFull << 52)) | ((unsigned long long)ne << 52);
}

__host__ __device__ constexpr int tmem_cols_for(int cols) {
  return cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
}

__device__ __forceinline__ float to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// Row exponent for the exact slices: |x| < 2^e for every x of the row (0 for
// an all-zero row), from the bits of the largest magnitude.
__device__ __forceinline__ int row_exponent(unsigned long long maxbits) {
  const int E = (int)(maxbits >> 52);
  return E == 0 ? 0 : E - 1022;
}

}  // namespace

}  // namespace qtt
