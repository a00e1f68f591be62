// Tensor-core (tcgen05) GEMM that reads the FP64 operands itself: one launch
// per product, for the products of the sketch and zip-up passes, where one
// operand is a tall stack of rows (up to ~17k) and the other a core, a sketch
// core or Q (at most 288 columns).
//
// Why: the packed GEMM (gemm_tc.cu) takes two to four dependent launches per
// product -- K balancing, row maxima, packing and the product -- that each
// stream the tall operand through memory; at chi = 128 the packing passes took
// as long as the products, and 8-20 us a launch of the chain of sites.  Here a
// CTA owns 128 rows and all (or half) of the columns.  Its 16 warps load a k-block of
// both operands from the strided FP64 views into registers, cut it into the
// slices of the mode and write them to shared memory in the 128-byte-swizzled
// K-major layout that tcgen05.mma reads, while the loads of the next operand
// block are in flight; one thread issues the MMAs into TMEM, asynchronously;
// the epilogue reads TMEM back and writes FP64.  The exact-slice modes first
// pass over the CTA's operands for their exponent fields (16 bits each, kept in
// the stage buffers), from which the power-of-two scales follow: a shift per K
// index that leaves both operands equally large there, then the exponents of
// the rows and columns.
//
// What bounds it: the latency of the loads unless a whole block of each
// operand is in flight (four loads a thread at a time made a 128 x 64 x 128
// product 50 us), then the conversions' integer and FP32 instructions (a tile
// of 128 x 144 x 64 takes ~17k element conversions against ~1.5k clocks of
// MMA).  Rows of all outer batch entries are one flat range when the column
// operand does not depend on the outer index, so ragged bonds fill their
// tiles.  A long K (the range product) is split over CTAs, with the FP64
// reduction of the packed GEMM.  Every wait is bounded.  Steps before and
// after, the other kernels as they were then: 40 sites chi 128 BF16X10 51.2 ->
// 41.5 ms, 30 sites chi 64 FP32 15.4 -> 12.9, an uneven grid chi 77 BF16X10 19.8
// -> 16.0, 20 sites chi 32 BF16X10 11.8 -> 5.4; half the launches (4068 -> 2067
// at chi 128).  Distance to the FP64 path after one step of 30 sites, chi 64
// (geometric mean over eight seeds, packed products -> these): FP32 3.0e-6 ->
// 3.0e-6, BF16X10 3.4e-7 -> 2.4e-7.
#include <cuda_bf16.h>

#include <algorithm>

#include "gemm_tc.cuh"
#include "tc_common.cuh"

namespace qtt {

namespace {

constexpr int FT = 512;          // threads: 16 warps
constexpr int FW = FT / 32;
constexpr int FK_MAX = 512;      // K of one exact-slice product (its shifts sit in shared memory)
constexpr int kAbsent = 4096;    // a shift that takes every value below the smallest one

template <int MODE>
struct FusedTraits;
template <>
struct FusedTraits<TC_TF32X3> {
  static constexpr bool tf32 = true, sliced = false;
  static constexpr int ns = 2, ngroups = 1, kb = 32, exact_kb = 1 << 30;
};
template <>
struct FusedTraits<TC_BF16X6> {
  static constexpr bool tf32 = false, sliced = true;
  static constexpr int ns = 3, ngroups = 3, kb = 64, exact_kb = 5;
};
template <>
struct FusedTraits<TC_BF16X10> {
  static constexpr bool tf32 = false, sliced = true;
  static constexpr int ns = 4, ngroups = 4, kb = 64, exact_kb = 4;
};

struct FusedArgs {
  MatView A, B;       // rows: A.p + o so + m rs + k cs + inner si; columns: B.p + k rs + n cs + inner si
  OutView C;
  int M;              // rows per outer entry
  long long R;        // rows over all outer entries
  int N, K, pieces;   // pieces (TF32X3): the sum of two products, each with its own accumulator
  long long pa, pb;   // offsets of the second piece
  int kblocks, kb_per_split, splitk;
  double alpha, beta;
  double* ws;
  int* err;
};

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// Exponent field of |x|.
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
// The field after a shift by a power of two (zeros stay zero, underflow flushes).
__device__ __forceinline__ int shifted(int E, int s) { return E == 0 ? 0 : max(E + s, 0); }
// Exponent e with |x| < 2^e of the values whose largest exponent field is E (0 for zeros).
__device__ __forceinline__ int field_exponent(int E) { return E == 0 ? 0 : E - 1022; }

// double -> float, round to nearest even; outside the normal float range by
// the general routine.
__device__ __forceinline__ float fast_float(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t h = hi & 0x7FFFFFFFu;
  if (h - 0x38100000u >= 0x47E00000u - 0x38100000u)
    return h < 0x38100000u ? 0.0f : double_bits_to_float((unsigned long long)__double_as_longlong(x));
  uint32_t r = __funnelshift_l(lo, h - 0x38000000u, 3);
  r += (lo >> 28) & ((lo & 0x0FFFFFFFu) ? 1u : (r & 1u)) & 1u;
  return __uint_as_float(r | (hi & 0x80000000u));
}

// The slices of one element as 32-bit words whose upper halves are the bf16
// values (exact-slice modes), or the hi and lo tf32 values.  Exact slices: x
// 2^(8 ns - 1 - c) rounded to an integer by its bits, written in balanced
// base-256 digits (|d| <= 128), largest first; c is the row's exponent less
// the shift of k.  Halves go to even: the operands are often results of such
// products, integers a few bits finer than the grid they are rounded to, and
// halves away from zero grew the mass by 2e-5 in 25 FP32 steps (4e-6 so).
template <int MODE>
__device__ __forceinline__ void cut(double x, int c, uint32_t* s) {
  constexpr int ns = FusedTraits<MODE>::ns;
  if constexpr (MODE == TC_TF32X3) {
    const float f = fast_float(x);
    const float h = to_tf32(f);
    s[0] = __float_as_uint(h);
    s[1] = __float_as_uint(to_tf32(f - h));
  } else {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int E = (int)(hi >> 20) & 0x7FF;
    const uint32_t m = (hi & 0xFFFFFu) | 0x100000u;
    // (m, lo) >> (sh - 1), sh = 52 - (E - 1023 + 8 ns - 1 - c) >= 53 - (8 ns - 1)
    const uint32_t t = (uint32_t)(1075 - 8 * ns + c - E);  // sh - 1; a zero under kAbsent wraps to the last case
    uint32_t v = t < 32 ? __funnelshift_r(lo, m, t) : (t < 64 ? m >> (t - 32) : 0u);
    if (E == 0) v = 0u;
    const uint32_t rest = t < 32 ? lo << (32 - t) : (lo | (t > 32 && t < 64 ? m << (64 - t) : 0u));  // below the half
    uint32_t u = (v >> 1) + (v & (rest ? 1u : (v >> 1)) & 1u);
    const uint32_t sign = hi & 0x80000000u;
#pragma unroll
    for (int i = ns - 1; i > 0; --i) {
      const uint32_t q = (u + 128u) >> 8;
      // a digit as float without the conversion pipe
      s[i] = __float_as_uint(__int_as_float(0x4B400000 + (int)(u - (q << 8))) - 12582912.0f) ^ sign;
      u = q;
    }
    s[0] = __float_as_uint(__int_as_float(0x4B400000 + (int)u) - 12582912.0f) ^ sign;
  }
}

// One operand's block of a k-block in the registers of the block's threads.
// kfast (k contiguous): a warp per row, 32 lanes x 4 bytes of the packed row;
// else a thread per (row, 16-byte chunk of k), lanes along the rows.
template <int MODE, int ROWS>
struct Frag {
  using Tr = FusedTraits<MODE>;
  static constexpr int PER = Tr::tf32 ? 1 : 2;                // elements in 4 bytes
  static constexpr int G = 4 * PER;                           // elements of a chunk
  static constexpr int UNITS = (ROWS * 8 + FT - 1) / FT;      // chunks of a thread
  static constexpr int RPW = (ROWS + FW - 1) / FW;            // rows of a warp
  static_assert(RPW * PER <= UNITS * G, "fragment");
  double x[UNITS * G];

  template <typename OffFn>
  __device__ __forceinline__ void load(const double* base, OffFn off, int rows, int k, int k1, long long kstr,
                                       bool kfast) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (kfast) {
      const int kk = k + PER * lane;
#pragma unroll
      for (int i = 0; i < RPW; ++i) {
        const int r = warp + i * FW;
        const double* p = base + (r < rows ? off(r) : 0);
#pragma unroll
        for (int e = 0; e < PER; ++e) x[i * PER + e] = (r < rows && kk + e < k1) ? p[(long long)(kk + e) * kstr] : 0.0;
      }
    } else {
#pragma unroll
      for (int i = 0; i < UNITS; ++i) {
        const int u = tid + i * FT, r = u % ROWS, kc = k + (u / ROWS) * G;
        const bool live = u < ROWS * 8 && r < rows;
        const double* p = base + (live ? off(r) : 0);
#pragma unroll
        for (int e = 0; e < G; ++e) x[i * G + e] = (live && kc + e < k1) ? p[(long long)(kc + e) * kstr] : 0.0;
      }
    }
  }
  // Slice t goes to dst + t ROWS 128: row pitch 128 bytes, the 16-byte chunk
  // index xored with row mod 8.  sh: the shifts of this k-block (times sgn).
  __device__ __forceinline__ void store(uint8_t* dst, int kleft, bool kfast, const int* ex, const int* sh, int sgn) const {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (kfast) {
      const uint32_t at = (uint32_t)(lane >> 2), in = (uint32_t)(lane & 3) * 4;
      int s[PER];
#pragma unroll
      for (int e = 0; e < PER; ++e) s[e] = (Tr::sliced && PER * lane + e < kleft) ? sgn * sh[PER * lane + e] : 0;
#pragma unroll
      for (int i = 0; i < RPW; ++i) {
        const int r = warp + i * FW;
        if (ROWS % FW != 0 && r >= ROWS) break;
        uint32_t v[PER][Tr::ns];
#pragma unroll
        for (int e = 0; e < PER; ++e) cut<MODE>(x[i * PER + e], Tr::sliced ? ex[r] - s[e] : 0, v[e]);
        uint8_t* o = dst + (uint32_t)r * 128u + ((at ^ (uint32_t)(r & 7)) << 4) + in;
#pragma unroll
        for (int t = 0; t < Tr::ns; ++t)
          *reinterpret_cast<uint32_t*>(o + t * ROWS * 128) = Tr::tf32 ? v[0][t] : __byte_perm(v[0][t], v[PER - 1][t], 0x7632);
      }
    } else {
#pragma unroll
      for (int i = 0; i < UNITS; ++i) {
        const int u = tid + i * FT, r = u % ROWS, g = u / ROWS;
        if ((ROWS * 8) % FT != 0 && u >= ROWS * 8) break;
        const int er = Tr::sliced ? ex[r] : 0;
        uint32_t w[Tr::ns][4];
#pragma unroll
        for (int e = 0; e < G; e += PER) {
          uint32_t v[PER][Tr::ns];
#pragma unroll
          for (int b = 0; b < PER; ++b)
            cut<MODE>(x[i * G + e + b], (Tr::sliced && g * G + e + b < kleft) ? er - sgn * sh[g * G + e + b] : er, v[b]);
#pragma unroll
          for (int t = 0; t < Tr::ns; ++t)
            w[t][e / PER] = Tr::tf32 ? v[0][t] : __byte_perm(v[0][t], v[PER - 1][t], 0x7632);
        }
        uint8_t* o = dst + (uint32_t)r * 128u + ((uint32_t)(g ^ (r & 7)) << 4);
#pragma unroll
        for (int t = 0; t < Tr::ns; ++t)
          *reinterpret_cast<uint4*>(o + t * ROWS * 128) = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
      }
    }
  }
};

// Exponent fields of an operand over k in [k0, k1) into tab[(k - k0) pitch + row].
template <int ROWS, typename OffFn>
__device__ __forceinline__ void read_fields(const double* base, OffFn off, int rows, int k0, int k1, long long kstr,
                                            bool kfast, uint16_t* tab, int pitch) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int U = 16;  // loads in flight
  const int nk = k1 - k0;
  if (kfast) {
    const int kc = (nk + 31) / 32, total = rows * kc;  // (row, chunk of 32 k)
    for (int p0 = warp; p0 < total; p0 += U * FW) {
      double x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int p = p0 + u * FW, r = p / kc, k = (p - r * kc) * 32 + lane;
        x[u] = (p < total && k < nk) ? base[off(r) + (long long)(k0 + k) * kstr] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int p = p0 + u * FW, r = p / kc, k = (p - r * kc) * 32 + lane;
        if (p < total && k < nk) tab[k * pitch + r] = (uint16_t)exp_field(x[u]);
      }
    }
  } else {
    const int total = nk * ROWS;
    for (int x0 = tid; x0 < total; x0 += U * FT) {
      double x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = x0 + u * FT, k = q / ROWS, r = q - k * ROWS;
        x[u] = (q < total && r < rows) ? base[off(r) + (long long)(k0 + k) * kstr] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = x0 + u * FT, k = q / ROWS, r = q - k * ROWS;
        if (q < total && r < rows) tab[k * pitch + r] = (uint16_t)exp_field(x[u]);
      }
    }
  }
}

// Largest shifted field of each row over the table into out[rows] (zeroed before).
template <int ROWS>
__device__ __forceinline__ void row_fields(const uint16_t* tab, int pitch, int rows, int nk, const int* sh, int sgn,
                                           int* out) {
  constexpr int PARTS = FT / ROWS > 4 ? 4 : FT / ROWS;
  const int r = threadIdx.x % ROWS, part = threadIdx.x / ROWS;
  if (part >= PARTS || r >= rows) return;
  int m = 0;
#pragma unroll 8
  for (int k = part; k < nk; k += PARTS) m = max(m, shifted(tab[k * pitch + r], sgn * sh[k]));
  if (m) atomicMax(out + r, m);
}

template <int MODE, int BN, int STAGES>
__global__ void __launch_bounds__(FT, 1) tc_fused_kernel(const FusedArgs g) {
  using Tr = FusedTraits<MODE>;
  constexpr int A_BYTES = BM * 128, B_BYTES = BN * 128;
  constexpr int STAGE_BYTES = Tr::ns * (A_BYTES + B_BYTES);
  constexpr uint32_t IDESC = make_idesc(Tr::tf32 ? 2u : 1u, (uint32_t)BN);
  constexpr int ACC = Tr::sliced ? Tr::ngroups : 2;  // accumulators: slice weights, or pieces
  constexpr int TMEM_COLS = tmem_cols_for(ACC * BN);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t empty[STAGES], done;
  __shared__ uint32_t tmem_slot;
  __shared__ long long aoff[BM], coff[BM];
  __shared__ int ea[BM], eb[BN], ksh[Tr::sliced ? FK_MAX : 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bi = blockIdx.z / g.splitk, sk = blockIdx.z - bi * g.splitk;
  const int n0 = blockIdx.x * BN;
  const long long row0 = (long long)blockIdx.y * BM;
  const int rows = (int)min((long long)BM, g.R - row0), cols = min(BN, g.N - n0);
  const int kb0 = sk * g.kb_per_split, kb1 = min(g.kblocks, kb0 + g.kb_per_split);
  const int k0 = kb0 * Tr::kb, k1 = min(g.K, kb1 * Tr::kb);

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) mbar_init(&empty[s], 1);
    mbar_init(&done, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&tmem_slot, TMEM_COLS);
    tmem_relinquish();
    tc_fence_before();
  }
  for (int r = tid; r < BM; r += FT) {
    const long long x = row0 + r, o = r < rows ? x / g.M : 0, m = r < rows ? x - o * g.M : 0;
    aoff[r] = o * g.A.so + m * g.A.rs;
    coff[r] = o * g.C.so + m * g.C.rs;
  }
  if constexpr (Tr::sliced) {
    for (int x = tid; x < BM; x += FT) ea[x] = 0;
    for (int x = tid; x < BN; x += FT) eb[x] = 0;
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const double* Ap = g.A.p + (long long)bi * g.A.si;
  const double* Bp = g.B.p + (long long)bi * g.B.si + (long long)n0 * g.B.cs;
  const bool a_kfast = g.A.cs == 1, b_kfast = g.B.rs == 1 && g.B.cs != 1;
  const long long bcs = g.B.cs;
  auto arow = [&](int r) { return aoff[r]; };
  auto brow = [&](int n) { return (long long)n * bcs; };

  if constexpr (Tr::sliced) {
    const int nk = k1 - k0;
    constexpr int PA = BM + 2, PB = BN + 2;  // odd word pitches
    uint16_t* ta = reinterpret_cast<uint16_t*>(smem);
    uint16_t* tb = ta + (size_t)nk * PA;
    read_fields<BN>(Bp, brow, cols, k0, k1, g.B.rs, b_kfast, tb, PB);
    read_fields<BM>(Ap, arow, rows, k0, k1, g.A.cs, a_kfast, ta, PA);
    __syncthreads();
    // K index shifts: half the difference of the two operands' largest
    // exponents at k, so that both carry the square root of the terms' sizes
    // and the terms far below the largest one keep the same relative
    // accuracy in either operand.  A k that is zero in one operand adds
    // nothing: it leaves the other one too, whose scales it would otherwise
    // set (1e9 there against balanced terms around 1 left no correct digit)
    for (int k = tid; k < nk; k += FT) {
      int ma = 0, mb = 0;
#pragma unroll 8
      for (int n = 0; n < cols; ++n) mb = max(mb, (int)tb[k * PB + n]);
#pragma unroll 8
      for (int r = 0; r < rows; ++r) ma = max(ma, (int)ta[k * PA + r]);
      ksh[k] = ma == 0 ? kAbsent : mb == 0 ? -kAbsent : (mb - ma) >> 1;
    }
    __syncthreads();
    row_fields<BM>(ta, PA, rows, nk, ksh, 1, ea);
    row_fields<BN>(tb, PB, cols, nk, ksh, -1, eb);
    __syncthreads();
    for (int x = tid; x < BM; x += FT) ea[x] = field_exponent(ea[x]);
    for (int x = tid; x < BN; x += FT) eb[x] = field_exponent(eb[x]);
    __syncthreads();
  }

  int it = 0;
  uint32_t drained = 0;  // phase of `done`
  bool alive = true;
  bool first_drain = true;
  Frag<MODE, BM> fa;
  Frag<MODE, BN> fb;
  fa.load(Ap, arow, rows, k0, k1, g.A.cs, a_kfast);
  fb.load(Bp, brow, cols, k0, k1, g.B.rs, b_kfast);
  for (int piece = 0; piece < g.pieces && alive; ++piece) {
    for (int kb = kb0; kb < kb1 && alive; ++kb, ++it) {
      const int s = it % STAGES;
      bool ok = it < STAGES || mbar_wait(&empty[s], (uint32_t)((it / STAGES - 1) & 1));
      uint8_t* st = smem + s * STAGE_BYTES;
      const int k = kb * Tr::kb;
      // the block after this one: the next of this piece, or the first of the next piece
      const int np = kb + 1 < kb1 ? piece : piece + 1, nk = kb + 1 < kb1 ? k + Tr::kb : k0;
      const int* sh = Tr::sliced ? ksh + (k - k0) : nullptr;
      fa.store(st, k1 - k, a_kfast, ea, sh, 1);
      if (np < g.pieces) fa.load(Ap + np * g.pa, arow, rows, nk, k1, g.A.cs, a_kfast);
      fb.store(st + Tr::ns * A_BYTES, k1 - k, b_kfast, eb, sh, -1);
      if (np < g.pieces) fb.load(Bp + np * g.pb, brow, cols, nk, k1, g.B.rs, b_kfast);
      fence_async_smem();
      alive = __syncthreads_and(ok ? 1 : 0) != 0;
      if (!alive) break;
      const bool chunk_start = Tr::sliced ? (kb - kb0) % Tr::exact_kb == 0 : kb == kb0;
      const bool chunk_end = kb + 1 == kb1 || (Tr::sliced && (kb + 1 - kb0) % Tr::exact_kb == 0);
      if (tid == 0) {
        tc_fence_after();
        const uint32_t sa = smem_u32(st), sb = sa + Tr::ns * A_BYTES;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {  // 4 x 32 bytes of K per 128-byte row
          const uint32_t o = kk * 32;
          const bool fresh0 = chunk_start && kk == 0;
          if constexpr (Tr::sliced) {
#pragma unroll
            for (int w = 0; w < Tr::ngroups; ++w) {
              bool fresh = fresh0;
#pragma unroll
              for (int ia = 0; ia < Tr::ns; ++ia) {
                const int jb = w - ia;
                if (jb < 0 || jb >= Tr::ns) continue;
                mma_issue<false>(tmem + (uint32_t)(w * BN), desc_sw128(sa + ia * A_BYTES + o),
                                 desc_sw128(sb + jb * B_BYTES + o), IDESC, fresh ? 0u : 1u);
                fresh = false;
              }
            }
          } else {
            const uint32_t d = tmem + (uint32_t)(piece * BN);
            mma_issue<true>(d, desc_sw128(sa + o), desc_sw128(sb + o), IDESC, fresh0 ? 0u : 1u);
            mma_issue<true>(d, desc_sw128(sa + o), desc_sw128(sb + B_BYTES + o), IDESC, 1u);
            mma_issue<true>(d, desc_sw128(sa + A_BYTES + o), desc_sw128(sb + o), IDESC, 1u);
          }
        }
        mma_commit(&empty[s]);
        if (chunk_end && (Tr::sliced || piece + 1 == g.pieces)) mma_commit(&done);
      }
      __syncwarp();
      if (!chunk_end || (!Tr::sliced && piece + 1 < g.pieces)) continue;
      // ---- drain the accumulators
      ok = mbar_wait(&done, drained);
      drained ^= 1u;
      alive = __syncthreads_and(ok ? 1 : 0) != 0;
      if (!alive) break;
      tc_fence_after();
      const int q = warp & 3;
      const int r = 32 * q + lane;
      const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16);
      const bool row_live = r < rows;
      const int erow = (Tr::sliced) ? ea[r] : 0;
      double* W = g.ws ? g.ws + (((long long)bi * g.splitk + sk) * g.R + row0) * g.N + n0 : nullptr;
      double* Cp = g.C.p + (long long)bi * g.C.si + (long long)n0 * g.C.cs;
      const bool plain = W || (first_drain && g.beta == 0.0 && (g.alpha == 1.0 || g.alpha == -1.0));
      const unsigned long long flip = (!W && g.alpha == -1.0) ? (1ull << 63) : 0ull;
      const double keep = first_drain ? g.beta : 1.0;
      // lanes along the columns through a staging tile unless the rows of C are contiguous; the stages are
      // free (every MMA that read them has completed)
      const bool along_rows = !W && g.C.rs < g.C.cs;
      unsigned long long* stg = reinterpret_cast<unsigned long long*>(smem) + warp * (32 * 9);
      auto put = [&](int row, int col, unsigned long long bits) {
        double* c = W ? W + (long long)row * g.N + col : Cp + coff[row] + (long long)col * g.C.cs;
        if (plain) *reinterpret_cast<unsigned long long*>(c) = bits ^ flip;
        else *c = g.alpha * __longlong_as_double((long long)bits) + (keep == 0.0 ? 0.0 : keep * (*c));
      };
#pragma unroll 1
      for (int c0 = 8 * (warp >> 2); c0 < cols; c0 += 8 * (FW / 4)) {
        uint32_t v[ACC][8];
#pragma unroll
        for (int w = 0; w < ACC; ++w)
          if (Tr::sliced || w < g.pieces) tmem_ld8(lane_base + (uint32_t)(w * BN + c0), v[w]);
        tmem_ld_wait();
        unsigned long long bits[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if constexpr (Tr::sliced) {
            long long S = 0;
#pragma unroll
            for (int w = 0; w < Tr::ngroups; ++w)
              S += (long long)__float2int_rn(__uint_as_float(v[w][j])) << (8 * (Tr::ngroups - 1 - w));
            bits[j] = int_to_double_bits(S, erow + eb[c0 + j] - 14 - 8 * (Tr::ngroups - 1));
          } else {
            bits[j] = float_to_double_bits(v[0][j]);
            if (g.pieces == 2)  // the pieces meet in FP64
              bits[j] = (unsigned long long)__double_as_longlong(
                  __longlong_as_double((long long)bits[j]) + __longlong_as_double((long long)float_to_double_bits(v[1][j])));
          }
        }
        if (along_rows) {
          if (row_live)
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (c0 + j < cols) put(r, c0 + j, bits[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) stg[lane * 9 + j] = bits[j];
          __syncwarp();
          const int j = lane & 7;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int lr = 4 * i + (lane >> 3);
            if (32 * q + lr < rows && c0 + j < cols) put(32 * q + lr, c0 + j, stg[lr * 9 + j]);
          }
          __syncwarp();
        }
      }
      first_drain = false;
      tc_fence_before();
      __syncthreads();  // TMEM and the staging tiles are free again
      tc_fence_after();
    }
  }
  if (!alive && tid == 0) {
    atomicOr(g.err, 32);
    mma_commit(&done);  // a bounded wait for the MMAs still in flight
    mbar_wait(&done, drained);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

// K of one exact-slice product: its exponent fields have to fit the stage
// buffers (asserted below); longer ones go to the packed GEMM.
constexpr int fused_max_k(int mode) { return mode == TC_BF16X10 ? 448 : 352; }

template <int MODE, int BN>
void launch_fused(cudaStream_t st, dim3 grid, const FusedArgs& g) {
  using Tr = FusedTraits<MODE>;
  constexpr int STAGE = Tr::ns * (BM + BN) * 128;
  // static shared memory: row offsets, exponents, shifts, barriers
  constexpr int FIXED = 2 * BM * 8 + BM * 4 + BN * 4 + (Tr::sliced ? FK_MAX * 4 : 4) + 256;
  constexpr int FIT = (232448 - FIXED - 1024) / STAGE;
  constexpr int STAGES = FIT > 3 ? 3 : FIT;
  static_assert(STAGES >= 1, "shared memory budget");
  static_assert((Tr::sliced ? Tr::ngroups : 2) * BN <= 512, "TMEM budget");
  // the staging tiles of the epilogue: 32 x 9 words a warp
  static_assert(STAGES * STAGE >= FW * 32 * 9 * 8, "staging");
  // the exponent fields of both operands in the stage buffers
  static_assert(!Tr::sliced || STAGES * STAGE >= fused_max_k(MODE) * (BM + BN + 4) * 2, "field tables");
  constexpr int SMEM = STAGES * STAGE + 1024;
  static const bool attr = [] {
    cudaFuncSetAttribute(tc_fused_kernel<MODE, BN, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    return true;
  }();
  (void)attr;
  tc_fused_kernel<MODE, BN, STAGES><<<grid, FT, SMEM, st>>>(g);
}

template <int MODE>
void launch_fused_bn(cudaStream_t st, int bn, dim3 grid, const FusedArgs& g) {
  switch (bn) {
    case 32: launch_fused<MODE, 32>(st, grid, g); return;
    case 48: launch_fused<MODE, 48>(st, grid, g); return;
    case 64: launch_fused<MODE, 64>(st, grid, g); return;
    case 80: launch_fused<MODE, 80>(st, grid, g); return;
    default: break;
  }
  if constexpr (MODE != TC_BF16X10) {
    switch (bn) {
      case 96: launch_fused<MODE, 96>(st, grid, g); return;
      case 112: launch_fused<MODE, 112>(st, grid, g); return;
      case 128: launch_fused<MODE, 128>(st, grid, g); return;
      default: launch_fused<MODE, 144>(st, grid, g); return;
    }
  }
}

int round16(int n) { return (n + 15) / 16 * 16; }

// Column tiles of a product: as few as the widest tile allows (two stages have
// to fit), more (down to 48 columns) while the grid would leave half of the
// SMs idle.
void column_tiles(int mode, int N, long long others, int* bn, int* tiles) {
  const int widest = mode == TC_BF16X10 ? 80 : 144;
  int t = (N + widest - 1) / widest;
  while (others * t < 76 && t < 4 && round16((N + t) / (t + 1)) >= 48) ++t;
  *bn = std::max(32, round16((N + t - 1) / t));
  *tiles = (N + *bn - 1) / *bn;
}

}  // namespace

bool gemm_fused(cudaStream_t st, int mode, int M, int N, int K, int outer, int inner, double alpha, MatView A, MatView B,
                double beta, OutView C, const SumPieces& P, double* ws, size_t ws_elems, int* err) {
  if (mode != TC_TF32X3 && mode != TC_BF16X6 && mode != TC_BF16X10) return false;
  if (M <= 0 || N <= 0 || K <= 0 || outer <= 0 || inner <= 0) return false;
  const bool sliced = mode != TC_TF32X3;
  if (P.n > (sliced ? 1 : 2)) return false;
  // The tall side: the operand that may vary over the outer index gives the
  // rows (all outer entries flat), the other one the columns.
  const bool keep_ok = outer == 1 || B.so == 0, swap_ok = outer == 1 || A.so == 0;
  // Wide column operands are converted once per row tile, and the rows once per
  // column tile.  Alone and from a cold L2, row-major, K = 136 (this / packed, us):
  // 17408 rows, BF16X6 136 columns 71 / 69, 208 102 / 89, 272 124 / 99, 400 178 /
  // 135; TF32X3 30 / 36, 47 / 43, 56 / 54, 80 / 83; 272 rows, BF16X6 37 / 47, 42 /
  // 35, 46 / 36, 43 / 36.  In whole steps the packed product's three to five
  // launches weigh more: with the line at 144 columns the step takes 40 sites chi
  // 128 38.5 -> 38.1 ms, uneven grid chi 77 14.3 -> 14.6, batch of 12 178 -> 180,
  // a drawn one 13.3 -> 13.7, and the first step up to 70 ms more (the packed
  // product's timed tile choices).  So the line takes 2 chi columns up to the
  // bond 144 that the other limits (float QR in registers, field tables) have.
  constexpr int kMaxCols = 288;
  auto cost = [&](int m, int n) {  // elements converted
    const long long rt = ((long long)m * outer + BM - 1) / BM;
    return n > kMaxCols ? 1e300 : (double)rt * ((n + 143) / 144) * (BM + std::min(n, 144));
  };
  const double ck = keep_ok ? cost(M, N) : 1e300, cs = swap_ok ? cost(N, M) : 1e300;
  if (std::min(ck, cs) >= 1e300) return false;
  const bool swap = cs < ck;
  FusedArgs g;
  g.A = A;
  g.B = B;
  g.C = C;
  g.M = M;
  g.N = N;
  g.pa = P.a;
  g.pb = P.b0;
  if (swap) {  // C^T = B^T A^T
    g.A.p = B.p;
    g.A.rs = B.cs;
    g.A.cs = B.rs;
    g.A.so = B.so;
    g.A.si = B.si;
    g.B.p = A.p;
    g.B.rs = A.cs;
    g.B.cs = A.rs;
    g.B.so = A.so;
    g.B.si = A.si;
    g.C.rs = C.cs;
    g.C.cs = C.rs;
    g.M = N;
    g.N = M;
    g.pa = P.b0;
    g.pb = P.a;
  }
  g.R = (long long)g.M * outer;
  g.K = K;
  g.pieces = P.n;
  const int kb = sliced ? 64 : 32;
  g.kblocks = (K + kb - 1) / kb;
  g.splitk = 1;
  g.kb_per_split = g.kblocks;
  const long long rt = (g.R + BM - 1) / BM;
  // a long K with few tiles (the range product) is split over the CTAs that are left instead of the columns
  const bool long_k = !sliced && P.n == 1 && outer == 1 && g.kblocks >= 8 && ws != nullptr;
  int bn, tiles;
  column_tiles(mode, g.N, long_k ? 1 << 30 : rt * inner, &bn, &tiles);
  if (rt > 65535 || (sliced && K > fused_max_k(mode))) return false;
  const long long ctas = rt * tiles * inner;
  if (long_k && ctas < 76) {
    int s = (int)std::min<long long>(g.kblocks / 2, 152 / ctas);
    while (s > 1 && (size_t)s * inner * (size_t)g.R * g.N > ws_elems) s /= 2;
    if (s > 1) {
      g.kb_per_split = (g.kblocks + s - 1) / s;
      g.splitk = (g.kblocks + g.kb_per_split - 1) / g.kb_per_split;
    }
  }
  if ((long long)inner * g.splitk > 65535) return false;
  g.alpha = alpha;
  g.beta = beta;
  g.ws = g.splitk > 1 ? ws : nullptr;
  g.err = err;
  const dim3 grid((unsigned)tiles, (unsigned)rt, (unsigned)(inner * g.splitk));
  count_launches(g.splitk > 1 ? 2 : 1);
  switch (mode) {
    case TC_TF32X3: launch_fused_bn<TC_TF32X3>(st, bn, grid, g); break;
    case TC_BF16X6: launch_fused_bn<TC_BF16X6>(st, bn, grid, g); break;
    default: launch_fused_bn<TC_BF16X10>(st, bn, grid, g); break;
  }
  if (g.splitk > 1) splitk_reduce(st, (int)g.R, g.N, inner, g.splitk, inner, alpha, ws, beta, g.C);
  return true;
}

}  // namespace qtt
