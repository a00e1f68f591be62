// Contractions with an operator (MPO) bond: batched GEMMs whose M is at most
// 32 and K at most 64 -- the MPO core applied to a site tensor in the sketch
// and zip-up passes (operator bond w <= ~26 for the stencil operators), the
// mixing term's products at small chi, and the first and last sites' products
// of every term.  They run on the CUDA cores without packing, in double for
// the FP64 form and in float (round to nearest, unbiased) for the
// reduced-precision forms; inputs and outputs are FP64.
//
// What bounds them: in FP64 the pipe (a warp FMA costs a scheduler 64 clocks
// here), in float the latency of the strided loads of B.  So the work is cut
// to fill the 608 schedulers: the columns of every outer batch entry are one
// flat range (A does not depend on the outer index), 32 columns a block; the
// rows come in groups of MG, one group a block; and the contraction -- K
// times up to four pieces, the (s, s') pairs of an operator core -- is split
// over the block's four warps, whose partial sums meet in shared memory and
// are added in FP64.  A warp keeps eight loads of B in flight; the rows of A
// sit in shared memory k-major, so a row group is read as vectors.
// One thread per column with all of M and K on it (the layout before) left a
// 32 x 40 x 32 product with 32 batch entries on 40 warps at 78 us in FP64,
// and the four pieces took four launches that re-read C.  Step before and
// after, the other kernels as they were then: 20 sites chi 32 FP64 19.1 -> 15.3 ms, 30 sites chi 64 FP64 46.6 ->
// 44.5 and FP32 20.7 -> 19.5, 40 sites chi 128 BF16X10 59.7 -> 57.1.
#include <algorithm>
#include <cstdint>

#include "kernels.cuh"

namespace qtt {

namespace {
constexpr int SG_THREADS = 128;
constexpr int SG_WARPS = SG_THREADS / 32;
constexpr int SG_MAXM = 32, SG_MAXK = 64;
constexpr int SG_UNROLL = 8;

// double -> float, round to nearest even, by bits (the FP64 pipe issues two
// operations per clock per SM); below the float normal range -> 0.
__device__ __forceinline__ float d2f_bits(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const uint32_t sign = (uint32_t)(u >> 32) & 0x80000000u;
  const int e = (int)((u >> 52) & 0x7FFull);
  const unsigned long long m = u & 0xFFFFFFFFFFFFFull;
  if (e == 0x7FF) return __uint_as_float(sign | 0x7F800000u | (m ? 0x400000u : 0u));
  const int fe = e - 1023 + 127;
  if (fe <= 0) return __uint_as_float(sign);
  if (fe >= 255) return __uint_as_float(sign | 0x7F800000u);
  const unsigned long long rem = m & 0x1FFFFFFFull;
  uint32_t r = ((uint32_t)fe << 23) | (uint32_t)(m >> 29);
  if (rem > 0x10000000ull || (rem == 0x10000000ull && (r & 1u))) r += 1u;
  return __uint_as_float(sign | r);
}

// float -> double, exact, by bits (denormals through the hardware conversion).
__device__ __forceinline__ double f2d_bits(float f) {
  const uint32_t b = __float_as_uint(f);
  const uint32_t e = (b >> 23) & 0xFFu;
  const unsigned long long sign = (unsigned long long)(b >> 31) << 63;
  if (e == 0u) return (b & 0x7FFFFFu) ? (double)f : __longlong_as_double((long long)sign);
  const unsigned long long de = (e == 0xFFu) ? 0x7FFull : (unsigned long long)(e + 896u);
  return __longlong_as_double((long long)(sign | (de << 52) | ((unsigned long long)(b & 0x7FFFFFu) << 29)));
}

template <typename T>
__device__ __forceinline__ T to_t(double x) {
  if constexpr (sizeof(T) == 4)
    return d2f_bits(x);
  else
    return x;
}
template <typename T>
__device__ __forceinline__ double to_d(T x) {
  if constexpr (sizeof(T) == 4)
    return f2d_bits(x);
  else
    return x;
}


// C[(outer, inner)] (M x N) = alpha sum_p A_p[inner] B_p[(outer, inner)] + beta C
// over the pieces p.  Block (x, y, z): flat columns 32 x .., rows MG y ..,
// inner index z (flat) or batch index z.
template <typename T, int MG>
__global__ void __launch_bounds__(SG_THREADS) small_gemm_kernel(int M, int N, int K, int inner, long long ncols,
                                                                int flat, double alpha, MatView A, MatView B,
                                                                double beta, OutView C, SumPieces P) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ __align__(16) unsigned char sg_smem[];
  T* As = reinterpret_cast<T*>(sg_smem);  // [pieces * K][MG]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int slots = P.n * K;
  const int bo0 = flat ? 0 : (int)blockIdx.z / inner;
  const int bi = flat ? (int)blockIdx.z : (int)blockIdx.z - bo0 * inner;
  const int m0 = blockIdx.y * MG;
  const double* Ab = A.p + bo0 * A.so + bi * A.si;
  for (int x = tid; x < slots * MG; x += SG_THREADS) {
    const int m = x % MG, s = x / MG, p = s / K, k = s - p * K;
    As[x] = m0 + m < M ? to_t<T>(Ab[p * P.a + (long long)(m0 + m) * A.rs + (long long)k * A.cs]) : (T)0;
  }
  const long long c = (long long)blockIdx.x * 32 + lane;
  const bool live = c < ncols;
  const int bo = flat ? (int)((live ? c : 0) / N) : bo0;
  const int n = (int)((live ? c : 0) - (flat ? (long long)bo * N : 0));
  const double* Bb = B.p + bo * B.so + bi * B.si + (long long)n * B.cs;
  // this warp's slots: whole pieces when there are at least as many as warps, else a part of one piece
  const int share = (slots + SG_WARPS - 1) / SG_WARPS;
  const int s0 = min(slots, warp * share), s1 = min(slots, s0 + share);
  __syncthreads();
  T acc[MG];
#pragma unroll
  for (int m = 0; m < MG; ++m) acc[m] = (T)0;
  for (int s = s0; s < s1; s += SG_UNROLL) {
    double b[SG_UNROLL];  // all loads in flight before the first use
#pragma unroll
    for (int u = 0; u < SG_UNROLL; ++u) {
      const int q = s + u, p = q / K;
      b[u] = (live && q < s1) ? Bb[(p & 1) * P.b0 + (p >> 1) * P.b1 + (long long)(q - p * K) * B.rs] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < SG_UNROLL; ++u) {
      if (s + u >= s1) break;  // warp-uniform
      const T bk = to_t<T>(b[u]);
      const T* a = As + (size_t)(s + u) * MG;
#pragma unroll
      for (int m = 0; m < MG; ++m) acc[m] += a[m] * bk;
    }
  }
  __syncthreads();
  T* red = As;  // [warp][MG][32], the operator rows are no longer needed
#pragma unroll
  for (int m = 0; m < MG; ++m) red[((size_t)warp * MG + m) * 32 + lane] = acc[m];
  __syncthreads();
  if (!live) return;
  double* Cb = C.p + bo * C.so + bi * C.si + (long long)n * C.cs;
  const bool plain = (alpha == 1.0 && beta == 0.0);
  for (int m = warp; m < MG && m0 + m < M; m += SG_WARPS) {
    double v = to_d<T>(red[(size_t)m * 32 + lane]);
#pragma unroll
    for (int w = 1; w < SG_WARPS; ++w) v += to_d<T>(red[((size_t)w * MG + m) * 32 + lane]);
    double* cp = Cb + (long long)(m0 + m) * C.rs;
    *cp = plain ? v : alpha * v + (beta == 0.0 ? 0.0 : beta * (*cp));
  }
}

template <typename T, int MG>
void launch_small(cudaStream_t st, int M, int N, int K, int outer, int inner, double alpha, MatView A, MatView B,
                  double beta, OutView C, const SumPieces& P) {
  const int flat = (A.so == 0 || outer == 1) ? 1 : 0;
  const long long ncols = flat ? (long long)outer * N : N;
  const dim3 grid((unsigned)((ncols + 31) / 32), (unsigned)((M + MG - 1) / MG), (unsigned)(flat ? inner : outer * inner));
  const size_t smem = (size_t)std::max(P.n * K, 32 * SG_WARPS) * MG * sizeof(T);
  launch_pdl(small_gemm_kernel<T, MG>, grid, dim3(SG_THREADS), smem, st, M, N, K, inner, ncols, flat, alpha, A, B, beta,
             C, P);
}
}  // namespace

bool small_gemm_fits(int M, int N, int K, int outer, int inner) {
  return M >= 1 && M <= SG_MAXM && K >= 1 && K <= SG_MAXK && N >= 1 && (long long)outer * inner <= 65535;
}

void small_gemm_sum(cudaStream_t st, bool fp32, int M, int N, int K, int outer, int inner, double alpha, MatView A,
                    MatView B, double beta, OutView C, const SumPieces& P) {
  count_launches(1);
  // Rows per block.  FP64: a block's time is its share of the contraction
  // times MG warp FMAs, so rows are grouped evenly (26 rows as 4 x 7, not 3 x 8
  // + 2) and by as few as keep every SM busy with its shared loads of B still
  // worth it.  Float: the loads bound it, so as many rows per load of B as
  // leave about two blocks per SM.
  const bool flat = A.so == 0 || outer == 1;
  const long long cg = flat ? ((long long)outer * N + 31) / 32 * inner : (long long)((N + 31) / 32) * outer * inner;
  if (fp32) {
    int mg = M > 16 ? 32 : M > 8 ? 16 : 8;
    while (mg > 8 && cg * ((M + mg - 1) / mg) < 304) mg /= 2;
    switch (mg) {
      case 8: launch_small<float, 8>(st, M, N, K, outer, inner, alpha, A, B, beta, C, P); break;
      case 16: launch_small<float, 16>(st, M, N, K, outer, inner, alpha, A, B, beta, C, P); break;
      default: launch_small<float, 32>(st, M, N, K, outer, inner, alpha, A, B, beta, C, P); break;
    }
    return;
  }
  int best = 8;
  double tbest = 1e300;
  for (int mg = 8; mg >= 1; --mg) {
    const long long blocks = cg * ((M + mg - 1) / mg);
    // clocks: warp FMAs of the blocks one SM takes, 64 each, plus the block's own latency
    const double t = (double)((blocks + 151) / 152) * (((P.n * K + 3) / 4) * mg * 64.0 + 600.0);
    if (t < tbest) {
      tbest = t;
      best = mg;
    }
  }
#define QTT_SG(MG_) \
  case MG_: launch_small<double, MG_>(st, M, N, K, outer, inner, alpha, A, B, beta, C, P); break;
  switch (best) {
    QTT_SG(1) QTT_SG(2) QTT_SG(3) QTT_SG(4) QTT_SG(5) QTT_SG(6) QTT_SG(7) QTT_SG(8)
  }
#undef QTT_SG
}

void small_gemm(cudaStream_t st, bool fp32, int M, int N, int K, int outer, int inner, double alpha, MatView A,
                MatView B, double beta, OutView C) {
  small_gemm_sum(st, fp32, M, N, K, outer, inner, alpha, A, B, beta, C, SumPieces{});
}

}  // namespace qtt
