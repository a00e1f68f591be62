// FP64 strided batched GEMM (CUDA cores, DFMA).  Used by the plain FP64
// path for every core contraction, and by all paths for the small FP64 Gram
// matrices of the SVD truncation sweep.
//
// FP64 issues at two FMAs per clock per SM: a warp FMA holds its scheduler for
// 64 clocks, with one lane active as with 32, while loads, shared-memory
// reads and address arithmetic are almost free beside it.  So the kernel is
// shaped by two things only: no masked FMAs, and equal numbers of FMAs on the
// 608 schedulers.  A block of 8 warps computes TM x 8 RN outputs: a warp holds
// 4 rows x 8 RN columns (lane: one row, RN columns 8 apart), TM / 4 warps cover
// the rows and the K range is dealt over the 32 / TM groups of warps, whose
// partial sums meet in shared memory.  Column counts of the bonds used
// (40, 72, 128, 136: 5, 9, 16 = 8 + 8, 17 = 9 + 8 groups of 8) fit RN <= 9 with
// little or no waste, where a 64 x 64 tile masks 38 to 47% of its FMAs at 40
// and 72 columns; TM = 4, 8 and 16 spread the bond-sized products (136 x 136)
// over all SMs in one launch, where 16 x 16 tiles gave 81 blocks and a K split
// over the grid needs a reduction launch.  That one remains for products with
// few outputs and a long K (the range product 272 x 136 x 16384).  Before and
// after, the other kernels as they were then: step of 20 sites chi 32 15.3 -> 10.0 ms, of 30 sites chi 64 44.5 ->
// 35.7; untruncated step of 10 sites 1.31 -> 0.40; truncation backward of 40
// sites chi 128 13.6 -> 11.5; 40 sites chi 128 BF16X10 (its Grams) 57.1 -> 55.1.
//
// The operands are read through general (row, column, batch) strides so that
// every reshape / transpose of the contraction is a view, not a copy: chunks
// of 32 k are loaded into registers while the chunk before is multiplied,
// along whichever index is contiguous.  Sums are in a fixed order.
#include <algorithm>

#include "kernels.cuh"

namespace qtt {

namespace {
constexpr int NT = 256, KC = 32;

template <int TM, int RN>
__global__ void __launch_bounds__(NT) gemm_f64_kernel(int M, int N, int K, int inner, int splitk, int kchunk,
                                                      double alpha, MatView A, MatView B, double beta, OutView C,
                                                      double* ws) {
  constexpr int TN = 8 * RN, KS = 32 / TM, LA = TM + 1, LB = TN + 1;
  constexpr int NA = (TM * KC + NT - 1) / NT, NB = TN * KC / NT;
  pdl_trigger();
  pdl_wait();
  __shared__ double smem[KC * (LA + LB)];
  double* As = smem;            // [KC][LA]
  double* Bs = smem + KC * LA;  // [KC][LB]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n0 = blockIdx.x * TN, m0 = blockIdx.y * TM;
  const int z = blockIdx.z;
  const int b = z / splitk, sk = z - b * splitk;
  const int bo = b / inner, bi = b - bo * inner;
  const double* Ap = A.p + bo * A.so + bi * A.si;
  const double* Bp = B.p + bo * B.so + bi * B.si;
  const int k0 = sk * kchunk, k1 = min(K, k0 + kchunk);
  const bool a_mfast = (A.rs < 0 ? -A.rs : A.rs) <= (A.cs < 0 ? -A.cs : A.cs);
  const bool b_nfast = (B.cs < 0 ? -B.cs : B.cs) <= (B.rs < 0 ? -B.rs : B.rs);
  const int wm = warp % (TM / 4), ks = warp / (TM / 4);
  const int row = 4 * wm + (lane >> 3), col = lane & 7;
  const bool rows_live = m0 + 4 * wm < M;  // warp-uniform: a warp with no rows adds no FMAs
  double acc[RN], ra[NA], rb[NB];
#pragma unroll
  for (int j = 0; j < RN; ++j) acc[j] = 0.0;

  auto fetch = [&](int kt) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int x = tid + q * NT;
      const int kk = a_mfast ? x / TM : x % KC, mm = a_mfast ? x % TM : x / KC;
      const int gm = m0 + mm, gk = kt + kk;
      ra[q] = (x < TM * KC && gm < M && gk < k1) ? Ap[(long long)gm * A.rs + (long long)gk * A.cs] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int x = tid + q * NT;
      const int kk = b_nfast ? x / TN : x % KC, nn = b_nfast ? x % TN : x / KC;
      const int gn = n0 + nn, gk = kt + kk;
      rb[q] = (gn < N && gk < k1) ? Bp[(long long)gk * B.rs + (long long)gn * B.cs] : 0.0;
    }
  };
  if (k0 < k1) fetch(k0);
  for (int kt = k0; kt < k1; kt += KC) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int x = tid + q * NT;
      const int kk = a_mfast ? x / TM : x % KC, mm = a_mfast ? x % TM : x / KC;
      if (x < TM * KC) As[kk * LA + mm] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int x = tid + q * NT;
      const int kk = b_nfast ? x / TN : x % KC, nn = b_nfast ? x % TN : x / KC;
      Bs[kk * LB + nn] = rb[q];
    }
    __syncthreads();
    if (kt + KC < k1) fetch(kt + KC);  // in flight during the multiplication
    const int kend = min(KC, k1 - kt);
    if (rows_live) {
#pragma unroll 4
      for (int kk = ks; kk < kend; kk += KS) {
        const double a = As[kk * LA + row];
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[j] = fma(a, Bs[kk * LB + col + 8 * j], acc[j]);
      }
    }
    __syncthreads();
  }
  double* W = ws ? ws + ((long long)b * splitk + sk) * (long long)M * N : nullptr;
  double* Cp = C.p + bo * C.so + bi * C.si;
  auto put = [&](int gm, int gn, double v) {
    if (gm >= M || gn >= N) return;
    if (W) {
      W[(long long)gm * N + gn] = v;
    } else {
      double* c = Cp + (long long)gm * C.rs + (long long)gn * C.cs;
      *c = (beta == 0.0) ? alpha * v : alpha * v + beta * (*c);
    }
  };
  if (KS == 1) {
#pragma unroll
    for (int j = 0; j < RN; ++j) put(m0 + row, n0 + col + 8 * j, acc[j]);
  } else {
    // [KS][TM][TN] partial sums: 32 TN doubles, within the operand buffers
#pragma unroll
    for (int j = 0; j < RN; ++j) smem[(ks * TM + row) * TN + col + 8 * j] = acc[j];
    __syncthreads();
    for (int x = tid; x < TM * TN; x += NT) {
      double v = smem[x];
#pragma unroll
      for (int q = 1; q < KS; ++q) v += smem[q * TM * TN + x];
      put(m0 + x / TN, n0 + x % TN, v);
    }
  }
}

__global__ void splitk_reduce_kernel(int M, int N, int inner, int splitk, int batch, double alpha, const double* ws,
                                     double beta, OutView C) {
  pdl_trigger();
  pdl_wait();
  const long long MN = (long long)M * N;
  const long long total = MN * batch;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(e / MN);
    const long long r = e - (long long)b * MN;
    const int gm = (int)(r / N), gn = (int)(r - (long long)gm * N);
    double s = 0.0;
    for (int k = 0; k < splitk; ++k) s += ws[((long long)b * splitk + k) * MN + r];
    const int bo = b / inner, bi = b - bo * inner;
    double* c = C.p + bo * C.so + bi * C.si + (long long)gm * C.rs + (long long)gn * C.cs;
    *c = (beta == 0.0) ? alpha * s : alpha * s + beta * (*c);
  }
}
__global__ void scale_out_kernel(int M, int N, int inner, int batch, double beta, OutView C) {
  pdl_trigger();
  pdl_wait();
  const long long MN = (long long)M * N;
  const long long total = MN * batch;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(e / MN);
    const long long r = e - (long long)b * MN;
    const int gm = (int)(r / N), gn = (int)(r - (long long)gm * N);
    const int bo = b / inner, bi = b - bo * inner;
    double* c = C.p + bo * C.so + bi * C.si + (long long)gm * C.rs + (long long)gn * C.cs;
    *c = (beta == 0.0) ? 0.0 : beta * (*c);
  }
}
// One Newton-Schulz step of an almost-orthonormal Q (m x n, row-major):
// out = Q (3 I - Q^T Q) / 2, in two launches.  FP64 issues at two operations
// per clock per SM, so both are sized to one wave of at most 152 blocks with
// one block per SM:
//   ns_gram_kernel: the upper-triangular 16 x 16 tiles of P = Q^T Q only (P is
//     symmetric), each over a slice of the m rows of Q (split s of S), raw
//     partial sums to P_s, written to the tile and to its mirror image;
//   ns_apply_kernel: out = Q G with G = 1.5 I - 0.5 sum_s P_s read row-wise
//     from the partials, 16 x 17 output tiles
//     (17 columns: 136 = 8 x 17 fills 136 blocks where 16 x 16 tiles would
//     make 153, one more than the SMs).
// Operand strips are staged through shared memory in chunks of 32.
constexpr int NS_T = 16;      // Gram tile, and rows of the apply tile
constexpr int NS_C = 17;      // columns of the apply tile
constexpr int NS_MAX_SPLIT = 8;

__global__ void __launch_bounds__(256) ns_gram_kernel(int m, int n, int nt, int rows_per_split,
                                                      const double* __restrict__ Q, double* __restrict__ P) {
  pdl_trigger();
  pdl_wait();
  __shared__ double A[32][NS_T + 1], B[32][NS_T + 1];
  // upper-triangular tile pair (ti <= tj) from the linear block index
  int ti = 0, rem = blockIdx.x;
  while (rem >= nt - ti) {
    rem -= nt - ti;
    ++ti;
  }
  const int tj = ti + rem;
  const int tx = threadIdx.x & (NS_T - 1), ty = threadIdx.x / NS_T;
  const int i0 = ti * NS_T, j0 = tj * NS_T;
  const int kbeg = blockIdx.y * rows_per_split, kend = min(m, kbeg + rows_per_split);
  double acc = 0.0;
  for (int k0 = kbeg; k0 < kend; k0 += 32) {
    for (int e = threadIdx.x; e < 32 * NS_T; e += blockDim.x) {
      const int kk = e / NS_T, c = e - kk * NS_T, k = k0 + kk;
      A[kk][c] = (k < kend && i0 + c < n) ? Q[(size_t)k * n + i0 + c] : 0.0;
      B[kk][c] = (k < kend && j0 + c < n) ? Q[(size_t)k * n + j0 + c] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < 32; ++kk) acc = fma(A[kk][ty], B[kk][tx], acc);
    __syncthreads();
  }
  const int i = i0 + ty, j = j0 + tx;
  if (i < n && j < n) {
    double* Ps = P + (size_t)blockIdx.y * n * n;
    Ps[(size_t)i * n + j] = acc;
    if (ti != tj) Ps[(size_t)j * n + i] = acc;  // the mirrored tile, so that the apply reads rows
  }
}

__global__ void __launch_bounds__(NS_T * NS_C) ns_apply_kernel(int m, int n, int splits, const double* __restrict__ Q,
                                                               const double* __restrict__ P, double* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  __shared__ double A[NS_T][33], B[32][NS_C + 1];
  const int tx = threadIdx.x % NS_C, ty = threadIdx.x / NS_C;
  const int r0 = blockIdx.y * NS_T, c0 = blockIdx.x * NS_C;
  double acc = 0.0;
  for (int k0 = 0; k0 < n; k0 += 32) {
    for (int e = threadIdx.x; e < NS_T * 32; e += blockDim.x) {
      const int rr = e / 32, kk = e - rr * 32;  // A[rr][kk] = Q[r0 + rr][k0 + kk]
      A[rr][kk] = (r0 + rr < m && k0 + kk < n) ? Q[(size_t)(r0 + rr) * n + k0 + kk] : 0.0;
    }
    for (int e = threadIdx.x; e < 32 * NS_C; e += blockDim.x) {
      const int kb = e / NS_C, cc = e - kb * NS_C;  // B[kb][cc] = G[k0 + kb][c0 + cc]
      const int k = k0 + kb, c = c0 + cc;
      double g = 0.0;
      if (k < n && c < n) {
        double p = 0.0;
        for (int sp = 0; sp < splits; ++sp) p += P[(size_t)sp * n * n + (size_t)k * n + c];
        g = (k == c ? 1.5 : 0.0) - 0.5 * p;
      }
      B[kb][cc] = g;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < 32; ++kk) acc = fma(A[ty][kk], B[kk][tx], acc);
    __syncthreads();
  }
  if (r0 + ty < m && c0 + tx < n) out[(size_t)(r0 + ty) * n + c0 + tx] = acc;
}
}  // namespace

void splitk_reduce(cudaStream_t st, int M, int N, int inner, int splitk, int batch, double alpha, const double* ws,
                   double beta, OutView C) {
  const long long total = (long long)M * N * batch;
  int blocks = (int)((total + 255) / 256);
  if (blocks > 4096) blocks = 4096;
  launch_pdl(splitk_reduce_kernel, dim3((unsigned)blocks), dim3(256), 0, st, M, N, inner, splitk, batch, alpha,
             (const double*)ws, beta, C);
}

namespace {
// Tile (TM rows, RN groups of 8 columns) and grid K split of a product, by the
// clocks of the SM with the most blocks: per block its share of the warp FMAs
// (two warps a scheduler, 64 clocks each) and what does not overlap with them
// (about 2000 clocks of load latency and epilogue, 100 per chunk of K).  A
// split over the grid adds its reduction launch and the partial tiles.
struct F64Plan {
  int tm = 32, rn = 9, split = 1, kchunk = 0;
};
F64Plan search_f64(int M, int N, int K, long long batch, size_t ws_elems) {
  F64Plan best;
  double tbest = 1e300;
  const int smax = (int)std::min<long long>(64, (K + KC - 1) / KC);
  for (int s = 1; s <= smax; s *= 2) {
    if (s > 1 && ((size_t)s * batch * (size_t)M * N > ws_elems || s * batch > 65535)) break;
    int kchunk = (K + s - 1) / s;
    if (s > 1) kchunk = (kchunk + KC - 1) / KC * KC;
    const int sr = (K + kchunk - 1) / kchunk;
    for (int tm = 4; tm <= 32; tm *= 2) {
      if ((M + tm - 1) / tm > 65535) continue;
      for (int rn = 1; rn <= 9; ++rn) {
        const long long tiles = (long long)((M + tm - 1) / tm) * ((N + 8 * rn - 1) / (8 * rn)) * batch * sr;
        const int ks = 32 / tm;
        const double block = (double)((kchunk + ks - 1) / ks) * rn * 128.0 + (kchunk + KC - 1) / KC * 100.0;
        double t = (double)((tiles + 151) / 152) * block + 2000.0;
        if (sr > 1) t += 6000.0 + (2.0 * sr + 1.0) * 8.0 * M * N * (double)batch / 2000.0;
        if (t < tbest) {
          tbest = t;
          best.tm = tm;
          best.rn = rn;
          best.split = sr;
          best.kchunk = kchunk;
        }
      }
    }
  }
  return best;
}

// The search is a few hundred evaluations, so each host thread keeps the plans
// of the shapes it met (a fixed table; a plan depends on nothing else).
F64Plan plan_f64(int M, int N, int K, long long batch, size_t ws_elems) {
  struct Entry {
    int M = 0, N = 0, K = 0;
    long long batch = 0;
    size_t ws = 0;
    F64Plan plan;
  };
  thread_local Entry table[512];
  const unsigned long long key = ((((unsigned long long)M * 1000003ull + N) * 1000003ull + K) * 1000003ull + batch) ^ ws_elems;
  Entry& e = table[(key * 0x9E3779B97F4A7C15ull) >> 55];
  if (e.M != M || e.N != N || e.K != K || e.batch != batch || e.ws != ws_elems) {
    e.M = M;
    e.N = N;
    e.K = K;
    e.batch = batch;
    e.ws = ws_elems;
    e.plan = search_f64(M, N, K, batch, ws_elems);
  }
  return e.plan;
}

template <int TM>
void launch_f64(cudaStream_t st, int rn, dim3 grid, int M, int N, int K, int inner, int splitk, int kchunk, double alpha,
                MatView A, MatView B, double beta, OutView C, double* ws) {
#define QTT_F64(RN_)                                                                                               \
  case RN_:                                                                                                        \
    launch_pdl(gemm_f64_kernel<TM, RN_>, grid, dim3(NT), 0, st, M, N, K, inner, splitk, kchunk, alpha, A, B, beta, \
               C, ws);                                                                                             \
    break;
  switch (rn) {
    QTT_F64(1) QTT_F64(2) QTT_F64(3) QTT_F64(4) QTT_F64(5) QTT_F64(6) QTT_F64(7) QTT_F64(8) QTT_F64(9)
  }
#undef QTT_F64
}
}  // namespace

void gemm_f64(cudaStream_t st, int M, int N, int K, int outer, int inner, double alpha, MatView A, MatView B,
              double beta, OutView C, double* ws, size_t ws_elems) {
  if (M <= 0 || N <= 0 || outer <= 0 || inner <= 0) return;
  // The row tiles run along grid.y (at most 65535 blocks): taller products
  // (the dense decompression of a large chain) are issued in row chunks.
  constexpr int kRowsPerCall = 1 << 19;
  if (M > kRowsPerCall) {
    for (int m0 = 0; m0 < M; m0 += kRowsPerCall) {
      MatView Ac = A;
      OutView Cc = C;
      Ac.p += (long long)m0 * A.rs;
      Cc.p += (long long)m0 * C.rs;
      gemm_f64(st, std::min(kRowsPerCall, M - m0), N, K, outer, inner, alpha, Ac, B, beta, Cc, ws, ws_elems);
    }
    return;
  }
  const int batch = outer * inner;
  if (K <= 0) {  // empty contraction: C = beta * C
    const long long total = (long long)M * N * batch;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    count_launches(1);
    scale_out_kernel<<<blocks, 256, 0, st>>>(M, N, inner, batch, beta, C);
    return;
  }
  const F64Plan p = plan_f64(M, N, K, batch, ws ? ws_elems : 0);
  const dim3 grid((unsigned)((N + 8 * p.rn - 1) / (8 * p.rn)), (unsigned)((M + p.tm - 1) / p.tm),
                  (unsigned)(batch * p.split));
  double* w = p.split > 1 ? ws : nullptr;
  count_launches(p.split == 1 ? 1 : 2);
  switch (p.tm) {
    case 4: launch_f64<4>(st, p.rn, grid, M, N, K, inner, p.split, p.kchunk, alpha, A, B, beta, C, w); break;
    case 8: launch_f64<8>(st, p.rn, grid, M, N, K, inner, p.split, p.kchunk, alpha, A, B, beta, C, w); break;
    case 16: launch_f64<16>(st, p.rn, grid, M, N, K, inner, p.split, p.kchunk, alpha, A, B, beta, C, w); break;
    default: launch_f64<32>(st, p.rn, grid, M, N, K, inner, p.split, p.kchunk, alpha, A, B, beta, C, w); break;
  }
  if (p.split > 1) splitk_reduce(st, M, N, inner, p.split, batch, alpha, ws, beta, C);
}

void newton_schulz_step(cudaStream_t st, int m, int n, const double* Q, double* G, double* out) {
  if (m <= 0 || n <= 0) return;
  count_launches(2);
  const int nt = (n + NS_T - 1) / NS_T;
  const int pairs = nt * (nt + 1) / 2;
  const int chunks = (m + 31) / 32;  // K slices come in chunks of 32 rows
  int splits = 152 / pairs;
  splits = std::max(1, std::min({splits, chunks, NS_MAX_SPLIT}));
  const int rows = ((chunks + splits - 1) / splits) * 32;
  splits = (m + rows - 1) / rows;
  launch_pdl_chain(ns_gram_kernel, dim3((unsigned)pairs, (unsigned)splits), dim3(256), 0, st, m, n, nt, rows, Q, G);
  const unsigned bc = (unsigned)((n + NS_C - 1) / NS_C), bm = (unsigned)((m + NS_T - 1) / NS_T);
  launch_pdl_chain(ns_apply_kernel, dim3(bc, bm), dim3(NS_T * NS_C), 0, st, m, n, splits, Q, (const double*)G, out);
}

}  // namespace qtt
