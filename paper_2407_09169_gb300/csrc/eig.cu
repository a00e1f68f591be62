// Symmetric eigen-decomposition for the SVD truncation sweep.
//
// The sweep truncates a bond through the Gram matrix G = M M^T = U diag(lam) U^T
// of the bond matrix (paper: "Matrix product state algorithm" -- the bond
// dimension is limited to chi with the singular value decomposition;
// lam = sigma^2, U = left singular vectors).
//
// Kernels, so that the FP64 work does not all sit on one SM per problem:
//   1. eig_tridiag_ql (one block): Householder reduction to tridiagonal form
//      (matrix in shared memory when it fits, lower-triangle updates); for
//      single-precision problems it then runs the implicit-shift QL iteration
//      on (d, e) in warp 0 (one lane carries the rotation chain; lanes of
//      warps 1 and 2 apply each rotation to e and d and record it in a list
//      of every sweep's rotations) and a stable descending order of the
//      eigenvalues;
//   2. FP64: divide and conquer on (d, e) (below): dc_leaves, then per level
//      dc_deflate, dc_roots, dc_zhat and dc_vectors over all merges of all
//      problems, and dc_order; single precision: eig_apply_rotations (one
//      thread per row of the eigenvector matrix Z of the tridiagonal problem,
//      over several blocks), which replays the rotation list on its row;
//   3. eig_back_transform_reg (FP64 up to n = 160: eight lanes per kept
//      eigenvector, in registers) or eig_back_transform (four lanes, in shared
//      memory): applies the Householder reflectors, U[:, r] = H_0 ... H_{n-3}
//      Z[:, order[r]].
// Every loop is bounded.  A QL iteration stops after 60 sweeps per eigenvalue
// (or when the rotation list is full; status bit 2), and the two QL lanes wait
// on each other for at most about a second (bit 8).  A secular root keeps the
// value it has after 100 steps, inside its bracket, and reports nothing: the
// vectors are formed from the recomputed z, orthogonal for any such roots.
#include <algorithm>

#include <cuda_runtime.h>

#include "kernels.cuh"

namespace qtt {

namespace {
constexpr int TRI_THREADS = 512;
constexpr int EIG_MAXN = 1024;
constexpr int QL_MAX_SWEEPS = 60;
constexpr size_t EIG_SMEM_LIMIT = 176 * 1024;  // + 6 * EIG_MAXN static values stays below 227 KB

template <typename T>
struct Eps;
template <>
struct Eps<double> {
  static __device__ double v() { return 2.220446049250313e-16; }
};
template <>
struct Eps<float> {
  static __device__ float v() { return 1.1920929e-7f; }
};

template <typename T>
__device__ T warp_sum_e(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double rhyp(double a, double b) { return rhypot(a, b); }
__device__ __forceinline__ float rhyp(float a, float b) { return rhypotf(a, b); }
// 1 / sqrt(a^2 + b^2) on the QL recurrence's dependency chain, with b^2
// given (b2 = b * b, computed off the chain): the plain reciprocal square
// root of the sum of squares (fewer dependent operations than the scaled
// rhypot) while the sum stays inside the normal range, else the scaled form.
__device__ __forceinline__ double rhyp_fast_sq(double a, double b, double b2) {
  const double q = fma(a, a, b2);
  const int ex = (__double2hiint(q) >> 20) & 0x7ff;
  return (ex > 27 && ex < 2019) ? rsqrt(q) : rhypot(a, b);
}
__device__ __forceinline__ float rhyp_fast_sq(float a, float b, float b2) {
  const float q = fmaf(a, a, b2);
  return (q > 1e-35f && q < 1e35f) ? rsqrtf(q) : rhypotf(a, b);
}

// Bounded spins on a flag in shared memory, between the QL chain and its
// helper lane: at most ~2^26 polls and about a second of wall time; on expiry
// the abort word is set so that the other side stops too.
constexpr long long QL_SPIN_LIMIT = 1LL << 26;
__device__ __forceinline__ bool ql_spin_expired(long long it, unsigned long long t0) {
  if ((it & 1023) != 1023) return it >= QL_SPIN_LIMIT;
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return it >= QL_SPIN_LIMIT || t - t0 > 1000000000ull;
}
__device__ __forceinline__ unsigned long long ql_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// waits for *w == v; false if it expired or the abort word was set
__device__ inline bool ql_wait_eq(volatile int* w, int v, volatile int* abort_w) {
  const unsigned long long t0 = ql_now();
  for (long long it = 0;; ++it) {
    if (*w == v) return true;
    if (*abort_w || ql_spin_expired(it, t0)) {
      *abort_w = 1;
      return false;
    }
  }
}
// waits for *w >= v
__device__ inline bool ql_wait_ge(volatile int* w, int v, volatile int* abort_w) {
  const unsigned long long t0 = ql_now();
  for (long long it = 0;; ++it) {
    if (*w >= v) return true;
    if (*abort_w || ql_spin_expired(it, t0)) {
      *abort_w = 1;
      return false;
    }
  }
}
// waits for *w != seen; returns the new value, or -2 on expiry / abort
__device__ inline int ql_wait_change(volatile int* w, int seen, volatile int* abort_w) {
  const unsigned long long t0 = ql_now();
  for (long long it = 0;; ++it) {
    const int v = *w;
    if (v != seen) return v;
    if (*abort_w || ql_spin_expired(it, t0)) {
      *abort_w = 1;
      return -2;
    }
  }
}

// Work layout, in elements of T: A n*n | Z n*n | rot_c R | rot_s R | (divide
// and conquer) V n*n | vectors 12 n; then ints: seg_lo S | seg_hi S |
// seg_off S | order n | nseg 4 | (divide and conquer) 8 n.  Float problems
// have R = 4 n^2 + 64 n rotations and S = 60 n sweeps, FP64 ones none.
struct EigLayout {
  size_t A, Z, rc, rs, R, S;
  size_t dcV, dcv;
  size_t ints_off;  // bytes
  size_t seg_lo, seg_hi, seg_off, order, nseg, dci;
  size_t bytes;
};

template <typename T>
__host__ __device__ EigLayout eig_layout(int n) {
  EigLayout L;
  const size_t nn = (size_t)n * n;
  constexpr bool ql = sizeof(T) == 4;
  L.R = ql ? 4 * nn + 64 * (size_t)n : 0;
  L.S = ql ? (size_t)QL_MAX_SWEEPS * n : 0;
  L.A = 0;
  L.Z = nn;
  L.rc = 2 * nn;
  L.rs = L.rc + L.R;
  L.dcV = L.rs + L.R;
  L.dcv = L.dcV + nn;
  L.ints_off = (L.dcv + 12 * (size_t)n) * sizeof(T);
  L.ints_off = (L.ints_off + 15) & ~(size_t)15;
  L.seg_lo = 0;
  L.seg_hi = L.S;
  L.seg_off = 2 * L.S;
  L.order = 3 * L.S;
  L.nseg = 3 * L.S + n;
  L.dci = L.nseg + 4;
  L.bytes = L.ints_off + (L.dci + 8 * (size_t)n) * sizeof(int);
  return L;
}

template <typename T>
__global__ void __launch_bounds__(TRI_THREADS) eig_tridiag_ql(const EigProblem* __restrict__ probs, int use_smem,
                                                              int* status, int dc) {
  const EigProblem P = probs[blockIdx.x];
  const int n = P.n;
  if (n <= 0) return;
  const double* __restrict__ G = P.G;
  double* __restrict__ lam = P.lam;
  unsigned char* work = P.work;
  const EigLayout L = eig_layout<T>(n);
  T* W = (T*)work;
  int* I = (int*)(work + L.ints_off);
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  T* A = use_smem ? (T*)dyn_smem : W + L.A;
  T* rcg = W + L.rc;
  T* rsg = W + L.rs;
  int* seg_lo = I + L.seg_lo;
  int* seg_hi = I + L.seg_hi;
  int* seg_off = I + L.seg_off;
  int* order = I + L.order;
  __shared__ T d[EIG_MAXN], e[EIG_MAXN], vb[EIG_MAXN], pb[EIG_MAXN], wb[EIG_MAXN], tauv[EIG_MAXN];
  __shared__ T s_tau, s_inv;
  __shared__ int ql_ctl[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // row stride of the working copy: n + 1 in shared memory (rows of
  // consecutive threads then fall on different banks), n in global memory
  const int lda = use_smem ? n + 1 : n;
  for (size_t x = tid; x < (size_t)n * n; x += TRI_THREADS) {
    const int i = (int)(x / n), c = (int)(x - (size_t)i * n);
    A[(size_t)i * lda + c] = (T)(0.5 * (G[x] + G[(size_t)c * n + i]));
  }
  __syncthreads();

  // ---- Householder tridiagonalisation.  Only the lower triangle (c <= i) of
  // the trailing block is kept current; reflector j is stored in row j,
  // columns > j + 1 (the strict upper part, unused otherwise).  FP64 issues
  // at a fraction of a lane per clock per scheduler, so the products are laid
  // out to keep whole warps busy: A22 v with four threads per row (no
  // reduction over a warp per row), the rank-2 update over the flattened lower
  // triangle (no lanes idle on short rows) with two FMAs per element.  Warp 0
  // updates column j + 1 first and forms the scalars of reflector j + 1 (two
  // reductions' worth of dependent FP64, a square root and two reciprocals)
  // while the other warps update the rest.
  // Scalars of the reflector of column c, by warp 0: tau, 1 / v0, d and e.
  auto reflector_scalars = [&](int c) {
    T s = 0;
    for (int i = c + 2 + lane; i < n; i += 32) {
      const T v = A[(size_t)i * lda + c];
      s += v * v;
    }
    s = warp_sum_e(s);
    if (lane == 0) {
      const T alpha = A[(size_t)(c + 1) * lda + c];
      d[c] = A[(size_t)c * lda + c];
      if (s == (T)0) {
        s_tau = 0;
        e[c] = alpha;
      } else {
        const T mu = sqrt(alpha * alpha + s);
        const T beta = alpha <= (T)0 ? mu : -mu;
        s_tau = (beta - alpha) / beta;
        s_inv = (T)1 / (alpha - beta);
        e[c] = beta;
      }
      tauv[c] = s_tau;
    }
  };
  if (n > 2 && warp == 0) reflector_scalars(0);
  for (int j = 0; j + 2 < n; ++j) {
    T* Aj = A + (size_t)j * lda;
    __syncthreads();  // the scalars of reflector j and the updated trailing block
    const T tau = s_tau;
    if (tau == (T)0) {  // uniform branch (shared value): no update
      __syncthreads();  // everyone has read s_tau
      if (warp == 0 && j + 3 < n) reflector_scalars(j + 1);
      continue;
    }
    {
      const T inv = s_inv;
      for (int i = j + 2 + tid; i < n; i += TRI_THREADS) {
        const T v = A[(size_t)i * lda + j] * inv;
        vb[i] = v;
        Aj[i] = v;
      }
      if (tid == 0) vb[j + 1] = (T)1;
    }
    __syncthreads();
    // p = tau * A22 v, A22 symmetric with its lower triangle stored: four
    // threads per row (lanes 4r .. 4r + 3), each over every fourth column
    const int m = n - j - 1;
    const int m4 = (4 * m + 31) & ~31;  // whole warps enter each pass (the shuffles)
    for (int x = tid; x < m4; x += TRI_THREADS) {
      const bool ok = x < 4 * m;
      const int i = j + 1 + (x >> 2), q = x & 3;
      T acc = 0, acc1 = 0;
      if (ok) {
        int c = j + 1 + q;
        for (; c + 4 < n; c += 8) {
          const T a0 = c <= i ? A[(size_t)i * lda + c] : A[(size_t)c * lda + i];
          const T a1 = c + 4 <= i ? A[(size_t)i * lda + c + 4] : A[(size_t)(c + 4) * lda + i];
          acc += a0 * vb[c];
          acc1 += a1 * vb[c + 4];
        }
        if (c < n) acc += (c <= i ? A[(size_t)i * lda + c] : A[(size_t)c * lda + i]) * vb[c];
        acc += acc1;
      }
      // the four partial sums of a row sit in lanes 4r .. 4r + 3 of one warp
      acc += __shfl_xor_sync(0xffffffffu, acc, 1, 4);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2, 4);
      if (ok && q == 0) pb[i] = tau * acc;
    }
    __syncthreads();
    if (warp == 0) {
      T acc = 0;
      for (int i = j + 1 + lane; i < n; i += 32) acc += pb[i] * vb[i];
      acc = warp_sum_e(acc);
      const T K = (T)0.5 * tau * acc;
      for (int i = j + 1 + lane; i < n; i += 32) wb[i] = pb[i] - K * vb[i];
    }
    __syncthreads();
    if (warp == 0) {
      // column j + 1, then the next reflector
      const T w1 = wb[j + 1];
      for (int i = j + 1 + lane; i < n; i += 32) {
        T* x = A + (size_t)i * lda + j + 1;
        *x = fma(-vb[i], w1, fma(-wb[i], vb[j + 1], *x));
      }
      __syncwarp();
      if (j + 3 < n) reflector_scalars(j + 1);
    } else {
      // lower-triangle rank-2 update, rows i >= j + 2, columns j + 2 <= c <= i,
      // over the flattened triangle: element x is (r, c') with r (r + 1) / 2 <= x
      const int tri = m * (m - 1) / 2;
      for (int x = tid - 32; x < tri; x += TRI_THREADS - 32) {
        int r = (int)((sqrtf(8.f * (float)x + 1.f) - 1.f) * 0.5f);
        while (r * (r + 1) / 2 > x) --r;
        while ((r + 1) * (r + 2) / 2 <= x) ++r;
        const int i = j + 2 + r, c = j + 2 + (x - r * (r + 1) / 2);
        T* y = A + (size_t)i * lda + c;
        *y = fma(-vb[i], wb[c], fma(-wb[i], vb[c], *y));
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (n >= 2) {
      d[n - 2] = A[(size_t)(n - 2) * lda + (n - 2)];
      e[n - 2] = A[(size_t)(n - 1) * lda + (n - 2)];
      tauv[n - 2] = 0;
    }
    d[n - 1] = A[(size_t)(n - 1) * lda + (n - 1)];
    e[n - 1] = 0;
    tauv[n - 1] = 0;
  }
  __syncthreads();
  // reflectors (and tau in the diagonal of A) for the back-transform kernel
  for (size_t x = tid; x < (size_t)n * n; x += TRI_THREADS) {
    const int i = (int)(x / n), c = (int)(x - (size_t)i * n);
    if (c > i + 1) W[L.A + x] = A[(size_t)i * lda + c];
    else if (c == i) W[L.A + x] = tauv[i];
  }

  if (dc) {  // the tridiagonal (d, e) for the divide and conquer, which finds its eigenpairs
    for (int i = tid; i < n; i += TRI_THREADS) {
      W[L.dcv + i] = d[i];
      W[L.dcv + n + i] = e[i];
    }
    return;
  }
  // ---- implicit QL with a Wilkinson-type shift, rotations recorded per sweep.
  // Warp 0 runs it: the search for the next negligible off-diagonal (32
  // entries per ballot) and the shift of the trailing diagonal are spread over
  // its lanes, and lane 0 carries the rotation chain.  FP64 instructions cost
  // the same whatever the number of active lanes, so the chain lane keeps only
  // the operations the next rotation depends on (sum of squares, reciprocal
  // square root, cosine, next p) and hands (p, 1/hypot, e_i) of every
  // rotation to lane 0 of warps 1 and 2, which run on two other schedulers'
  // FP64 pipes one rotation behind: both form the cosine and sine, warp 1
  // updates e[i+1] and records the rotation, warp 2 updates d[i+1] (positions
  // the chain has passed).  The chain waits for both at the end of each
  // sweep.  Every wait is bounded (status bit 8 on expiry).
  {
    T* qlP = vb;  // the tridiagonalisation's vectors are dead from here on
    T* qlR = pb;
    T* qlE2 = wb;
    T* qlEi = tauv;
    volatile int* ctl = ql_ctl;  // 0 sweep number (-1: end), 1 l, 2 m, 3 off, 4 published, 5 / 7 done (e / d), 6 abort
    if (tid == 0) {
      ctl[0] = 0;
      ctl[4] = 0;
      ctl[5] = 0;
      ctl[6] = 0;
      ctl[7] = 0;
    }
    __syncthreads();
    if (warp == 0) {
      const T eps = Eps<T>::v();
      T f = 0, tst1 = 0;
      int nseg = 0, sweep = 0;
      size_t off = 0;
      bool aborted = false;  // warp-uniform (lane 0's view of the abort word)
      for (int l = 0; l < n && !aborted; ++l) {
        const T hl = fabs(d[l]) + fabs(e[l]);
        tst1 = hl > tst1 ? hl : tst1;
        for (int iter = 0;; ++iter) {
          int m = n - 1;
          for (int base = l; base < n - 1; base += 32) {
            const int i = base + lane;
            const bool small = i < n - 1 && !(fabs(e[i]) > eps * tst1);
            const unsigned bal = __ballot_sync(0xffffffffu, small);
            if (bal) {
              m = base + __ffs(bal) - 1;
              break;
            }
          }
          if (m == l) break;
          if (iter >= QL_MAX_SWEEPS || nseg >= (int)L.S || off + (size_t)(m - l) > L.R) {
            if (lane == 0) atomicOr(status, 2);
            break;
          }
          T g = d[l];
          T p = (d[l + 1] - g) / ((T)2 * e[l]);
          T r = (T)1 / rhyp(p, (T)1);
          if (p < 0) r = -r;
          const T dl0 = e[l] / (p + r);
          const T dl1 = e[l] * (p + r);
          const T h = g - dl0;
          __syncwarp();
          if (lane == 0) {
            d[l] = dl0;
            d[l + 1] = dl1;
          }
          for (int i = l + 2 + lane; i < n; i += 32) d[i] -= h;
          for (int i = l + lane; i < m; i += 32) qlE2[i] = e[i] * e[i];  // e_i^2 for the chain
          f += h;
          __syncwarp();
          ++sweep;
          if (lane == 0) {
            p = d[m];
            const T el1 = e[l + 1];
            seg_lo[nseg] = l;
            seg_hi[nseg] = m - 1;
            seg_off[nseg] = (int)off;
            ctl[1] = l;
            ctl[2] = m;
            ctl[3] = (int)off;
            ctl[4] = 0;
            __threadfence_block();
            ctl[0] = sweep;
            // c: cosine of the previous rotation (1 before the first); c2, c3
            // the two before it; (e_i, rr) of the last two for the sines
            T c = 1, c2 = 1, c3 = 1, e1 = 0, r1 = 0, e2 = 0, r2 = 0;
            int k = 0;
            for (int i = m - 1; i >= l; --i, ++k) {
              c3 = c2;
              c2 = c;
              e2 = e1;
              r2 = r1;
              const T ei = e[i], di = d[i], e2 = qlE2[i];
              // the next p = c' d_i - s' g = rr (p d_i - e_i g), e_i g = c e_i^2:
              // the bracket does not wait for rr
              const T tq = fma(p, di, -(c * e2));
              const T rr = rhyp_fast_sq(p, ei, e2);  // 1 / hypot(p, e_i); e_i != 0 inside an unreduced block
              qlP[i] = p;
              qlR[i] = rr;
              qlEi[i] = ei;
              __threadfence_block();
              ctl[4] = k + 1;
              c = p * rr;
              p = rr * tq;
              e1 = ei;
              r1 = rr;
            }
            const T s = e1 * r1, s2 = e2 * r2;  // sines of the last two rotations (0 when absent)
            p = -s * s2 * c3 * el1 * e[l] / dl1;
            // the helper reads e[l] and d[l] in the last rotation and writes
            // d[l+1 ..], e[l+1 ..]: wait for it before e[l], d[l] and the next search
            if (!ql_wait_eq(ctl + 5, sweep, ctl + 6) || !ql_wait_eq(ctl + 7, sweep, ctl + 6)) atomicOr(status, 8);
            __threadfence_block();
            e[l] = s * p;
            d[l] = c * p;
          }
          off += (size_t)(m - l);
          ++nseg;
          __syncwarp();
          __threadfence_block();  // the helper's d and e, seen by lane 0, for every lane
          aborted = __shfl_sync(0xffffffffu, ctl[6], 0) != 0;
          if (aborted) break;
        }
        if (lane == 0) {
          d[l] += f;
          e[l] = 0;
        }
        __syncwarp();
      }
      if (lane == 0) {
        I[L.nseg] = nseg;
        __threadfence_block();
        ctl[0] = -1;
      }
    } else if ((warp == 1 || warp == 2) && lane == 0) {
      // warp 1: e[i+1] and the rotation list; warp 2: d[i+1] (two schedulers'
      // FP64 pipes).  Each reads the original e_i and d_i of its own
      // positions; warp 2 takes e_i from the chain's copy, since warp 1 may
      // already have overwritten it.
      const bool upd_e = warp == 1;
      int seen = 0;
      for (;;) {
        const int sw = ql_wait_change(ctl, seen, ctl + 6);
        if (sw == -2) {  // expired
          atomicOr(status, 8);
          break;
        }
        if (sw < 0) break;
        seen = sw;
        __threadfence_block();
        const int l = ctl[1], m = ctl[2];
        const size_t off = (size_t)ctl[3];
        T c = 1, s = 0;
        bool ok = true;
        for (int k = 0; k < m - l && ok; ++k) {
          ok = ql_wait_ge(ctl + 4, k + 1, ctl + 6);
          if (!ok) break;
          __threadfence_block();
          const int i = m - 1 - k;
          const T p = qlP[i], rr = qlR[i];
          if (upd_e) {
            const T ei = e[i];
            const T cn = p * rr, sn = ei * rr;
            const T r = p * cn + ei * sn;  // hypot(p, e_i)
            e[i + 1] = s * r;               // previous sine
            s = sn;
            c = cn;
            rcg[off + (size_t)k] = c;
            rsg[off + (size_t)k] = s;
          } else {
            const T ei = qlEi[i], di = d[i];
            const T g = c * ei;
            const T hh = c * p;
            const T cn = p * rr, sn = ei * rr;
            s = sn;
            c = cn;
            d[i + 1] = hh + s * (c * g + s * di);
          }
        }
        if (!ok) {
          atomicOr(status, 8);
          break;
        }
        __threadfence_block();
        ctl[upd_e ? 5 : 7] = seen;
      }
    }
  }
  __syncthreads();
  // ---- stable descending order of the eigenvalues
  for (int i = tid; i < n; i += TRI_THREADS) {
    const T di = d[i];
    int rank = 0;
    for (int q = 0; q < n; ++q) {
      const T dq = d[q];
      rank += (dq > di) || (dq == di && q < i);
    }
    order[rank] = i;
  }
  __syncthreads();
  for (int r = tid; r < n; r += TRI_THREADS) lam[r] = (double)d[order[r]];
}

// ---------------------------------------------------------------------------
// Divide and conquer on the tridiagonal (FP64): the QL chain above issues one
// dependent FP64 rotation after another, about 1.7k cycles each on this GPU,
// and a full 136 x 136 spectrum takes ~10k of them plus their replay on Z.
// Here the tridiagonal T is cut recursively in halves (Cuppen):
//   T = diag(T1, T2) + beta (e_a + e_b)(e_a + e_b)^T,  beta = T[a][b] at the
// cut, T1's last and T2's first diagonal entries minus beta;
// leaves of at most DC_LEAF rows are solved by the implicit QL iteration in
// one warp each (every lane runs the same scalar recurrence and rotates its
// own row of Z), and two solved halves T1 = Q1 D1 Q1^T, T2 = Q2 D2 Q2^T are
// merged by the eigen-decomposition of D + rho z z^T, z = (last row of Q1,
// first row of Q2): deflation of the negligible components of z and of
// (nearly) equal poles by plane rotations, one root of the secular equation
// 1 + rho sum_i z_i^2 / (d_i - lambda) = 0 per remaining pole (a rational
// model of each side's poles, safeguarded by the bracket), eigenvector
// components from the recomputed z of Gu and Eisenstat (orthogonal vectors
// from computed roots), and the product of the block-diagonal Q with the
// merged vectors.  Every loop is bounded.
//
// The work is FP64 and an SM does two FMAs a clock, so one block per problem
// (25 to 39 problems on 152 SMs) took 2.5 ms at n = 136, most of it the
// secular sums of the top merge, the product and the leaves.  Each phase is a
// launch over all merges of a level of all problems instead (a launch costs
// about 2 us, the phases 5 to 150): eight lanes per root and per recomputed
// z, eight columns of the product a block, a warp per leaf.  The reciprocals
// are Newton steps on the hardware approximation (five instructions where the
// division takes about ten).  The vectors alternate between Z and V from
// level to level.  With it, the tridiagonalisation's look-ahead and a
// four-lane back-transform, the other kernels as they were then: eigensolver
// class of the 40-site chi = 128 step 8.1 -> 4.6 ms, truncation backward of 40
// sites 11.5 -> 8.0 and of 20 sites (n = 40) 3.5 -> 2.0, 20-site chi = 32 step
// 10.0 -> 8.1.  Now, per stage of 25 problems of n = 136: leaves 160 us, roots
// 440 (four levels), the other phases 210.
constexpr int DC_LEAF = 12;
constexpr int DC_SECULAR_ITERS = 100;
constexpr int DC_THREADS = 128;
constexpr int DC_LANES = 8;                        // lanes of a root
constexpr int DC_GROUPS = DC_THREADS / DC_LANES;   // roots of a block
constexpr int DC_COLS = 8;                         // columns of the product a block forms
constexpr int DC_VEC_THREADS = 256;

// Levels of merges of an n x n problem: 2^depth leaves of at most DC_LEAF rows.
__host__ __device__ inline int dc_depth(int n) {
  int depth = 0;
  while (((n + (1 << depth) - 1) >> depth) > DC_LEAF) ++depth;
  return depth;
}

// 1 / x: the approximate reciprocal (about 20 bits) and two Newton steps
// r <- r + r (1 - x r); x outside the normal range by the division.
__device__ __forceinline__ double dc_rcp(double x) {
  const int ex = (__double2hiint(x) >> 20) & 0x7ff;
  if (ex < 24 || ex > 2022) return 1.0 / x;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// Doubles as integers of the same order (no NaN), so that sorting does not
// use the FP64 pipe.
__device__ __forceinline__ long long dc_key(double x) {
  const long long u = __double_as_longlong(x + 0.0);  // -0 counts as 0
  return u < 0 ? (u ^ 0x7FFFFFFFFFFFFFFFll) : u;
}

// The arrays of one problem and the rows of one merge.
struct DcView {
  double *Z, *V;          // vectors of the level below, of this level
  double *vd, *ve;        // eigenvalues so far; off-diagonal (ve[i] couples i, i + 1)
  double *pk, *zk;        // kept poles ascending; kept z^2
  double *ds, *zs;        // poles in ascending order; z in the same order
  double *tau, *zh;       // root offsets; the kept z, then the recomputed z
  double *rcs, *rss;      // deflation rotations (c, s)
  double *rho, *zsum;     // one value per merge (at its first row)
  int *perm, *jr, *kept;  // sorted position -> local row; origin pole; sorted positions of the kept poles
  int *rl, *ri, *act;     // rotation pairs; columns that are not a copy of one column of Q
  int *kinv, *cnt;        // sorted position -> index among the kept (-1: deflated); per merge kk, nrot
  int n, s0, s1, sp;      // rows s0 .. s1 - 1, cut before sp
};

// False when the problem has no such merge.  lev = 1 .. depth of the launch
// from the leaves up, q the merge of that level.
__device__ bool dc_view(const EigProblem& P, int lev, int depth, int q, DcView& w) {
  const int n = P.n;
  if (n <= 0) return false;
  const int own = dc_depth(n);
  // problems of fewer levels take part in the last ones
  const int l = lev - (depth - own);
  if (l < 1) return false;
  const int dd = own - l;
  if (q >= (1 << dd)) return false;
  const EigLayout L = eig_layout<double>(n);
  double* W = (double*)P.work;
  int* I = (int*)(P.work + L.ints_off);
  w.Z = W + ((l & 1) ? L.Z : L.dcV);
  w.V = W + ((l & 1) ? L.dcV : L.Z);
  w.n = n;
  w.s0 = (q * n) >> dd;
  w.s1 = ((q + 1) * n) >> dd;
  w.sp = ((2 * q + 1) * n) >> (dd + 1);
  double* v = W + L.dcv;
  w.vd = v;
  w.ve = v + n;
  double** dp[10] = {&w.pk, &w.zk, &w.ds, &w.zs, &w.tau, &w.zh, &w.rcs, &w.rss, &w.rho, &w.zsum};
  for (int t = 0; t < 10; ++t) *dp[t] = v + (size_t)(2 + t) * n + w.s0;
  int* p = I + L.dci;
  int** ip[8] = {&w.perm, &w.jr, &w.kept, &w.rl, &w.ri, &w.act, &w.kinv, &w.cnt};
  for (int t = 0; t < 8; ++t) *ip[t] = p + (size_t)t * n + w.s0;
  return true;
}

// Leaf eigenpairs, one warp (block) each, on copies of (d, e) in shared memory
// (the entry of e at a cut is the coupling its merge needs).  Every lane runs
// the same scalar recurrence; lane r rotates row r of the leaf's block of Z,
// which starts as the identity.
__global__ void __launch_bounds__(32) dc_leaves(const EigProblem* __restrict__ probs, int* status) {
  const EigProblem P = probs[blockIdx.y];
  const int n = P.n, q = blockIdx.x, lane = threadIdx.x;
  if (n <= 0) return;
  const int depth = dc_depth(n);
  if (q >= (1 << depth)) return;
  const EigLayout L = eig_layout<double>(n);
  double* W = (double*)P.work;
  double* vd = W + L.dcv;
  const double* ve = vd + n;
  __shared__ double d[DC_LEAF], e[DC_LEAF], zs[DC_LEAF][DC_LEAF + 1];
  const int s0 = (q * n) >> depth, s1 = ((q + 1) * n) >> depth, m = s1 - s0;
  if (lane < m) {
    // the entries beside a cut lose the coupling
    double x = vd[s0 + lane];
    if (lane == 0 && s0 > 0) x -= ve[s0 - 1];
    if (lane == m - 1 && s1 < n) x -= ve[s1 - 1];
    d[lane] = x;
    e[lane] = lane < m - 1 ? ve[s0 + lane] : 0.0;
    for (int c = 0; c < m; ++c) zs[lane][c] = c == lane ? 1.0 : 0.0;
  }
  __syncwarp();
  double* zrow = zs[lane < m ? lane : 0];
  const double eps = Eps<double>::v();
  double f = 0.0, tst1 = 0.0;
  for (int l = 0; l < m; ++l) {
    const double hl = fabs(d[l]) + fabs(e[l]);
    tst1 = hl > tst1 ? hl : tst1;
    for (int iter = 0;; ++iter) {
      int mm = l;
      while (mm < m - 1 && fabs(e[mm]) > eps * tst1) ++mm;
      if (mm == l) break;
      if (iter >= QL_MAX_SWEEPS) {
        if (lane == 0) atomicOr(status, 2);
        break;
      }
      const double g0 = d[l];
      double p = (d[l + 1] - g0) / (2.0 * e[l]);
      double r = hypot(p, 1.0);
      if (p < 0) r = -r;
      const double dl0 = e[l] / (p + r), dl1 = e[l] * (p + r);
      const double h0 = g0 - dl0;
      __syncwarp();
      if (lane == 0) {
        d[l] = dl0;
        d[l + 1] = dl1;
      }
      if (lane >= l + 2 && lane < m) d[lane] -= h0;
      __syncwarp();
      f += h0;
      p = d[mm];
      double c = 1.0, c2 = 1.0, c3 = 1.0, s = 0.0, s2 = 0.0;
      const double el1 = e[l + 1];
      for (int i = mm - 1; i >= l; --i) {
        c3 = c2;
        c2 = c;
        s2 = s;
        const double ei = e[i], di = d[i];
        const double g = c * ei, h = c * p;
        // 1 / hypot(p, e_i) and, from it, the sine, the cosine and hypot
        const double rinv = rhyp_fast_sq(p, ei, ei * ei);
        const double sn = ei * rinv, cn = p * rinv;
        const double ei1 = s * fma(p, cn, ei * sn);
        s = sn;
        c = cn;
        p = c * di - s * g;
        const double di1 = h + s * (c * g + s * di);
        __syncwarp();
        if (lane == 0) {
          e[i + 1] = ei1;
          d[i + 1] = di1;
        }
        if (lane < m) {
          const double zi = zrow[i], zi1 = zrow[i + 1];
          zrow[i + 1] = s * zi + c * zi1;
          zrow[i] = c * zi - s * zi1;
        }
        __syncwarp();
      }
      p = -s * s2 * c3 * el1 * e[l] / dl1;
      __syncwarp();
      if (lane == 0) {
        e[l] = s * p;
        d[l] = c * p;
      }
      __syncwarp();
      if (!(fabs(e[l]) > eps * tst1)) break;
    }
    __syncwarp();
    if (lane == 0) {
      d[l] += f;
      e[l] = 0.0;
    }
    __syncwarp();
  }
  if (lane < m) {
    vd[s0 + lane] = d[lane];
    for (int c = 0; c < m; ++c) (W + L.Z)[(size_t)(s0 + lane) * n + s0 + c] = zs[lane][c];
  }
}

// Poles and z of a merge in ascending order, deflation, the kept poles.
__global__ void __launch_bounds__(DC_THREADS) dc_deflate(const EigProblem* __restrict__ probs, int lev, int depth) {
  DcView w;
  if (!dc_view(probs[blockIdx.y], lev, depth, blockIdx.x, w)) return;
  __shared__ double s_red[DC_THREADS / 32];
  __shared__ int s_kk, s_nrot, s_any;
  __shared__ double sd[EIG_MAXN], sz[EIG_MAXN];  // sorted poles and z
  __shared__ int sprev[EIG_MAXN], sflag[EIG_MAXN];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = w.s1 - w.s0, n1 = w.sp - w.s0;
  const double beta = w.ve[w.sp - 1];
  const double sgn = beta < 0 ? -1.0 : 1.0;
  // poles (sign-flipped for beta < 0) and z = (last row of Q1, first row of Q2)
  double part = 0.0;
  for (int j = tid; j < k; j += DC_THREADS) {
    sd[j] = sgn * w.vd[w.s0 + j];
    const double zj = w.Z[(size_t)(j < n1 ? w.sp - 1 : w.sp) * w.n + w.s0 + j];
    sz[j] = zj;
    part += zj * zj;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane == 0) s_red[warp] = part;
  __syncthreads();
  double z2 = 0.0;
  for (int q = 0; q < DC_THREADS / 32; ++q) z2 += s_red[q];
  const double rho = fabs(beta) * z2, zn = sqrt(z2);
  // ascending order of the poles (stable)
  for (int j = tid; j < k; j += DC_THREADS) {
    const long long pj = dc_key(sd[j]);
    int rank = 0;
    for (int t = 0; t < k; ++t) {
      const long long pt = dc_key(sd[t]);
      rank += (pt < pj) || (pt == pj && t < j);
    }
    w.perm[rank] = j;
    w.ds[rank] = sd[j];
    w.zs[rank] = zn > 0.0 ? sz[j] / zn : 0.0;
  }
  if (tid == 0) s_any = 0;
  __syncthreads();
  for (int r = tid; r < k; r += DC_THREADS) {
    sd[r] = w.ds[r];
    sz[r] = w.zs[r];
  }
  __syncthreads();
  // poles are ascending: the largest magnitude is at an end
  const double tol = 8.0 * Eps<double>::v() * fmax(fmax(fabs(sd[0]), fabs(sd[k - 1])), rho);
  for (int r = tid; r < k; r += DC_THREADS) sflag[r] = fabs(rho * sz[r]) <= tol ? 1 : 0;
  __syncthreads();
  // the pairs to rotate, as long as none has been: each kept pole against the one before it
  for (int r = tid; r < k; r += DC_THREADS) {
    if (sflag[r]) continue;
    int l = r - 1;
    while (l >= 0 && sflag[l]) --l;
    // |(d_r - d_l) c s| <= tol with c s = z_l z_r / t^2
    if (l >= 0 && fabs((sd[r] - sd[l]) * sz[l] * sz[r]) <= tol * (sz[l] * sz[l] + sz[r] * sz[r])) s_any = 1;
  }
  __syncthreads();
  if (s_any) {
    // rotations change the poles and z that later pairs meet: one thread, in order
    if (tid == 0) {
      int nrot = 0, last = -1;
      for (int r = 0; r < k; ++r) {
        if (sflag[r]) continue;
        const double zl = last >= 0 ? sz[last] : 0.0, zr = sz[r];
        if (last >= 0 && fabs((sd[r] - sd[last]) * zl * zr) <= tol * (zl * zl + zr * zr)) {
          const double t = hypot(zl, zr);
          const double c = zl / t, s = zr / t;
          const double dl = sd[last], dr = sd[r];
          sz[r] = t;
          sz[last] = 0.0;
          sd[r] = dl * c * c + dr * s * s;
          sd[last] = dl * s * s + dr * c * c;
          sflag[last] = 1;
          w.rl[nrot] = last;
          w.ri[nrot] = r;
          w.rcs[nrot] = c;
          w.rss[nrot] = s;
          ++nrot;
        }
        last = r;
      }
      s_nrot = nrot;
    }
  } else if (tid == 0) {
    s_nrot = 0;
  }
  __syncthreads();
  // positions of the kept poles: one warp, by ballots
  if (warp == 0) {
    int kk = 0;
    for (int b = 0; b < k; b += 32) {
      const bool live = b + lane < k && !sflag[b + lane];
      const unsigned m = __ballot_sync(0xffffffffu, live);
      if (live) sprev[kk + __popc(m & ((1u << lane) - 1u))] = b + lane;
      kk += __popc(m);
    }
    if (lane == 0) s_kk = kk;
  }
  __syncthreads();
  const int kk = s_kk, nrot = s_nrot;
  for (int r = tid; r < k; r += DC_THREADS) {
    w.act[r] = !sflag[r] ? 1 : 0;
    w.kinv[r] = -1;
    w.ds[r] = sd[r];
  }
  __syncthreads();
  for (int t = tid; t < nrot; t += DC_THREADS) w.act[w.rl[t]] = w.act[w.ri[t]] = 1;
  // the kept poles in ascending order (a rotation may have moved one by <= tol)
  double zpart = 0.0;
  for (int m = tid; m < kk; m += DC_THREADS) {
    const int at = sprev[m];
    const long long pm = dc_key(sd[at]);
    int rank = m;
    if (nrot > 0) {
      rank = 0;
      for (int t = 0; t < kk; ++t) {
        const long long pt = dc_key(sd[sprev[t]]);
        rank += (pt < pm) || (pt == pm && t < m);
      }
    }
    const double zm = sz[at];
    w.kept[rank] = at;
    w.kinv[at] = rank;
    w.pk[rank] = sd[at];
    w.zk[rank] = zm * zm;
    w.zh[rank] = zm;  // its sign, for the recomputed z
    zpart += zm * zm;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) zpart += __shfl_xor_sync(0xffffffffu, zpart, o);
  __syncthreads();
  if (lane == 0) s_red[warp] = zpart;
  __syncthreads();
  if (tid == 0) {
    double zsum = 0.0;
    for (int q = 0; q < DC_THREADS / 32; ++q) zsum += s_red[q];
    w.cnt[0] = kk;  // a merge has at least two rows
    w.cnt[1] = nrot;
    w.rho[0] = rho;
    w.zsum[0] = zsum;
  }
}

// Sum over the DC_LANES lanes of a group (every lane gets it).
__device__ __forceinline__ double dc_group_sum(double v) {
#pragma unroll
  for (int o = DC_LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, DC_LANES);
  return v;
}

// The roots of 1 + rho sum_q z2[q] / (p[q] - lambda) (rho > 0, p increasing,
// kk poles): root i in (p[i], p[i + 1]), or above p[kk - 1] for i = kk - 1, as
// lambda = p[j] + tau with j the pole nearer to the root, so that the
// differences p[q] - lambda = (p[q] - p[j]) - tau keep their relative
// accuracy.  Each step fits psi (the poles <= i) by q / (p_i - tau) + const
// and phi (the others) by s / (p_{i+1} - tau) + const through their values
// and slopes, and takes the model's root inside the bracket.  A group of
// lanes shares the sums of a root and carries the same scalars; the groups of
// a warp iterate together until all are done.
__global__ void __launch_bounds__(DC_THREADS) dc_roots(const EigProblem* __restrict__ probs, int lev, int depth) {
  DcView w;
  if (!dc_view(probs[blockIdx.z], lev, depth, blockIdx.y, w)) return;
  const int kk = w.cnt[0];
  if ((int)blockIdx.x * DC_GROUPS >= kk) return;
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  double* pole = (double*)dyn_smem;
  double* z2 = pole + kk;
  const int tid = threadIdx.x, gl = tid & (DC_LANES - 1);
  for (int q = tid; q < kk; q += DC_THREADS) {
    pole[q] = w.pk[q];
    z2[q] = w.zk[q];
  }
  __syncthreads();
  const double eps = Eps<double>::v(), rho = w.rho[0], zsum = w.zsum[0];
  const int i0 = blockIdx.x * DC_GROUPS + tid / DC_LANES;
  const bool own = i0 < kk;
  const int i = own ? i0 : kk - 1;  // spare groups repeat the last root, so that whole warps shuffle
  const bool last = i == kk - 1;
  const double lo = pole[i], hi = last ? pole[i] + rho * zsum : pole[i + 1];
  const double mid = 0.5 * (lo + hi);
  double part = 0.0;
  for (int q = gl; q < kk; q += DC_LANES) part += z2[q] * dc_rcp(pole[q] - mid);
  const double fmid = 1.0 + rho * dc_group_sum(part);
  const int j = (!last && fmid < 0) ? i + 1 : i;
  const double org = pole[j];
  double a = lo - org, b = hi - org;
  if (fmid < 0) a = fmax(a, mid - org);
  else b = fmin(b, mid - org);
  double tau = 0.5 * (a + b);
  const double pi = pole[i] - org, pi1 = last ? 0.0 : pole[i + 1] - org;
  bool done = false;
  for (int it = 0; it < DC_SECULAR_ITERS; ++it) {
    double psi = 0, dpsi = 0, phi = 0, dphi = 0;
    for (int q = gl; q < kk; q += DC_LANES) {
      const double inv = dc_rcp((pole[q] - org) - tau);
      const double t = z2[q] * inv;
      if (q <= i) {
        psi += t;
        dpsi = fma(t, inv, dpsi);
      } else {
        phi += t;
        dphi = fma(t, inv, dphi);
      }
    }
    psi = dc_group_sum(psi);
    dpsi = dc_group_sum(dpsi);
    phi = dc_group_sum(phi);
    dphi = dc_group_sum(dphi);
    if (!done) {
      const double f = 1.0 + rho * (psi + phi);
      if (fabs(f) <= 8.0 * kk * eps * (1.0 + rho * (fabs(psi) + fabs(phi)))) {
        done = true;
      } else {
        if (f < 0) a = fmax(a, tau);
        else b = fmin(b, tau);
        const double di = pi - tau;
        const double qq = rho * dpsi * di * di;
        double c = f - qq / di;
        double eta;
        if (last) {
          eta = c != 0.0 ? di + qq / c : 0.5 * (a + b) - tau;
        } else {
          const double di1 = pi1 - tau;
          const double ss = rho * dphi * di1 * di1;
          c -= ss / di1;
          // c (di - eta)(di1 - eta) + qq (di1 - eta) + ss (di - eta) = 0
          const double A = c, B = -(c * (di + di1) + qq + ss), C = c * di * di1 + qq * di1 + ss * di;
          eta = 0.5 * (di + di1);
          if (fabs(A) < 1e-300) {
            if (B != 0.0) eta = -C / B;
          } else {
            const double sq = sqrt(fmax(B * B - 4.0 * A * C, 0.0));
            const double den = B > 0 ? -B - sq : -B + sq;
            const double r1 = den != 0.0 ? den / (2.0 * A) : 0.5 * (di + di1);
            const double r2 = (r1 != 0.0) ? C / (A * r1) : 0.5 * (di + di1);
            if (di < r1 && r1 < di1) eta = r1;
            else if (di < r2 && r2 < di1) eta = r2;
          }
        }
        double tn = tau + eta;
        if (!(a < tn && tn < b)) tn = 0.5 * (a + b);
        if (!(a < tn && tn < b)) {
          done = true;  // the bracket is down to adjacent doubles
        } else {
          done = fabs(tn - tau) <= 4.0 * eps * fabs(tn);
          tau = tn;
        }
      }
    }
    if (__all_sync(0xffffffffu, done)) break;
  }
  if (own && gl == 0) {
    w.jr[i] = j;
    w.tau[i] = tau;
  }
}

// Recomputed z (Gu-Eisenstat): zhat_m^2 = prod_i (lambda_i - p_m) / (rho prod_{i != m} (p_i - p_m)).
__global__ void __launch_bounds__(DC_THREADS) dc_zhat(const EigProblem* __restrict__ probs, int lev, int depth) {
  DcView w;
  if (!dc_view(probs[blockIdx.z], lev, depth, blockIdx.y, w)) return;
  const int kk = w.cnt[0];
  if ((int)blockIdx.x * DC_GROUPS >= kk) return;
  const int gl = threadIdx.x & (DC_LANES - 1);
  const int m0 = blockIdx.x * DC_GROUPS + threadIdx.x / DC_LANES;
  const bool own = m0 < kk;
  const int m = own ? m0 : kk - 1;
  const double pm = w.pk[m];
  double v = 1.0;
  for (int t = gl; t < kk; t += DC_LANES)
    if (t != m) v *= -((pm - w.pk[w.jr[t]]) - w.tau[t]) * dc_rcp(w.pk[t] - pm);
#pragma unroll
  for (int o = DC_LANES / 2; o > 0; o >>= 1) v *= __shfl_xor_sync(0xffffffffu, v, o, DC_LANES);
  v *= -((pm - w.pk[w.jr[m]]) - w.tau[m]) / w.rho[0];
  const double a = sqrt(fabs(v));
  if (own && gl == 0) w.zh[m] = w.zh[m] < 0 ? -a : a;
}

// DC_COLS columns of the merged vectors (columns in the order of the sorted
// poles) and their eigenvalues.  The columns in sorted coordinates: the unit
// vector on a deflated position, zhat_m / (p_m - lambda_i) normalised on a
// kept one, then the deflation rotations, last first; moved to the local rows
// and multiplied by blockdiag(Q1, Q2).  A column deflated without a rotation
// is Q's own column.
__global__ void __launch_bounds__(DC_VEC_THREADS) dc_vectors(const EigProblem* __restrict__ probs, int lev, int depth) {
  DcView w;
  if (!dc_view(probs[blockIdx.z], lev, depth, blockIdx.y, w)) return;
  const int k = w.s1 - w.s0, n1 = w.sp - w.s0, n = w.n;
  const int c0 = blockIdx.x * DC_COLS;
  if (c0 >= k) return;
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  double* us = (double*)dyn_smem;       // [sorted position][DC_COLS]
  double* ul = us + (size_t)k * DC_COLS;  // [local row][DC_COLS]
  __shared__ double s_inv[DC_COLS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nrot = w.cnt[1];
  const double sgn = w.ve[w.sp - 1] < 0 ? -1.0 : 1.0;
  // entries: lane = 8 columns x 4 positions
  const int cc = tid & (DC_COLS - 1), c = c0 + cc;
  const int ki = c < k ? w.kinv[c] : -1;
  const double org = ki >= 0 ? w.pk[w.jr[ki]] : 0.0, off = ki >= 0 ? w.tau[ki] : 0.0;
  for (int r = tid / DC_COLS; r < k; r += DC_VEC_THREADS / DC_COLS) {
    const int m = w.kinv[r];
    double v = 0.0;
    if (ki >= 0) {
      if (m >= 0) v = w.zh[m] * dc_rcp((w.pk[m] - org) - off);
    } else if (r == c) {
      v = 1.0;
    }
    us[r * DC_COLS + cc] = v;
  }
  __syncthreads();
  // norms: one warp per column
  for (int x = warp; x < DC_COLS; x += DC_VEC_THREADS / 32) {
    double s2 = 0.0;
    for (int r = lane; r < k; r += 32) {
      const double v = us[r * DC_COLS + x];
      s2 = fma(v, v, s2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    if (lane == 0) s_inv[x] = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
  }
  __syncthreads();
  if (nrot > 0) {
    if (tid < DC_COLS) {
      for (int t = nrot - 1; t >= 0; --t) {
        const int a = w.rl[t], b = w.ri[t];
        const double co = w.rcs[t], si = w.rss[t];
        const double va = us[a * DC_COLS + tid], vb = us[b * DC_COLS + tid];
        us[a * DC_COLS + tid] = -si * va + co * vb;
        us[b * DC_COLS + tid] = co * va + si * vb;
      }
    }
    __syncthreads();
  }
  for (int r = tid / DC_COLS; r < k; r += DC_VEC_THREADS / DC_COLS)
    ul[w.perm[r] * DC_COLS + cc] = us[r * DC_COLS + cc] * s_inv[cc];
  __syncthreads();
  // the product: a warp takes 4 rows x 8 columns at a time
  const int act = c < k ? w.act[c] : 0;
  const int src = c < k ? w.perm[c] : 0;
  for (int r = (tid / DC_COLS); r < k; r += DC_VEC_THREADS / DC_COLS) {
    if (c >= k) continue;
    const double* zr = w.Z + (size_t)(w.s0 + r) * n + w.s0;
    double* out = w.V + (size_t)(w.s0 + r) * n + w.s0 + c;
    const int j0 = r < n1 ? 0 : n1, j1 = r < n1 ? n1 : k;
    if (!act) {  // Q's column src has entries in its own half only
      *out = (src >= j0 && src < j1) ? zr[src] : 0.0;
      continue;
    }
    double a0 = 0.0, a1 = 0.0;
    int j = j0;
    for (; j + 8 <= j1; j += 8) {
      double z[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) z[u] = zr[j + u];
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        a0 = fma(z[u], ul[(j + u) * DC_COLS + cc], a0);
        a1 = fma(z[u + 1], ul[(j + u + 1) * DC_COLS + cc], a1);
      }
    }
    for (; j < j1; ++j) a0 = fma(zr[j], ul[j * DC_COLS + cc], a0);
    *out = a0 + a1;
  }
  // eigenvalue of column c: the root of the kept pole there, or the (rotated) deflated pole itself
  if (tid < DC_COLS && c < k) w.vd[w.s0 + c] = sgn * (ki >= 0 ? org + off : w.ds[c]);
}

// Stable descending order of the eigenvalues.
__global__ void __launch_bounds__(DC_THREADS) dc_order(const EigProblem* __restrict__ probs) {
  const EigProblem P = probs[blockIdx.x];
  const int n = P.n;
  if (n <= 0) return;
  const EigLayout L = eig_layout<double>(n);
  const double* vd = (const double*)P.work + L.dcv;
  int* order = (int*)(P.work + L.ints_off) + L.order;
  __shared__ double sd[EIG_MAXN];
  for (int i = threadIdx.x; i < n; i += DC_THREADS) sd[i] = vd[i];
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += DC_THREADS) {
    const long long di = dc_key(sd[i]);
    int rank = 0;
    for (int q = 0; q < n; ++q) {
      const long long dq = dc_key(sd[q]);
      rank += (dq > di) || (dq == di && q < i);
    }
    order[rank] = i;
    P.lam[rank] = sd[i];
  }
}

// Row `row` of Z (eigenvectors of the tridiagonal matrix as columns) starts as
// e_row and receives every recorded rotation in order.
template <typename T>
__global__ void eig_apply_rotations(const EigProblem* __restrict__ probs) {
  const EigProblem P = probs[blockIdx.y];
  const int n = P.n;
  unsigned char* work = P.work;
  const EigLayout L = eig_layout<T>(n);
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= n) return;
  T* W = (T*)work;
  const int* I = (const int*)(work + L.ints_off);
  const T* rc = W + L.rc;
  const T* rs = W + L.rs;
  T* z = W + L.Z + (size_t)row * n;
  for (int c = 0; c < n; ++c) z[c] = (c == row) ? (T)1 : (T)0;
  const int nseg = I[L.nseg];
  for (int sg = 0; sg < nseg; ++sg) {
    const int lo = I[L.seg_lo + sg], hi = I[L.seg_hi + sg];
    const size_t off = (size_t)I[L.seg_off + sg];
    T zi1 = z[hi + 1];
    for (int i = hi, q = 0; i >= lo; --i, ++q) {
      const T c = rc[off + q], s = rs[off + q];
      const T zi = z[i];
      z[i + 1] = s * zi + c * zi1;
      zi1 = c * zi - s * zi1;
    }
    z[lo] = zi1;
  }
}

// U[:, r] = H_0 ... H_{n-3} Z[:, order[r]] for r < k; four lanes per vector
// (rows i = lane mod 4), eight vectors a warp.  FP64 instructions bound it, so
// the sum v . z takes m / 4 FMAs and two shuffled adds for eight vectors,
// where a warp per vector spent as many instructions on the five levels of
// its reduction as on the sum.  zv: the vectors of dc_vectors' last level (V)
// or of the rotation replay (Z).
constexpr int BT_WARPS = 2, BT_VECS = 8;
template <typename T>
__global__ void __launch_bounds__(32 * BT_WARPS) eig_back_transform(const EigProblem* __restrict__ probs, int dc) {
  const EigProblem P = probs[blockIdx.y];
  const int n = P.n, k = P.k;
  unsigned char* work = P.work;
  double* __restrict__ U = P.U;
  const EigLayout L = eig_layout<T>(n);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = (blockIdx.x * BT_WARPS + w) * BT_VECS;
  if (r0 >= k) return;
  const T* W = (const T*)work;
  const int* I = (const int*)(work + L.ints_off);
  const T* A = W + L.A;
  const T* Z = W + ((dc && (dc_depth(n) & 1)) ? L.dcV : L.Z);
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  T* z = (T*)dyn_smem + (size_t)w * n * BT_VECS;  // [i][vector]
  for (int x = lane; x < n * BT_VECS; x += 32) {
    const int i = x / BT_VECS, r = r0 + x % BT_VECS;
    z[x] = r < k ? Z[(size_t)i * n + I[L.order + r]] : (T)0;
  }
  __syncwarp();
  const int v = lane & 7, q = lane >> 3;  // vector, row residue
  for (int j = n - 3; j >= 0; --j) {
    const T tau = A[(size_t)j * n + j];
    if (tau == (T)0) continue;
    const T* Aj = A + (size_t)j * n;
    T a0 = 0, a1 = 0;
    int i = j + 2 + q;
    for (; i + 4 < n; i += 8) {
      a0 += Aj[i] * z[i * BT_VECS + v];
      a1 += Aj[i + 4] * z[(i + 4) * BT_VECS + v];
    }
    if (i < n) a0 += Aj[i] * z[i * BT_VECS + v];
    a0 += a1;
    a0 += __shfl_xor_sync(0xffffffffu, a0, 8);
    a0 += __shfl_xor_sync(0xffffffffu, a0, 16);
    const T f = -tau * (a0 + z[(j + 1) * BT_VECS + v]);
    __syncwarp();
    if (q == 0) z[(j + 1) * BT_VECS + v] += f;
    for (int x = j + 2 + q; x < n; x += 4) z[x * BT_VECS + v] = fma(f, Aj[x], z[x * BT_VECS + v]);
    __syncwarp();
  }
  for (int x = lane; x < n * BT_VECS; x += 32) {
    const int i = x / BT_VECS, r = r0 + x % BT_VECS;
    if (r < k) U[(size_t)i * k + r] = (double)z[x];
  }
}

// The same in FP64 for n <= 32 NG, with eight lanes per vector and the vectors in
// registers: lane q of a vector holds its rows q + 8 t, in groups of four t that
// a reflector below them skips.  What bounds it is a warp's FP64 instructions, 64
// clocks each with none overlapping (four warps of an SM do): with the vectors in
// shared memory the loads of the reflector and of the vector came on top.  The
// next reflector is loaded meanwhile; with four lanes per vector (half the
// reduction steps) its 36 loads no longer fit the registers and wait.
// The whole eigensolver, 25 problems of n = 136 with 128 vectors: 2.71 -> 2.45 ms,
// 3 of them 2.12 -> 1.83, 17 of n = 72 1.00 -> 0.91.  Larger problems keep the
// vectors in shared memory (above).
template <int NG>
__global__ void __launch_bounds__(64) eig_back_transform_reg(const EigProblem* __restrict__ probs) {
  constexpr int LPV = 8, VECS = 32 / LPV, NR = 4 * NG;  // lanes per vector, vectors per warp, rows per lane
  const EigProblem P = probs[blockIdx.y];
  const int n = P.n, k = P.k;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = (blockIdx.x * 2 + w) * VECS;
  if (r0 >= k) return;
  const EigLayout L = eig_layout<double>(n);
  const double* W = (const double*)P.work;
  const int* I = (const int*)(P.work + L.ints_off);
  const double* A = W + L.A;
  const double* Z = W + ((dc_depth(n) & 1) ? L.dcV : L.Z);
  const int q = lane % LPV, r = r0 + lane / LPV;
  const int col = r < k ? I[L.order + r] : 0;
  double z[NR], an[NR], taun = 0.0;
#pragma unroll
  for (int t = 0; t < NR; ++t) {
    const int x = q + LPV * t;
    z[t] = (r < k && x < n) ? Z[(size_t)x * n + col] : 0.0;
  }
  auto load = [&](int j) {  // v_j: 1 in row j + 1, zeros above
    taun = A[(size_t)j * n + j];
#pragma unroll
    for (int t = 0; t < NR; ++t) {
      const int x = q + LPV * t;
      an[t] = (x > j + 1 && x < n) ? A[(size_t)j * n + x] : (x == j + 1 ? 1.0 : 0.0);
    }
  };
  if (n > 2) load(n - 3);
  for (int j = n - 3; j >= 0; --j) {
    const double tau = taun;
    double a[NR];
#pragma unroll
    for (int t = 0; t < NR; ++t) a[t] = an[t];
    if (j > 0) load(j - 1);
    double d = 0.0;
#pragma unroll
    for (int g = 0; g < NG; ++g)
      if (4 * LPV * (g + 1) > j + 1)
#pragma unroll
        for (int t = 4 * g; t < 4 * g + 4; ++t) d = fma(a[t], z[t], d);
#pragma unroll
    for (int o = 1; o < LPV; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    const double f = -tau * d;
#pragma unroll
    for (int g = 0; g < NG; ++g)
      if (4 * LPV * (g + 1) > j + 1)
#pragma unroll
        for (int t = 4 * g; t < 4 * g + 4; ++t) z[t] = fma(f, a[t], z[t]);
  }
#pragma unroll
  for (int t = 0; t < NR; ++t) {
    const int x = q + LPV * t;
    if (r < k && x < n) P.U[(size_t)x * k + r] = z[t];
  }
}

// false where n is too large for the registers
inline bool back_transform_reg(cudaStream_t st, const EigProblem* probs_dev, int nprob, int nmax, int kmax) {
  const dim3 grid((kmax + 7) / 8, nprob);
  if (nmax <= 64) eig_back_transform_reg<2><<<grid, 64, 0, st>>>(probs_dev);
  else if (nmax <= 96) eig_back_transform_reg<3><<<grid, 64, 0, st>>>(probs_dev);
  else if (nmax <= 160) eig_back_transform_reg<5><<<grid, 64, 0, st>>>(probs_dev);
  else return false;
  return true;
}

template <typename T>
void eig_launch(cudaStream_t st, const EigProblem* probs_dev, int nprob, int nmax, int kmax, int* status) {
  const size_t smem_A = (size_t)nmax * (nmax + 1) * sizeof(T);  // row stride n + 1 in shared memory
  const int use_smem = smem_A <= EIG_SMEM_LIMIT ? 1 : 0;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(eig_tridiag_ql<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)EIG_SMEM_LIMIT);
    attr = true;
  }
  // FP64 problems: tridiagonalisation, then divide and conquer; float ones
  // keep the QL iteration and the replay of its rotations
  constexpr bool dc = sizeof(T) == sizeof(double);
  count_launches(kmax > 0 ? 3 : 2);
  eig_tridiag_ql<T><<<nprob, TRI_THREADS, use_smem ? smem_A : 0, st>>>(probs_dev, use_smem, status, dc ? 1 : 0);
  if constexpr (dc) {
    const int depth = dc_depth(nmax);
    dc_leaves<<<dim3(1u << depth, nprob), 32, 0, st>>>(probs_dev, status);
    const size_t vec_smem = 2 * (size_t)nmax * DC_COLS * sizeof(double);
    static bool vattr = false;
    if (!vattr) {
      cudaFuncSetAttribute(dc_vectors, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(2 * EIG_MAXN * DC_COLS * sizeof(double)));
      vattr = true;
    }
    // problems of a smaller depth skip the levels they do not have
    for (int lev = 1; lev <= depth; ++lev) {
      const int merges = 1 << (depth - lev);
      const int kmx = (nmax + merges - 1) / merges;  // rows of the largest merge of this level
      dc_deflate<<<dim3(merges, nprob), DC_THREADS, 0, st>>>(probs_dev, lev, depth);
      dc_roots<<<dim3((kmx + DC_GROUPS - 1) / DC_GROUPS, merges, nprob), DC_THREADS, 2 * (size_t)kmx * sizeof(double),
                 st>>>(probs_dev, lev, depth);
      dc_zhat<<<dim3((kmx + DC_GROUPS - 1) / DC_GROUPS, merges, nprob), DC_THREADS, 0, st>>>(probs_dev, lev, depth);
      dc_vectors<<<dim3((kmx + DC_COLS - 1) / DC_COLS, merges, nprob), DC_VEC_THREADS, vec_smem, st>>>(probs_dev, lev,
                                                                                                   depth);
    }
    dc_order<<<nprob, DC_THREADS, 0, st>>>(probs_dev);
    count_launches(1 + 4 * depth);
  } else {
    const int rows_per_block = 32;
    eig_apply_rotations<T><<<dim3((nmax + rows_per_block - 1) / rows_per_block, nprob), rows_per_block, 0, st>>>(
        probs_dev);
  }
  if (kmax > 0) {
    if constexpr (dc) {
      if (back_transform_reg(st, probs_dev, nprob, nmax, kmax)) return;
    }
    const int per_block = BT_WARPS * BT_VECS;
    const size_t bt_smem = (size_t)per_block * nmax * sizeof(T);
    static bool battr = false;
    if (!battr) {
      cudaFuncSetAttribute(eig_back_transform<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)((size_t)per_block * EIG_MAXN * sizeof(T)));
      battr = true;
    }
    eig_back_transform<T><<<dim3((kmax + per_block - 1) / per_block, nprob), 32 * BT_WARPS, bt_smem, st>>>(probs_dev,
                                                                                                          dc ? 1 : 0);
  }
}
}  // namespace

size_t eig_work_bytes(int n, int prec_bits) {
  return prec_bits == 32 ? eig_layout<float>(n).bytes : eig_layout<double>(n).bytes;
}

void eig_sym_batched(cudaStream_t st, const EigProblem* probs_dev, int nprob, int nmax, int kmax, int prec_bits,
                     int* status) {
  if (nprob <= 0 || nmax <= 0) return;
  if (nmax > EIG_MAXN || kmax > nmax || kmax < 0) {
    cudaMemsetAsync(status, 0xff, sizeof(int), st);
    return;
  }
  if (prec_bits == 32)
    eig_launch<float>(st, probs_dev, nprob, nmax, kmax, status);
  else
    eig_launch<double>(st, probs_dev, nprob, nmax, kmax, status);
}

void eig_sym(cudaStream_t st, int n, int k, const double* G, double* U, double* lam, void* work, int prec_bits,
             int* status) {
  if (n <= 0) return;
  if (n > EIG_MAXN || k > n || k < 0) {
    cudaMemsetAsync(status, 0xff, sizeof(int), st);
    return;
  }
  // the one-problem descriptor lives at the end of the caller's work area
  const size_t wb = eig_work_bytes(n, prec_bits);
  EigProblem P;
  P.n = n;
  P.k = k;
  P.G = G;
  P.U = U;
  P.lam = lam;
  P.work = (unsigned char*)work;
  EigProblem* d = (EigProblem*)((unsigned char*)work + ((wb + 255) & ~(size_t)255));
  cudaMemcpyAsync(d, &P, sizeof(P), cudaMemcpyHostToDevice, st);
  eig_sym_batched(st, d, 1, n, k, prec_bits, status);
}

}  // namespace qtt
