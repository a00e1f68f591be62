// Device kernels of the QTT Fokker-Planck path (launch wrappers).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

namespace qtt {

constexpr int kMaxSites = 64;

// Number of kernels launched by this library since it was loaded.
unsigned long long launch_count();
void count_launches(int n);

// Programmatic dependent launch (optional).  The step is a long chain of
// small kernels on one stream; with programmatic stream serialisation the
// next kernel can be scheduled, and run its prologue (barrier init, TMEM
// allocation), while the previous one finishes.  Every kernel launched
// through launch_pdl calls pdl_trigger() first and pdl_wait() before its first
// global-memory access (read or write), which returns once the preceding
// kernel has completed and its memory is visible.  Without the launch
// attribute both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Whether launch_pdl sets the attribute (environment QTT_PDL=1 turns it on;
// read once).
bool pdl_enabled();

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
// The same with the attribute always set: for the short chain QR factorisation
// -> Q formation -> Newton-Schulz Gram -> apply, whose kernels occupy few SMs
// each, so that the next one is resident (waiting in pdl_wait) when the
// previous one ends.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_chain(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                    Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Operand view for the strided batched GEMM: element (i, j) of batch
// (bo, bi) lives at p[bo * so + bi * si + i * rs + j * cs].
struct MatView {
  const double* p = nullptr;
  long long rs = 0, cs = 0, so = 0, si = 0;
};
struct OutView {
  double* p = nullptr;
  long long rs = 0, cs = 0, so = 0, si = 0;
};

// A chain of MPS cores passed by value to kernels: core n is
// [bond[n]][2][bond[n+1]] row-major.
struct Chain {
  const double* core[kMaxSites];
  int bond[kMaxSites + 1];
  int n;
};

// Points a block of the point evaluation carries, and its shared memory.  FP64
// issue bounds it (one FMA per point and core entry of its bit), so few points
// go eight to a block, sharing each load of a core between them, once there
// are enough to fill the SMs that way, and four otherwise; bonds whose rows do
// not fit take fewer.
constexpr int kEvalThreads = 256;
inline size_t eval_points_smem(int pt, int max_bond) {
  return ((size_t)2 * pt * max_bond + (size_t)kEvalThreads * pt) * sizeof(double);
}
inline int eval_points_per_block(int npts, int max_bond) {
  int pt = npts > 8 * 304 ? 8 : 4;
  while (pt > 1 && eval_points_smem(pt, max_bond) > 160 * 1024) pt /= 2;
  return pt;
}

#ifdef __CUDACC__
// f at up to PT grid points, evaluated by one block of kEvalThreads: the row
// vectors v (length of the current bond) are carried through the chain, v <- v
// A_n[:, s_n, :], with s_n the n-th index bit of each point, read by bit(p, n)
// (any flag type: bytes or 0/1 doubles).  A warp takes 32 columns and a part
// of the rows of a core (the parts' sums meet in shared memory), so a core
// entry is loaded once for all points of the block and eight are in flight.
// sm: eval_points_smem(PT, max_bond) bytes.  4096 points of a 30-site chi = 64
// state with copies take 0.8 ms and 512 points of a 40-site chi = 128 state 0.6.
// (Before, a warp per point kept its row in global memory, one dependent load
// and FMA after another.  This, the joint chain of the mean fields and the kept
// scratch took the points, mean fields and scalars of the 30-site state from
// 3.3 to 2.3 ms, with the FP64 GEMM that they share already as it is now.)
template <int PT, typename BitFn>
__device__ __forceinline__ void eval_points_block(const Chain& f, BitFn bit, int npts, int max_bond, double* sm,
                                                  double* out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* v = sm;
  double* v2 = sm + (size_t)PT * max_bond;
  double* red = v2 + (size_t)PT * max_bond;
  for (int p = tid; p < PT; p += kEvalThreads) v[(size_t)p * max_bond] = 1.0;
  __syncthreads();
  for (int n = 0; n < f.n; ++n) {
    const int bl = f.bond[n], br = f.bond[n + 1];
    const double* A = f.core[n];
    bool s[PT];
#pragma unroll
    for (int p = 0; p < PT; ++p) s[p] = p < npts && bit(p, n);
    const int chunks = (br + 31) / 32;
    const int wc = chunks >= 8 ? 8 : chunks > 4 ? 8 : chunks > 2 ? 4 : chunks;  // warps across the columns
    const int parts = 8 / wc, part = warp / wc;
    const int b0 = bl * part / parts, b1 = bl * (part + 1) / parts;
    for (int ch = warp % wc; ch < chunks; ch += wc) {
      const int c = ch * 32 + lane;
      double acc[PT];
#pragma unroll
      for (int p = 0; p < PT; ++p) acc[p] = 0.0;
      for (int b = b0; b < b1; b += 4) {
        double a0[4], a1[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool live = c < br && b + u < b1;
          a0[u] = live ? A[((size_t)(b + u) * 2) * br + c] : 0.0;
          a1[u] = live ? A[((size_t)(b + u) * 2 + 1) * br + c] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (b + u >= b1) break;  // warp-uniform
#pragma unroll
          for (int p = 0; p < PT; ++p) acc[p] = fma(v[(size_t)p * max_bond + b + u], s[p] ? a1[u] : a0[u], acc[p]);
        }
      }
      if (parts == 1) {
        if (c < br)
#pragma unroll
          for (int p = 0; p < PT; ++p) v2[(size_t)p * max_bond + c] = acc[p];
      } else {
#pragma unroll
        for (int p = 0; p < PT; ++p) red[((size_t)part * PT + p) * (32 * wc) + c] = acc[p];
      }
    }
    __syncthreads();
    if (parts > 1) {
      for (int x = tid; x < PT * br; x += kEvalThreads) {
        const int p = x / br, c = x - p * br;
        double t = red[(size_t)p * (32 * wc) + c];
        for (int q = 1; q < parts; ++q) t += red[((size_t)q * PT + p) * (32 * wc) + c];
        v2[(size_t)p * max_bond + c] = t;
      }
      __syncthreads();
    }
    double* t = v;
    v = v2;
    v2 = t;
  }
  for (int p = tid; p < npts; p += kEvalThreads) out[p] = v[(size_t)p * max_bond];
}
#endif

// C[b] = alpha * A[b] * B[b] + beta * C[b] for b in [0, outer * inner).
// M x K times K x N.  A split of K accumulates partial products in `ws`
// (reduced in a fixed order, so results are deterministic); ws must hold
// split * outer * inner * M * N doubles or the product runs unsplit.
void gemm_f64(cudaStream_t st, int M, int N, int K, int outer, int inner, double alpha, MatView A,
              MatView B, double beta, OutView C, double* ws, size_t ws_elems);
// C = alpha * sum_k ws[b][k] + beta * C: the fixed-order reduction of split-K partial tiles.
void splitk_reduce(cudaStream_t st, int M, int N, int inner, int splitk, int batch, double alpha, const double* ws,
                   double beta, OutView C);

// Batched GEMM with a small M (<= 32) and K (<= 64) on the CUDA cores, same
// views as gemm_f64; fp32 selects float arithmetic (round to nearest).
bool small_gemm_fits(int M, int N, int K, int outer, int inner);
void small_gemm(cudaStream_t st, bool fp32, int M, int N, int K, int outer, int inner, double alpha, MatView A,
                MatView B, double beta, OutView C);
// A sum of up to four such products in one launch: C = alpha sum_p A_p B_p +
// beta C, p = 0 .. n-1, A_p the view A moved by p a elements and B_p the view
// B moved by (p & 1) b0 + (p >> 1) b1.
struct SumPieces {
  int n = 1;
  long long a = 0, b0 = 0, b1 = 0;
};
void small_gemm_sum(cudaStream_t st, bool fp32, int M, int N, int K, int outer, int inner, double alpha, MatView A,
                    MatView B, double beta, OutView C, const SumPieces& P);

// Thin Householder QR of an m x n row-major matrix (m >= n): Q (m x n,
// row-major) overwrites Qout.  Computed in float (prec_bits 32) or double;
// work must hold 2 * m * n + n doubles.  *status != 0 on failure.
void qr_thin(cudaStream_t st, int m, int n, const double* A, double* Qout, void* work, int prec_bits,
             int* status);

// Symmetric eigen-decomposition of an n x n row-major matrix G (n <= 1024).
// Eigenvalues descending in lam[0..n); eigenvectors of the leading k in the
// columns of U (n x k, row-major).  Computed in float (Householder
// tridiagonalisation, implicit QL) or double (tridiagonalisation, divide and
// conquer with QL on its leaves); work must hold eig_work_bytes(n, prec_bits)
// bytes.  *status |= 2 when a QL iteration hits its cap.
size_t eig_work_bytes(int n, int prec_bits);  // plus 256 + sizeof(EigProblem) for eig_sym
void eig_sym(cudaStream_t st, int n, int k, const double* G, double* U, double* lam, void* work, int prec_bits,
             int* status);
// Many independent problems in one pass (the tridiagonalisation takes one
// block per problem, the other phases several); the descriptors live in device
// memory, nmax / kmax bound every n / k.
struct EigProblem {
  int n = 0, k = 0;
  const double* G = nullptr;
  double* U = nullptr;
  double* lam = nullptr;
  unsigned char* work = nullptr;  // eig_work_bytes(n, prec_bits) bytes
};
void eig_sym_batched(cudaStream_t st, const EigProblem* probs_dev, int nprob, int nmax, int kmax, int prec_bits,
                     int* status);

// Rank selection of the bond truncation, one block per problem: with
// lam (descending, n values) and U (n x k, k = kept columns at most), keep
// kk = min(k, #{lam_i > thr}) columns, thr = max(tol^2, floor_rel) * lam_0,
// zero the columns kk..k-1 of U, add sum_{i >= kk} lam_i to *discarded and
// store kk in ranks[problem].
void truncate_select(cudaStream_t st, const EigProblem* probs_dev, int nprob, double tol, double floor_rel,
                     double* discarded, int* ranks);

// core[a][s][b] = (b == 2a + s): an r x 2 x 2r left identity core.
void fill_identity_left(cudaStream_t st, double* core, int r);
// core[a][s][b] = (a == s * c + b): a 2c x 2 x c right identity core.
void fill_identity_right(cudaStream_t st, double* core, int c);
void fill_value(cudaStream_t st, double* p, size_t n, double v);
// Gaussian N(0, sigma^2) entries from a counter-based generator (splitmix64
// hashing of (seed, stream, index), Box-Muller).
void fill_gaussian(cudaStream_t st, double* p, size_t n, double sigma, unsigned long long seed,
                   unsigned long long stream_id);
// The Gaussian sketch cores of one stage: cores n = 1 .. om.n - 1 (bond
// l_n x 2 x l_{n+1}) with sigma_n = 1 / sqrt(2 l_{n+1}), drawn with the same
// generator from the stream ((*step) * 2 + stage) * kMaxSites + n.  The step
// count is read on the device, so a replayed graph draws fresh cores and a
// restart from a checkpoint (which restores the count) draws the same ones.
void fill_gaussian_sketch(cudaStream_t st, const Chain& om, size_t max_core, unsigned long long seed,
                          const unsigned long long* step, int stage);
// out[x] = in[0][x] + ... + in[n_in - 1][x], n_in <= 4.
void sum_arrays(cudaStream_t st, double* out, const double* const* in, int n_in, size_t n);
// p = the n x n identity (row-major).
void fill_eye(cudaStream_t st, double* p, int n);
// One Newton-Schulz step in FP64 of an almost-orthonormal Q (m x n,
// row-major): out = Q (3 I - Q^T Q) / 2.  G is work space of 8 n n doubles
// (split partial sums of Q^T Q).
void newton_schulz_step(cudaStream_t st, int m, int n, const double* Q, double* G, double* out);
// *c += 1 on the device.
void bump_counter(cudaStream_t st, unsigned long long* c);

// out[q * ldo + b] = contraction of the sites [0, nsites) of the weight
// chain w (bond <= 4) with the MPS chain f, left to right; result indexed by
// the weight's last bond q and f's bond b at position nsites.  One block;
// work holds 16 * max_bond doubles.
void left_weight_env(cudaStream_t st, const Chain& f, const Chain& w, int nsites, int max_bond, double* out,
                     int ldo, double* work);
// The same for nw weight chains (device array wchains_dev[0..nw)) in one
// launch, one block per chain, chain i writing out + i * out_stride;
// environments in shared memory (16 * max_bond doubles, max_bond <= 1600).
void left_weight_envs(cudaStream_t st, const Chain& f, const Chain* wchains_dev, int nw, int nsites, int max_bond,
                      double* out, long long out_stride, int ldo);
// u[b] = sum over the indices of sites [n0, N) of f(..)[b]: right environment
// with the all-ones vector.  One block, a warp per row; work holds 2 * max_bond doubles.
void right_ones_env(cudaStream_t st, const Chain& f, int n0, int max_bond, double* out, double* work);
// Diagonal cores of the mixing term under the subgrid closures: the x cores
// of f (the first one replaced by hf, [2][2][b], the conditional means
// absorbed) times the x cores of the Omega_mix(x) train, site by site as a
// Kronecker product: out_n[(o, h)][s][(o', h')] = Om_j[o][s][o'] F_n[h][s][h']
// with j = n - kphi; out's bonds are the products of the two.
void kron_diag_cores(cudaStream_t st, const Chain& om, const Chain& f, const Chain& out, const double* hf, int kphi);
// One explicit RK2 stage of the first-moment equation Eq. FPMoms (S = 0) on
// the dense x grid (x1 slowest, 2^K per dimension), both species at once:
// out = a m0 + b m + c dt R(m), R(m) = -u . D1 m + div(g grad m) with
// periodic CFD2 differences; g = null: the constant gamma times the compact
// second difference, else the flux form with face values averaged from the
// two neighbours.  m0 is read point-wise only, so out may be m0.
void moment_stage(cudaStream_t st, const double* m0, const double* m, double* out, const double* u, const double* g,
                  double gamma, const int K[3], double dt, double a, double b, double c);
// The space sums of an error sample: acc[0..5) += (M1 - r1)^2, (M2 - r2)^2,
// (N - 1)^2, M1, M2 over the x grid (fields [3][Mx] = <1>, <Phi_1>, <Phi_2>;
// ref [2][Mx]); acc must be zeroed first.
void error_sums(cudaStream_t st, const double* fields, const double* ref, size_t Mx, double* acc);
// Evaluates f at npts multi-indices given as bits[p * N + n].
void eval_points(cudaStream_t st, const Chain& f, int npts, const unsigned char* bits, int max_bond, double* out);
// flag[0] = 1 if any of the n entries is NaN or infinite.
void check_finite(cudaStream_t st, const double* p, size_t n, int* flag);

}  // namespace qtt
